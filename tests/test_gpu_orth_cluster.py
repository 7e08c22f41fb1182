"""The one-launch factorisation Q <- qr(F Q).Q of orders below 1600, through the C-ABI (set_state, refresh_basis,
get_state), at the orders where its tiling can go wrong: less than one panel, whole and ragged panels, one CTA
more or less in the cluster, odd orders (8-byte instead of 16-byte copies), the largest order, and orders that go
through the chain of launches.

Reference: LAPACK QR of the float64 product with a positive diagonal of R.  Both sides then round to (library) or
start from (reference) the same fp32 inputs, so what remains is the rounding of Q to fp32 -- at most 2^-24 relative
per entry, 6e-8 of a column's length -- and what one sweep of block Gram-Schmidt leaves when no second one runs, up
to 1e-16 / 1e-7 = 1e-9 per column in each of up to k directions (4.5e-8 at order 2047; the factors with a strong
signal come close to that threshold).  The asserted 1.2e-7 is their sum, rounded up."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1.2e-7


def _refresh(k, F, Q0):
    import torch
    import paper_2602_03515_b200 as br
    from workloads import LayerSpec
    w = torch.zeros(k, 8, device="cuda")
    opt = br.BasisRotation([LayerSpec("W", k, 8, br.BR_GEOM_BILATERAL, br.BR_SRC_SECOND, 0)], [w], grad_dtype="f32",
                           gemm_prec=br.BR_GEMM_FP32, freq=10 ** 6)
    try:
        opt.step([torch.randn(k, 8, device="cuda") * 0.01], 0)
        opt.set_state(0, br.BR_BUF_L, torch.from_numpy(F))
        opt.set_state(0, br.BR_BUF_U, torch.from_numpy(Q0))
        opt.refresh_basis(0)
        opt.sync_status()
        return opt.get_state(0, br.BR_BUF_U).numpy().astype(np.float64)
    finally:
        opt.close()


@pytest.mark.parametrize("k,one", [(1599, True), (1600, False), (2040, False), (2304, False)])
def test_form_by_order(k, one):
    """Which form a refresh takes, told by its launches: the product and the factorisation, or the chain."""
    import torch
    import paper_2602_03515_b200 as br
    from workloads import LayerSpec
    opt = br.BasisRotation([LayerSpec("W", k, k, br.BR_GEOM_UNILATERAL, br.BR_SRC_SECOND, 0)], [torch.zeros(k, k, device="cuda")],
                           grad_dtype="f32", gemm_prec=br.BR_GEMM_FP32, freq=10 ** 6)
    try:
        opt.step([torch.randn(k, k, device="cuda") * 0.01], 0)
        before, _ = opt.launch_stats()
        opt.refresh_basis(0)
        launches = opt.launch_stats()[0] - before
        assert opt.sync_status() == br.BR_OK
        assert launches <= 4 if one else launches > 20, launches
    finally:
        opt.close()


@pytest.mark.parametrize("k", [130, 1599, 1601, 2304])
def test_rank_deficient_product(k):
    """A factor with an exactly empty block, whose rank the host does not know: the factorisation finds the product
    F Q short of rank (some |R_jj| <= 1e-12 of the largest) and, in the same refresh, factorises it with
    1e-6 ||(F Q)_j|| Q_j added to every column -- as branches of the one launch, and from order 1600 on as launches of the
    chain that a device flag turns on.  The completed product has full rank and the completed directions come out of
    it at 1e-6 of its columns: fp64 rounding is 1e-10 of them, far below the fp32 result."""
    import torch
    import paper_2602_03515_b200 as br
    from workloads import LayerSpec
    rng = np.random.default_rng(k)
    r = k - k // 5
    N = rng.standard_normal((r, r)) / np.sqrt(r)
    F = np.zeros((k, k), dtype=np.float32)
    F[:r, :r] = np.eye(r) + 0.1 * (N + N.T)
    Q0 = np.linalg.qr(rng.standard_normal((k, k)))[0].astype(np.float32)
    A = F.astype(np.float64) @ Q0.astype(np.float64)
    A += 1e-6 * np.linalg.norm(A, axis=0) * Q0.astype(np.float64)
    want, R = np.linalg.qr(A)
    want *= np.sign(np.diag(R))
    opt = br.BasisRotation([LayerSpec("W", k, k, br.BR_GEOM_UNILATERAL, br.BR_SRC_SECOND, 0)], [torch.zeros(k, k, device="cuda")],
                           grad_dtype="f32", gemm_prec=br.BR_GEMM_FP32, freq=10 ** 6)
    try:
        opt.step([torch.randn(k, k, device="cuda") * 0.01], 0)
        opt.set_state(0, br.BR_BUF_L, torch.from_numpy(F))
        opt.set_state(0, br.BR_BUF_U, torch.from_numpy(Q0))
        for again in range(2):                 # (the second time the chain comes out of its graph)
            opt.refresh_basis(0)
            assert opt.sync_status() == br.BR_WARN_RANK_DEFICIENT
            got = opt.get_state(0, br.BR_BUF_U).numpy().astype(np.float64)
            assert br.br_get_basis_flags(opt.handle, 0) & 4
            err = np.linalg.norm(got - want) / np.linalg.norm(want)
            assert err <= TOL, (k, again, err)
            opt.set_state(0, br.BR_BUF_U, torch.from_numpy(Q0))
        # a full-rank factor on the same handle: nothing of the completion runs
        F[r:, r:] = np.eye(k - r)
        want, R = np.linalg.qr(F.astype(np.float64) @ Q0.astype(np.float64))
        want *= np.sign(np.diag(R))
        opt.set_state(0, br.BR_BUF_L, torch.from_numpy(F))
        opt.refresh_basis(0)
        assert opt.sync_status() == br.BR_OK
        got = opt.get_state(0, br.BR_BUF_U).numpy().astype(np.float64)
        err = np.linalg.norm(got - want) / np.linalg.norm(want)
        assert err <= TOL, (k, err)
    finally:
        opt.close()


@pytest.mark.parametrize("m,n", [(66000, 260), (260, 66000), (66001, 257), (4200, 4100)])
def test_first_source_product_in_slices(m, n):
    """S = 1st with a momentum of more than 2^24 entries: M^T (M V), or M (M^T U), in slices of the unrotated dimension.
    The error is that of the orders above: the products are exact up to fp64 rounding whatever the slices."""
    import torch
    import paper_2602_03515_b200 as br
    from workloads import LayerSpec
    rng = np.random.default_rng(m)
    k = min(m, n)
    M = rng.standard_normal((m, n)).astype(np.float32)
    if (m, n) == (4200, 4100):
        M += 60 * np.eye(m, n, dtype=np.float32)           # (a square random matrix alone is nearly singular)
    Q0 = np.linalg.qr(rng.standard_normal((k, k)))[0].astype(np.float32)
    M64, Q64 = M.astype(np.float64), Q0.astype(np.float64)
    want, R = np.linalg.qr(M64 @ (M64.T @ Q64) if m <= n else M64.T @ (M64 @ Q64))
    want *= np.sign(np.diag(R))
    which = br.BR_BUF_U if m <= n else br.BR_BUF_V
    opt = br.BasisRotation([LayerSpec("W", m, n, br.BR_GEOM_UNILATERAL, br.BR_SRC_FIRST, 0)], [torch.zeros(m, n, device="cuda")],
                           grad_dtype="f32", gemm_prec=br.BR_GEMM_FP32, freq=10 ** 6)
    try:
        opt.step([torch.randn(m, n, device="cuda") * 0.01], 0)
        opt.set_state(0, br.BR_BUF_M, torch.from_numpy(M))
        opt.set_state(0, which, torch.from_numpy(Q0))
        opt.refresh_basis(0)
        assert opt.sync_status() == br.BR_OK
        got = opt.get_state(0, which).numpy().astype(np.float64)
    finally:
        opt.close()
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err <= TOL, (m, n, err)


@pytest.mark.parametrize("signal", [0.0, 300.0])      # well-conditioned: one sweep; a strong low-rank part: two
@pytest.mark.parametrize("k", [1, 7, 8, 63, 64, 65, 127, 128, 129, 130, 255, 384, 511, 513, 1000, 1537, 1599, 1600, 1601, 2047, 2049])
def test_order(k, signal):
    rng = np.random.default_rng(k)
    N = rng.standard_normal((k, k)) / np.sqrt(k)
    F = np.eye(k) + 0.1 * (N + N.T)
    if signal and k > 4:
        A = signal * rng.standard_normal((k, 4)) / np.sqrt(k)
        F += A @ A.T
    F = F.astype(np.float32)
    Q0 = np.linalg.qr(rng.standard_normal((k, k)))[0].astype(np.float32)
    want, R = np.linalg.qr(F.astype(np.float64) @ Q0.astype(np.float64))
    want *= np.sign(np.diag(R))
    got = _refresh(k, F, Q0)
    err = np.linalg.norm(got - want) / np.linalg.norm(want)
    assert err <= TOL, (k, signal, err)
