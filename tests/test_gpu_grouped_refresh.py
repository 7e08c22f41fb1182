"""Several S = 2nd bases below order 1600 in one refresh: grouped products F Q, of orders from 1024 on in digits and of the others on the
fp64 unit, and one grouped factorisation: many different orders, short-of-rank factors among others, and more bases than the
pool or a launch holds.  Reference: LAPACK QR of the float64 product; asserted as in test_gpu_orth_cluster.py, 1.2e-7."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1.2e-7


def _refresh(F, Q0, power_iters=1):
    import torch
    import paper_2602_03515_b200 as br
    from workloads import LayerSpec
    ks = [f.shape[0] for f in F]
    ws = [torch.zeros(k, k, device="cuda") for k in ks]
    opt = br.BasisRotation([LayerSpec("W%d" % i, k, k, br.BR_GEOM_UNILATERAL, br.BR_SRC_SECOND, 0) for i, k in enumerate(ks)], ws,
                           grad_dtype="f32", gemm_prec=br.BR_GEMM_FP32, freq=10 ** 6, power_iters=power_iters)
    try:
        opt.step([torch.randn(k, k, device="cuda") * 0.01 for k in ks], 0)
        for i in range(len(F)):
            opt.set_state(i, br.BR_BUF_L, torch.from_numpy(F[i]))
            opt.set_state(i, br.BR_BUF_U, torch.from_numpy(Q0[i]))
        before = opt.launch_stats()[0]
        opt.refresh_basis()
        launches = opt.launch_stats()[0] - before
        status = opt.sync_status()
        flags = [br.br_get_basis_flags(opt.handle, i) for i in range(len(F))]
        return [opt.get_state(i, br.BR_BUF_U).numpy().astype(np.float64) for i in range(len(F))], launches, status, flags
    finally:
        opt.close()


def _qr(A):
    Q, R = np.linalg.qr(A)
    return Q * np.sign(np.diag(R))


def _want(F, Q, power_iters=1):
    for _ in range(power_iters):
        Q = _qr(F.astype(np.float64) @ Q.astype(np.float64)).astype(np.float32 if power_iters > 1 else np.float64)
    return Q


def _graded(k, rng, low):
    """A factor with eigenvalues from 1 down to 10^low, and a basis close to its eigenvectors."""
    E = np.linalg.qr(rng.standard_normal((k, k)))[0]
    F = ((E * np.logspace(0, low, k)) @ E.T).astype(np.float32)
    Q = np.linalg.qr(E + 1e-3 * rng.standard_normal((k, k)) / np.sqrt(k))[0]
    return np.triu(F) + np.triu(F, 1).T, Q.astype(np.float32)


def _error(got, want):
    return np.linalg.norm(got - want, axis=0).max()


@pytest.mark.parametrize("power_iters", [1, 2])
def test_mixed_orders(power_iters):
    """Orders on one CTA, on part of a cluster and on a whole one in one refresh, the products of six in digits, several to a launch
    (their planes lie in the work areas of the factorisations, also behind those of the first application).  A second application starts from the first
    one's result rounded to fp32, which moves its columns by at most 6e-8 times the condition number of the column-scaled
    product (about 10 with eigenvalues from 1 to 1e-2): 1e-6."""
    rng = np.random.default_rng(11)
    F, Q = zip(*[_graded(k, rng, -2) for k in (130, 1599, 17, 1030, 64, 700, 1536, 257, 1281, 1111, 1025)])
    got, launches, status, _ = _refresh(F, Q, power_iters)
    # an application of the orders above 128: at least two calls of the digits, the other products, the factorisation; of the
    # others product and factorisation; the copy of the notes
    assert status == 0 and 12 * power_iters + 1 <= launches < (4 * 6 + 4) * power_iters + 1, launches
    for f, q, u in zip(F, Q, got):
        assert _error(u, _want(f, q, power_iters)) <= (TOL if power_iters == 1 else 1e-6), f.shape


def test_more_bases_than_the_pool_and_a_launch_hold():
    """The pool holds twelve products of the largest order: fourteen of order 260 and forty-four of order 40 take two rounds,
    the second one of more bases than one launch takes."""
    rng = np.random.default_rng(13)
    F, Q = zip(*[_graded(k, rng, -6) for k in [260] * 14 + [40] * 44])
    got, launches, status, _ = _refresh(F, Q)
    assert status == 0 and launches == 2 + 4 + 1, launches     # product and factorisation, two of each, copy of the notes
    for f, q, u in zip(F, Q, got):
        assert _error(u, _want(f, q)) <= TOL, f.shape


def test_deficient_products_among_others():
    """A product found short of rank is formed once more by the cluster that factorises it and completed from its basis; the
    others of the launch are not touched."""
    rng = np.random.default_rng(17)
    F, Q, want = [], [], []
    for k, short in ((1100, True), (1100, False), (700, False), (130, True), (33, True), (1090, False)):
        f, q = _graded(k, rng, -2)
        r = k - k // 5
        if short:
            N = rng.standard_normal((r, r)) / np.sqrt(r)
            f = np.zeros((k, k), dtype=np.float32)
            f[:r, :r] = np.eye(r) + 0.1 * (N + N.T)
            q = np.linalg.qr(rng.standard_normal((k, k)))[0].astype(np.float32)
        A = f.astype(np.float64) @ q.astype(np.float64)
        if short:
            A += 1e-6 * np.linalg.norm(A, axis=0) * q.astype(np.float64)
        F.append(f); Q.append(q); want.append(_qr(A))
    got, _, status, flags = _refresh(F, Q)
    assert status == 2                                         # BR_WARN_RANK_DEFICIENT
    for i, (u, w) in enumerate(zip(got, want)):
        assert bool(flags[i] & 4) == (i in (0, 3, 4))
        assert _error(u, w) <= TOL, i
