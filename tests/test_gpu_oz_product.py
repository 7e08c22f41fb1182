"""The power product F Q in 8-bit digits on the integer tensor cores (orders from 1024 on, several bases in a handle),
through a refresh: orders that no tile divides, rows of very different size, and what is not finite.

The factors are graded: eigenvalues from 1 down to 1e-6, and a basis that is close to their eigenvectors, so that the trailing
columns of F Q are what is left of a cancellation a million times their size.  What the digits leave out, at most 2^-59 times the order of
the largest entries of a row and a column, 2^-48, is then 4e-9 of such a column, below the rounding of the basis to fp32 (6e-8); single
precision anywhere in the product would leave 6e-2.  Reference: LAPACK QR of the float64 product; asserted as in
test_gpu_orth_cluster.py, 1.2e-7."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 1.2e-7


def _refresh(F, Q0):
    import torch
    import paper_2602_03515_b200 as br
    from workloads import LayerSpec
    k = F[0].shape[0]
    ws = [torch.zeros(k, k, device="cuda") for _ in F]
    opt = br.BasisRotation([LayerSpec("W%d" % i, k, k, br.BR_GEOM_UNILATERAL, br.BR_SRC_SECOND, 0) for i in range(len(F))], ws,
                           grad_dtype="f32", gemm_prec=br.BR_GEMM_FP32, freq=10 ** 6)
    try:
        opt.step([torch.randn(k, k, device="cuda") * 0.01 for _ in F], 0)
        for i in range(len(F)):
            opt.set_state(i, br.BR_BUF_L, torch.from_numpy(F[i]))
            opt.set_state(i, br.BR_BUF_U, torch.from_numpy(Q0[i]))
        before = opt.launch_stats()[0]
        opt.refresh_basis()
        launches = opt.launch_stats()[0] - before
        opt.sync_status()
        return [opt.get_state(i, br.BR_BUF_U).numpy().astype(np.float64) for i in range(len(F))], launches
    finally:
        opt.close()


def _graded(k, rng, spread=1.0):
    E = np.linalg.qr(rng.standard_normal((k, k)))[0]
    F = (E * np.logspace(0, -6, k)) @ E.T
    s = spread ** np.linspace(-1, 1, k)                # rows and columns of different size
    F = (s[:, None] * F * s[None, :]).astype(np.float32)
    F = np.triu(F) + np.triu(F, 1).T
    Q = np.linalg.qr(E + 1e-3 * rng.standard_normal((k, k)) / np.sqrt(k))[0] if spread == 1.0 else np.linalg.qr(rng.standard_normal((k, k)))[0]
    return F, Q.astype(np.float32)


@pytest.mark.parametrize("k", [1024, 1025, 1111, 1280, 1599])
def test_graded_factor(k):
    rng = np.random.default_rng(k)
    F, Q = zip(*[_graded(k, rng) for _ in range(2)])
    got, launches = _refresh(F, Q)
    assert launches >= 5, launches                     # digits of rows, of columns, product, factorisation, copy of the notes
    for f, q, u in zip(F, Q, got):
        want, R = np.linalg.qr(f.astype(np.float64) @ q.astype(np.float64))
        want *= np.sign(np.diag(R))
        assert np.linalg.norm(u - want, axis=0).max() <= TOL


def test_rows_of_different_size():
    """Rows and columns whose sizes span a factor of 900, from a basis far from the eigenvectors: the errors of the product,
    at most 2^-48 of the size of its row and column, reach the result times the condition number of the column-scaled product."""
    rng = np.random.default_rng(7)
    F, Q = _graded(1090, rng, spread=30.0)
    got, _ = _refresh([F, F], [Q, Q])
    A = F.astype(np.float64) @ Q.astype(np.float64)
    want, R = np.linalg.qr(A)
    want *= np.sign(np.diag(R))
    cond = np.linalg.cond(A / np.linalg.norm(A, axis=0))
    assert np.linalg.norm(got[0] - want, axis=0).max() <= TOL + 4e-15 * cond
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(bad):
    rng = np.random.default_rng(3)
    F, Q = _graded(1032, rng)
    F = F.copy()
    F[5, 7] = F[7, 5] = bad
    got, _ = _refresh([F, F], [Q, Q])
    assert not np.isfinite(got[0]).all() and not np.isfinite(got[1]).all()
