"""The products in 8-bit digits (oz.cu) by themselves: their error against extended precision is no larger than that of fp64 sums in
order, also where the parameters behind a factor have gradients of very different size.  (Through a refresh it cannot be seen: the
basis is rounded to fp32.)  The source is compiled here with an entry point for the test, as the library exports none."""
import ctypes as C
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HARNESS = r"""
#include "oz.cu"
namespace br {
void* tensor_map_encoder() {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  return cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess ? p : nullptr;
}
}
extern "C" __attribute__((visibility("default"))) size_t scratch_bytes(long M, long N, long K) { return br::oz_scratch_bytes(M, N, K); }
extern "C" __attribute__((visibility("default"))) int products(const br::OzProduct* v, int n, char* scratch, size_t bytes, int* status) {
  int launches = 0;
  const cudaError_t e = br::oz_product_group(v, n, scratch, bytes, status, 0, &launches);
  return e == cudaSuccess && cudaDeviceSynchronize() == cudaSuccess ? launches : -1;
}
"""


class Product(C.Structure):
    _fields_ = [("X", C.c_void_p), ("Y", C.c_void_p), ("C", C.c_void_p), ("M", C.c_int64), ("N", C.c_int64), ("K", C.c_int64),
                ("diag", C.c_void_p), ("stride", C.c_int64)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2602_03515_b200 import build
    d = tmp_path_factory.mktemp("digits")
    (d / "harness.cu").write_text(HARNESS)
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", "-cudart", "static", "-o", str(d / "harness.so"), str(d / "harness.cu")],
                   check=True, capture_output=True)
    lib = C.CDLL(str(d / "harness.so"))
    lib.scratch_bytes.restype = C.c_size_t
    lib.scratch_bytes.argtypes = [C.c_long] * 3
    lib.products.argtypes = [C.POINTER(Product), C.c_int, C.c_void_p, C.c_size_t, C.c_void_p]
    return lib


def _products(lib, pairs, balanced, room=None):
    """[X Y] of the pairs in one call; balanced[i]: by the diagonal of X.  -> results, launches"""
    import torch
    v = (Product * len(pairs))()
    keep, out = [], []
    for p, (X, Y), b in zip(v, pairs, balanced):
        x, y = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
        c = torch.full((X.shape[0], Y.shape[1]), float("nan"), dtype=torch.float64, device="cuda")
        keep += [x, y]
        out.append(c)
        p.X, p.Y, p.C, p.M, p.N, p.K = x.data_ptr(), y.data_ptr(), c.data_ptr(), X.shape[0], Y.shape[1], X.shape[1]
        p.diag, p.stride = (x.data_ptr(), X.shape[1] + 1) if b else (None, 0)
    room = room or sum(lib.scratch_bytes(p.M, p.N, p.K) for p in v)
    scratch = torch.empty(room, dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    launches = lib.products(v, len(pairs), scratch.data_ptr(), room, status.data_ptr())
    assert launches > 0 and int(status) == 0
    return [c.cpu().numpy() for c in out], launches


def _exact(X, Y):
    return X.astype(np.longdouble) @ Y.astype(np.longdouble)


def _in_order(X, Y):
    s = np.zeros((X.shape[0], Y.shape[1]))
    for k in range(X.shape[1]):
        s += X[:, k:k + 1].astype(np.float64) * Y[k:k + 1].astype(np.float64)
    return s


def _column_errors(got, want):
    d = (got - want).astype(np.float64)
    return np.sqrt(np.mean((np.linalg.norm(d, axis=0) / np.sqrt(np.sum(want * want, axis=0)).astype(np.float64)) ** 2))


@pytest.mark.parametrize("spread", [0.0, 2.0, 4.0, 5.5])
@pytest.mark.parametrize("signal", [0.0, 10.0])
@pytest.mark.parametrize("start", ["random", "tracking"])
def test_error_no_larger_than_that_of_fp64_sums(lib, spread, signal, start):
    """Factors of independent entries or of a strong signal over noise, gradient rows of equal size or over 10^-spread."""
    k = 393
    rng = np.random.default_rng(int(10 * spread + signal))
    s = 10.0 ** (-spread * np.arange(k) / (k - 1))
    rng.shuffle(s)
    G = rng.standard_normal((k, 2 * k)) + signal * rng.standard_normal((k, 16)) @ rng.standard_normal((16, 2 * k))
    G *= s[:, None]
    F = (G @ G.T / (2 * k)).astype(np.float32)
    Q = np.linalg.qr(rng.standard_normal((k, k)))[0].astype(np.float32) if start == "random" else np.eye(k, dtype=np.float32)
    for _ in range(4 if start == "tracking" else 0):
        Q = np.linalg.qr(F.astype(np.float64) @ Q.astype(np.float64))[0].astype(np.float32)
    (got,), _ = _products(lib, [(F, Q)], [True])
    want = _exact(F, Q)
    assert _column_errors(got, want) <= _column_errors(_in_order(F, Q), want)


def test_ragged_products_in_one_call(lib):
    """Eleven products (eight to a launch, and a scratch for some of them at a time), edges of the 128 x 64 tiles and of the 64-step
    stages, with and without a diagonal; every entry within what the digits leave out and the rounding of the final sum."""
    rng = np.random.default_rng(5)
    sizes = [(1, 1, 1), (129, 63, 64), (128, 64, 65), (127, 65, 63), (300, 130, 259), (16, 200, 17), (257, 7, 128), (64, 64, 192), (5, 129, 300),
             (200, 64, 200), (131, 66, 131)]
    pairs = [(rng.standard_normal((m, k)).astype(np.float32), rng.standard_normal((k, n)).astype(np.float32)) for m, n, k in sizes]
    pairs[4][0][:, ::7] = 0.0
    pairs[6][0][3] = 0.0                                    # an empty row
    pairs[7][1][:, 5] = 0.0
    pairs[8][0][0, 0] = 1e-42                               # below the normal numbers
    pairs[9][0][:] = pairs[9][0] @ pairs[9][0].T
    pairs[9][0][11, :] = pairs[9][0][:, 11] = 0.0
    balanced = [False] * 9 + [True, True]                   # (the last one's diagonal has negative entries)
    need = [lib.scratch_bytes(m, n, k) for m, n, k in sizes]
    results = []
    for room in (sum(need), max(need)):
        got, launches = _products(lib, pairs, balanced, room)
        assert launches == 8 if room == sum(need) else launches > 8
        results.append(got)
    for (X, Y), a, b, bal in zip(pairs, *results, balanced):
        assert np.array_equal(a, b)                         # whatever the launches
        d = np.diag(X).astype(np.float64) if bal else np.ones(X.shape[1])
        s = 2.0 ** (np.frexp(np.where(d > 0, d, 0.5))[1] >> 1)
        top = np.abs(X / s).max(1)[:, None] * np.abs(Y * s[:, None]).max(0)[None, :]
        bound = 4 * 2.0 ** -59 * X.shape[1] * top + 2.0 ** -50 * np.abs(X).astype(np.float64) @ np.abs(Y).astype(np.float64)
        assert (np.abs(a - _exact(X, Y)) <= bound).all(), X.shape


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_not_finite(lib, bad):
    rng = np.random.default_rng(9)
    X, Y = rng.standard_normal((140, 140)).astype(np.float32), rng.standard_normal((140, 70)).astype(np.float32)
    X[130, 3] = bad                                         # a row of the result
    Y[7, 66] = bad                                          # and a column
    for balanced in (False, True):
        (got,), _ = _products(lib, [(X, Y)], [balanced])
        hit = np.zeros(got.shape, dtype=bool)
        hit[130] = hit[:, 66] = True
        assert np.array_equal(np.isnan(got), hit)
