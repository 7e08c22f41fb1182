"""The quotient by a square root of over_sqrt.h against fp64: no further off than IEEE square root and division, whose results for special
values it has too."""
import ctypes as C
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HARNESS = r"""
#include "over_sqrt.h"
__global__ void k_float(const float* m, const float* x, float* ours, float* ieee, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) { ours[i] = br::over_sqrt(m[i], x[i]); ieee[i] = m[i] / sqrtf(x[i]); }
}
extern "C" __attribute__((visibility("default"))) int run_float(const float* m, const float* x, float* a, float* b, int n) {
  k_float<<<(n + 255) / 256, 256>>>(m, x, a, b, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2602_03515_b200 import build
    d = tmp_path_factory.mktemp("over_sqrt")
    (d / "harness.cu").write_text(HARNESS)
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", "-cudart", "static", "-o", str(d / "harness.so"), str(d / "harness.cu")],
                   check=True, capture_output=True)
    return C.CDLL(str(d / "harness.so"))


def _call(fn, *arrays):
    import torch
    ins = [torch.from_numpy(a).cuda() for a in arrays]
    outs = [torch.empty_like(ins[0]) for _ in range(2)]
    torch.cuda.synchronize()
    assert fn(*[C.c_void_p(t.data_ptr()) for t in ins + outs], C.c_int(arrays[0].size)) == 0
    return [t.cpu().numpy() for t in outs]


def _float_error(got, m, x):
    want = m.astype(np.float64) / np.sqrt(x.astype(np.float64))
    ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
    return (np.abs(got.astype(np.float64) - want) / ulp).max()


@pytest.mark.parametrize("low,high", [(-1, 1), (-30, 30), (-44, -36), (30, 38)])
def test_quotient(lib, low, high):
    rng = np.random.default_rng(high - low)
    n = 1 << 21
    x = (10.0 ** rng.uniform(low, high, n)).astype(np.float32)
    m = (np.where(rng.random(n) < 0.5, -1, 1) * 10.0 ** rng.uniform(-8, 8, n)).astype(np.float32)
    x, m = x[x > 0], m[x > 0]
    ours, ieee = _call(lib.run_float, m, x)
    assert _float_error(ours, m, x) <= 0.501 < _float_error(ieee, m, x)


def test_quotient_special_values(lib):
    v = np.array([0.0, -0.0, 1e-45, 1e-38, 1.0, 3e38, np.inf, -np.inf, np.nan, -1.0, -1e-40, 7.0], dtype=np.float32)
    m, x = [a.ravel().copy() for a in np.meshgrid(v, v)]
    ours, ieee = _call(lib.run_float, m, x)
    assert np.array_equal(np.isnan(ours), np.isnan(ieee)) and np.array_equal(np.isinf(ours), np.isinf(ieee))
    ok = np.isfinite(ieee)
    assert (np.abs(ours[ok].astype(np.float64) - ieee[ok]) <= np.spacing(np.abs(ieee[ok])).astype(np.float64)).all()
    assert np.array_equal(np.sign(ours[~np.isnan(ours)]), np.sign(ieee[~np.isnan(ieee)]))
