// m / sqrt(x) in the epilogue of the tensor-core contraction.
#pragma once
#include <cuda_runtime.h>

namespace br {
namespace {

// Without the branches that sqrtf and a division take for their special cases (the rotated-Adam launches of four d = 384 blocks
// with those: 1.2 % of their refresh period).  From the hardware's approximation r of x^(-1/2) and the binomial series
//   m / sqrt(x) = m r (1 - e)^(-1/2) = m r (1 + e / 2 + ...),   e = 1 - x r^2,
// of which one term is enough: |e| < 2^-21.  What the products x r and m r lose to rounding is their fused multiply-add's remainder (the
// error-free product, Dekker 1971), so that only the last sum rounds: at most 0.501 ulp, where the two IEEE operations leave up
// to 0.998 (tests/test_gpu_over_sqrt.py).  Where the correction is not finite (x = 0 or infinite, an infinite m or m r), m r is the result.
__device__ __forceinline__ float over_sqrt(float m, float x) {
  const float r = rsqrtf(x), h = x * r, y = m * r;
  const float e = fmaf(-fmaf(x, r, -h), r, fmaf(-h, r, 1.0f));
  const float t = fmaf(0.5f * y, e, fmaf(m, r, -y));
  return fabsf(t) < __int_as_float(0x7f800000) ? y + t : y;
}

}  // namespace
}  // namespace br
