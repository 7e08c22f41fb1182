// fp64-accumulating contractions for the basis refresh (Power(F, Q) of Sec. 3.2): the product
// F Q and the block projections of the QR must be resolved far below the fp32 rounding level
// (F mixes eigenvalues that differ by 1e5, and the small ones are what the trailing basis vectors
// are made of), so they run on the fp64 matrix unit:
//
//   C = alpha * op(A) op(B) + beta * C,  C fp64, A and B fp32 or fp64, all row-major.
//
// The kernels are in orth.cu (64 x 64 tiles of mma.sync.m8n8k4.f64, two CTAs per SM, operands by cp.async three
// stages deep; fp32 operands widened while they are staged, so every product is exact and only the fp64
// accumulation rounds).  Against 128 x 128 tiles with register prefetch, one CTA per SM: 4096^3 30.8 -> 33.2
// TFLOP/s of the unit's 37.2, 1024 x 1024 x 4096 21.6 -> 27.5, 4096 x 256 x 256 11.3 -> 21.3, 2560 x 128 x 2560
// 4.2 -> 14.0: a small tile fills the GPU at the sizes of a factorisation, and its operands still come out of L2.
// A contraction that is long and narrow (projections, rank-128 terms) is split over K into partial sums that a
// second kernel adds in a fixed order, which keeps the result reproducible from run to run.
#include <algorithm>

#include "br_internal.h"

namespace br {
namespace {

// C = alpha * (sum of the partial products, in split order) + beta * C
__global__ void __launch_bounds__(256)
k_splitk_reduce(const double* __restrict__ partial, int nsplit, int64_t M, int64_t N, double alpha, double beta,
                double* __restrict__ C, int64_t ldc, const int* __restrict__ skip) {
  if (skip && *skip) return;
  const int64_t total = M * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    double s = 0.0;
#pragma unroll 8
    for (int z = 0; z < nsplit; ++z) s += partial[(int64_t)z * total + i];
    double* p = C + (i / N) * ldc + (i % N);
    s *= alpha;
    if (beta != 0.0) s = fma(beta, *p, s);
    *p = s;
  }
}

inline int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

}  // namespace

cudaError_t sdgemm(int ta, int64_t M, int64_t N, int64_t K, double alpha, const float* A, int64_t lda, const float* B,
                   int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  return product64(ta, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s);
}

cudaError_t fdgemm(int ta, int64_t M, int64_t N, int64_t K, double alpha, const float* A, int64_t lda, const double* B,
                   int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  return product64(ta, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s);
}

cudaError_t dgemm(int ta, int tb, int64_t M, int64_t N, int64_t K, double alpha, const double* A,
                  int64_t lda, const double* B, int64_t ldb, double beta, double* C, int64_t ldc,
                  cudaStream_t s) {
  return dgemm_ex(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, 1, nullptr, nullptr, s);
}

cudaError_t dgemm_ex(int ta, int tb, int64_t M, int64_t N, int64_t K, double alpha, const double* A,
                     int64_t lda, const double* B, int64_t ldb, double beta, double* C, int64_t ldc,
                     int nsplit, double* partial, const int* skip, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (nsplit < 1 || !partial) nsplit = 1;
  const int64_t k_per_split = std::max<int64_t>(16, cdiv(cdiv(K, nsplit), 16) * 16);      // whole stages
  nsplit = (int)cdiv(std::max<int64_t>(K, 1), k_per_split);
  cudaError_t e = dgemm64(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, nsplit, k_per_split, partial, skip, s);
  if (e == cudaSuccess && nsplit > 1) {
    const int64_t blocks = cdiv(M * N, 256);
    k_splitk_reduce<<<(unsigned)(blocks < 1184 ? blocks : 1184), 256, 0, s>>>(partial, nsplit, M, N, alpha, beta, C, ldc, skip);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace br
