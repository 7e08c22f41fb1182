// fp64-accurate products on the int8 tensor cores: C = X Y (fp64 result of fp32 operands), for the power products F Q of a
// refresh.
//
// C = (X S^-1) (S Y) with S a diagonal of powers of two (below).  Every row of X S^-1 and every column of S Y is scaled by a power
// of two so that its largest entry lies below 1, rounded to 54 bits and cut into seven signed 8-bit digits, most significant first:
// x = 2^(e - 6) sum_s 2^(-8 s) d_s.  (Splitting a product into exact low-precision ones is Ozaki, Ogita, Oishi and Rump's
// error-free transformation, Numer. Algorithms 2012; integer digits and integer accumulators for it: Ootomo, Ozaki and
// Yokota, 2023.)  The products of digits i and j with i + j = d share a scale, so one integer accumulator per d adds them up
// without rounding, and
//   C = 2^(ex + ey - 12) sum_{d < 8} 2^(-8 d) sum_{i + j = d} X_i Y_j,
// 34 products of the 49.  What is lost is relative to the largest entries of a row of X S^-1 and of a column of S Y, not to the
// terms themselves as in an fp64 sum: the rounding of entries more than 2^30 smaller than those, at 2^-55, and the digit
// products left out, each at most 2^(-12 - 64 + 14) = 2^-62 (a digit reaches 128) and five with i + j = 8 in a step, so less than
// 2^-59 K, typically 2^-64 sqrt(K), times the two maxima.
//   That has to stay below the rounding of an fp64 sum, 2^-53 of its partial sums, also where the parameters behind a factor F = X
// have gradients of different size: |F_ik| <= sqrt(F_ii F_kk), so with S_kk = 2^(half the exponent of F_kk) the rows of F S^-1 are
// balanced whatever the sizes, and the columns of S Q are where Q tracks F.  Errors of the columns, relative to their lengths, rms at
// order 393: fp64 sums in order, these digits, and without S and without the products with i + j = 7 (28 of the 49): independent
// entries, tracked 1.0e-15, 5.2e-17, 6e-15; a low-rank signal a hundred times the noise, tracked 5.0e-12, 4.6e-14, 9e-12;
// gradient rows over 10^-4, tracked 4.1e-13, 1.5e-14, 4e-8.
//
// A CTA computes one 128 x 64 tile: eight 128 x 64 accumulators take all 512 columns of tensor memory, and 128 x 64
// is the widest tile for which they fit.  A stage holds all seven digit planes of both operands for 64 steps of the
// contraction (86 KB, one TMA load each), from which 34 x 2 instructions of 128 x 64 x 32 are issued.  An instruction takes 32 cycles, so
// the loops over digits are unrolled: with the addresses worked out in a loop the issuing thread was the bound.  Eight products of
// order 1536 and eight of 1152: 1191 us, 2012 in a loop (1528 with 28 digit products in a loop), and 417 for the digits:
// 51 TFLOP/s of fp64-accurate arithmetic in all, the fp64 unit 26.
#include <cuda.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "br_internal.h"
#include "tc_ptx.h"

namespace br {
namespace {

constexpr int kS = 7, kD = 8;                     // digits, and scales of their products
constexpr int kBM = 128, kBN = 64, kBK = 64;
constexpr int kPlaneA = kBM * kBK, kPlaneB = kBN * kBK;
constexpr int kStage = kS * (kPlaneA + kPlaneB), kStages = 2;
constexpr int kSmem = kStages * kStage + 1024;
constexpr int kThreads = 192;                     // warp 0: TMA, warp 1: MMA, warps 2..5: epilogue
constexpr int kGroup = 8;                         // products of one launch

inline size_t al256(size_t x) { return (x + 255) / 256 * 256; }
inline int64_t padk(int64_t K) { return (K + 15) / 16 * 16; }

// ---- digits ---------------------------------------------------------------------------------------------------------
constexpr int kNotFinite = 1 << 20, kZero = -kNotFinite;
// the e with |x| < 2^e <= 2 |x|
__device__ __forceinline__ int exponent_of(float x) {
  const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
  if (u >= 0x7f800000u) return kNotFinite;
  return u >= 0x00800000u ? (int)(u >> 23) - 126 : u ? 32 - __clz((int)u) - 149 : kZero;
}
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + e) << 20, 0); }       // |e| <= 1022
// Scale of a row (column) with entries below 2^e: x 2^up rounds to its 54-bit integer, down * (digit sums) is its value; an
// entry that is not finite (`e` from kNotFinite / 2 on) makes the factor, and with it the row (column) of the product, NaN.
__device__ __forceinline__ bool scale_of(int e, int* up, double* down) {
  const bool finite = e < kNotFinite / 2;
  if (!finite || e < kZero / 2) e = 0;
  *up = 8 * kS - 2 - e;
  *down = finite ? pow2(e - 6) : __longlong_as_double(0x7ff8000000000000ll);
  return finite;
}
// The digits of four entries, plane s in p[s + 1], a byte per entry.  Digits in [-128, 127] are the bytes of the integer with 128
// added at each place, less 128; the leading one needs no bias.  (Taken off one by one with 64-bit shifts, 16 products of orders 1536
// and 1152: 484 us for the splits, 344 like this.)
__device__ __forceinline__ void transpose4(const uint32_t (&a)[4], uint32_t* out) {          // out[3 - j]: byte j of the four
  const uint32_t t0 = __byte_perm(a[0], a[1], 0x5140), t1 = __byte_perm(a[0], a[1], 0x7362);
  const uint32_t u0 = __byte_perm(a[2], a[3], 0x5140), u1 = __byte_perm(a[2], a[3], 0x7362);
  out[3] = __byte_perm(t0, u0, 0x5410); out[2] = __byte_perm(t0, u0, 0x7632);
  out[1] = __byte_perm(t1, u1, 0x5410); out[0] = __byte_perm(t1, u1, 0x7632);
}
__device__ __forceinline__ void digits4(const float (&x)[4], const int (&up)[4], uint32_t (&p)[kS + 1]) {
  static_assert(kS == 7, "a digit per byte of the integer, the topmost byte unused");
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    constexpr unsigned long long bias = 0x0000808080808080ull;
    const unsigned long long v = ((unsigned long long)__double2ll_rn((double)x[u] * pow2(up[u])) + bias) ^ bias;
    hi[u] = (uint32_t)(v >> 32); lo[u] = (uint32_t)v;
  }
  transpose4(hi, p);
  transpose4(lo, p + 4);
}

// The exponents of S: half of those of the diagonal of X, 0 where an entry is not positive and finite or there is no diagonal.
// A CTA per product.  (Gathered by every CTA of the two splits instead, 8 + 8 products of orders 1536 and 1152: 524 us for the splits.)
struct InnerJobs { const float* diag[kGroup]; int64_t stride[kGroup]; signed char* inner[kGroup]; int K[kGroup]; };
__global__ void __launch_bounds__(512) k_oz_inner(const __grid_constant__ InnerJobs g) {
  const int job = blockIdx.x;
  const float* const diag = g.diag[job];
  for (int k = threadIdx.x; k < (g.K[job] + 15) / 16 * 16; k += blockDim.x) {
    const float f = diag && k < g.K[job] ? diag[(int64_t)k * g.stride[job]] : 0.f;
    const int e = exponent_of(f);
    g.inner[job][k] = (signed char)(f > 0.f && e < kNotFinite ? e >> 1 : 0);
  }
}

struct SplitJobs {
  const float* src[kGroup];
  const signed char* inner[kGroup];
  unsigned char* planes[kGroup];
  double* factor[kGroup];
  int R[kGroup], K[kGroup], begin[kGroup + 1], n;
};

// Rows of a row-major matrix (R x K, leading dimension K): a warp per row, four entries per lane and step.
__global__ void __launch_bounds__(256) k_oz_rows(const __grid_constant__ SplitJobs g) {
  const int gw = (int)blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  int job = 0;
  while (job + 1 < g.n && g.begin[job + 1] <= gw) ++job;
  const int row = gw - g.begin[job], K = g.K[job], Kp = (K + 15) / 16 * 16;
  if (row >= g.R[job]) return;
  const signed char* const inner = g.inner[job];
  const float* x = g.src[job] + (int64_t)row * K;
  int m = kZero;
#pragma unroll 8
  for (int k = lane; k < K; k += 32) m = max(m, exponent_of(x[k]) - inner[k]);
  m = __reduce_max_sync(0xffffffffu, m);
  int up;
  double down;
  const bool finite = scale_of(m, &up, &down);
  if (lane == 0) g.factor[job][row] = down;
  const int64_t plane = (int64_t)g.R[job] * Kp;
  for (int k = 4 * lane; k < Kp; k += 128) {
    const char4 c = *reinterpret_cast<const char4*>(inner + k);
    const int e[4] = {up - c.x, up - c.y, up - c.z, up - c.w};
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = finite && k + u < K ? x[k + u] : 0.f;
    uint32_t d[kS + 1];
    digits4(v, e, d);
#pragma unroll
    for (int s = 0; s < kS; ++s) *reinterpret_cast<uint32_t*>(g.planes[job] + s * plane + (int64_t)row * Kp + k) = d[s + 1];
  }
}

// Columns of a row-major matrix (K x R, leading dimension R), written with the contraction contiguous: a CTA of 1024 threads
// per 32 columns, transposed through shared memory 256 steps at a time (order 1536: 47 us on 256 threads, latency of its loads; two
// CTAs of 512 threads on an SM are a third slower).
constexpr int kColThreads = 1024, kColStep = 256;
__global__ void __launch_bounds__(kColThreads) k_oz_cols(const __grid_constant__ SplitJobs g) {
  __shared__ float tile[kColStep][33];
  int job = 0;
  while (job + 1 < g.n && g.begin[job + 1] <= (int)blockIdx.x) ++job;
  const int R = g.R[job], K = g.K[job], Kp = (K + 15) / 16 * 16, c0 = ((int)blockIdx.x - g.begin[job]) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const float* x = g.src[job];
  const signed char* const inner = g.inner[job];
  int m = kZero;
  if (c0 + tx < R)
#pragma unroll 8
    for (int k = ty; k < K; k += 32) m = max(m, exponent_of(x[(int64_t)k * R + c0 + tx]) + inner[k]);
  tile[ty][tx] = __int_as_float(m);
  __syncthreads();
  // this thread's column when it writes: 32 threads to a column, 8 steps of the contraction each
  const int wc = threadIdx.x >> 5, wk = (threadIdx.x & 31) * 8;
  m = __reduce_max_sync(0xffffffffu, __float_as_int(tile[threadIdx.x & 31][wc]));
  int up;
  double down;
  const bool finite = scale_of(m, &up, &down);
  if (c0 + wc < R && wk == 0) g.factor[job][c0 + wc] = down;
  const int64_t plane = (int64_t)R * Kp;
  for (int k0 = 0; k0 < Kp; k0 += kColStep) {
    __syncthreads();
#pragma unroll
    for (int k = ty; k < kColStep; k += 32) tile[k][tx] = (k0 + k < K && c0 + tx < R) ? x[(int64_t)(k0 + k) * R + c0 + tx] : 0.f;
    __syncthreads();
    if (c0 + wc >= R || k0 + wk >= Kp) continue;  // (Kp is a multiple of 8)
    uint32_t d[2][kS + 1];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const char4 c = *reinterpret_cast<const char4*>(inner + k0 + wk + 4 * h);
      const int e[4] = {up + c.x, up + c.y, up + c.z, up + c.w};
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = finite ? tile[wk + 4 * h + u][wc] : 0.f;
      digits4(v, e, d[h]);
    }
#pragma unroll
    for (int s = 0; s < kS; ++s)
      *reinterpret_cast<uint2*>(g.planes[job] + s * plane + (int64_t)(c0 + wc) * Kp + k0 + wk) = make_uint2(d[0][s + 1], d[1][s + 1]);
  }
}

// ---- product --------------------------------------------------------------------------------------------------------
struct Prob { CUtensorMap a, b; const double *fa, *fb; double* C; int M, N, K, tiles_n, tile0; };
struct Probs { Prob p[kGroup]; int n; int* status; };

__device__ __forceinline__ void umma_i8(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// K-major operand, 64-byte swizzle: rows of 64 bytes, groups of eight rows 512 bytes apart
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (uint64_t)(512 >> 4) << 32 | 1ull << 46 | 4ull << 61;
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1) k_oz_gemm(const __grid_constant__ Probs g) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ alignas(8) uint64_t bars[2 * kStages + 1];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word, dead_word;
  volatile int* abort_flag = &abort_word;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int pi = 0;
  while (pi + 1 < g.n && g.p[pi + 1].tile0 <= (int)blockIdx.x) ++pi;
  const Prob& p = g.p[pi];
  const int tile = (int)blockIdx.x - p.tile0, m0 = tile / p.tiles_n * kBM, n0 = tile % p.tiles_n * kBN;
  const int nk = (p.K + kBK - 1) / kBK;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u, bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kStages + s); };
  const uint32_t done = bar0 + 8u * (2 * kStages);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
    mbar_init(done, 1);
    abort_word = 0;
    dead_word = *reinterpret_cast<volatile int*>(g.status) < 0;      // an earlier launch failed: nothing to do
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  if (!dead_word) {
    if (warp == 0) {
      if (lane == 0) {
        for (int kb = 0; kb < nk; ++kb) {
          const int s = kb % kStages;
          if (!mbar_wait(empty(s), ((kb / kStages) & 1) ^ 1, abort_flag, g.status)) break;
          mbar_expect_tx(full(s), kStage);
          tma_load_3d(base + s * kStage, &p.a, full(s), kb * kBK, m0, 0);
          tma_load_3d(base + s * kStage + kS * kPlaneA, &p.b, full(s), kb * kBK, n0, 0);
        }
        outlast_copies(abort_flag);
      }
    } else if (warp == 1) {
      if (lane == 0) {
        // signed 8-bit operands, 32-bit integer accumulators, 128 x 64, both operands K-major
        const uint32_t idesc = 2u << 4 | 1u << 7 | 1u << 10 | (uint32_t)(kBN >> 3) << 17 | (uint32_t)(kBM >> 4) << 24;
        bool ok = true;
        for (int kb = 0; kb < nk; ++kb) {
          const int s = kb % kStages;
          if (!mbar_wait(full(s), (kb / kStages) & 1, abort_flag, g.status)) { ok = false; break; }
          tc_fence_after();
          const uint64_t a = desc64(base + s * kStage), b = desc64(base + s * kStage + kS * kPlaneA);
#pragma unroll
          for (int d = 0; d < kD; ++d)
#pragma unroll
            for (int i = d < kS ? 0 : d - kS + 1; i <= (d < kS ? d : kS - 1); ++i)
#pragma unroll
              for (int k = 0; k < kBK / 32; ++k)
                umma_i8(tmem + d * kBN, a + (uint64_t)((i * kPlaneA + 32 * k) >> 4), b + (uint64_t)(((d - i) * kPlaneB + 32 * k) >> 4), idesc,
                        kb > 0 || i > (d < kS ? 0 : d - kS + 1) || k > 0);
          umma_commit(empty(s));
        }
        if (ok) umma_commit(done);
      }
    } else {
      // a thread per row, eight columns at a time: the eight sums in order of their weight, smallest first
      const int quad = warp & 3, row = m0 + quad * 32 + lane;
      if (mbar_wait(done, 0, abort_flag, g.status)) {
        tc_fence_after();
        const double fa = row < p.M ? p.fa[row] : 0.0;
        for (int c0 = 0; c0 < kBN && n0 + c0 < p.N; c0 += 8) {
          int acc[kD][8];
          __syncwarp();
#pragma unroll
          for (int d = 0; d < kD; ++d) tmem_ld8(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(d * kBN + c0), acc[d]);
          tmem_wait_ld();
          double* c = p.C + (int64_t)row * p.N + n0 + c0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            double v = (double)acc[kD - 1][j];
#pragma unroll
            for (int d = kD - 2; d >= 0; --d) v = fma(v, 1.0 / 256.0, (double)acc[d][j]);
            if (row < p.M && n0 + c0 + j < p.N) c[j] = v * (fa * __ldg(p.fb + n0 + c0 + j));
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// ---- host -----------------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

bool encode(CUtensorMap* map, void* planes, int64_t R, int64_t Kp, int box_rows) {
  const EncodeTiledFn enc = reinterpret_cast<EncodeTiledFn>(tensor_map_encoder());
  if (!enc) return false;
  cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)R, (cuuint64_t)kS}, strides[2] = {(cuuint64_t)Kp, (cuuint64_t)(Kp * R)};
  cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)box_rows, (cuuint32_t)kS}, estr[3] = {1u, 1u, 1u};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, planes, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// planes and factors of one operand
size_t operand_bytes(int64_t R, int64_t K) { return al256((size_t)kS * R * padk(K)) + al256(sizeof(double) * R); }
size_t inner_bytes(int64_t K) { return al256(padk(K)); }

}  // namespace

size_t oz_scratch_bytes(int64_t M, int64_t N, int64_t K) { return operand_bytes(M, K) + operand_bytes(N, K) + inner_bytes(K); }

// The integer sums of a contraction of up to 2^14 steps cannot overflow (seven products of at most 2^14 each a step).
bool oz_eligible(int64_t M, int64_t N, int64_t K) { return M >= 1 && N >= 1 && K >= 1 && K <= (1 << 14) && M <= (1 << 14) && N <= (1 << 14); }

cudaError_t oz_product_group(const OzProduct* v, int n, char* scratch, size_t bytes, int* status, cudaStream_t s, int* launches) {
  static OncePerDevice once;
  cudaError_t e = once.run([] { return cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem); });
  if (e != cudaSuccess) return e;
  for (int first = 0; first < n;) {
    InnerJobs inner;
    SplitJobs rows, cols;
    Probs g;
    std::memset(&g, 0, sizeof g);
    rows.n = cols.n = 0;
    rows.begin[0] = cols.begin[0] = 0;
    g.status = status;
    size_t used = 0;
    int tiles = 0, i = 0;
    for (; i < kGroup && first + i < n; ++i) {
      const OzProduct& q = v[first + i];
      if (!oz_eligible(q.M, q.N, q.K)) return cudaErrorInvalidValue;
      const size_t need = oz_scratch_bytes(q.M, q.N, q.K);
      if (used + need > bytes) break;
      Prob& p = g.p[i];
      char* at = scratch + used;
      const size_t pa = al256((size_t)kS * q.M * padk(q.K)), pb = al256((size_t)kS * q.N * padk(q.K));
      unsigned char* A = reinterpret_cast<unsigned char*>(at);
      double* fa = reinterpret_cast<double*>(at + pa);
      unsigned char* B = reinterpret_cast<unsigned char*>(at + operand_bytes(q.M, q.K));
      double* fb = reinterpret_cast<double*>(at + operand_bytes(q.M, q.K) + pb);
      used += need;
      if (!encode(&p.a, A, q.M, padk(q.K), kBM) || !encode(&p.b, B, q.N, padk(q.K), kBN)) return cudaErrorInvalidValue;
      p.fa = fa; p.fb = fb; p.C = q.C; p.M = (int)q.M; p.N = (int)q.N; p.K = (int)q.K;
      p.tiles_n = (int)((q.N + kBN - 1) / kBN); p.tile0 = tiles;
      tiles += p.tiles_n * (int)((q.M + kBM - 1) / kBM);
      inner.diag[i] = q.diag; inner.stride[i] = q.stride; inner.K[i] = (int)q.K;
      rows.inner[i] = cols.inner[i] = inner.inner[i] = reinterpret_cast<signed char*>(at + operand_bytes(q.M, q.K) + operand_bytes(q.N, q.K));
      rows.src[i] = q.X; rows.planes[i] = A; rows.factor[i] = fa; rows.R[i] = (int)q.M; rows.K[i] = (int)q.K;
      rows.begin[i + 1] = rows.begin[i] + (int)((q.M + 7) / 8 * 8);
      cols.src[i] = q.Y; cols.planes[i] = B; cols.factor[i] = fb; cols.R[i] = (int)q.N; cols.K[i] = (int)q.K;
      cols.begin[i + 1] = cols.begin[i] + (int)((q.N + 31) / 32);
    }
    if (i == 0) return cudaErrorInvalidValue;     // (scratch smaller than one product)
    rows.n = cols.n = g.n = i;
    k_oz_inner<<<(unsigned)i, 512, 0, s>>>(inner);
    k_oz_rows<<<(unsigned)(rows.begin[i] / 8), 256, 0, s>>>(rows);
    k_oz_cols<<<(unsigned)cols.begin[i], kColThreads, 0, s>>>(cols);
    k_oz_gemm<<<(unsigned)tiles, kThreads, kSmem, s>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (launches) *launches += 4;
    first += i;
  }
  return cudaSuccess;
}

}  // namespace br
