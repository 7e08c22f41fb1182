// fp64-accurate products on the int8 tensor cores: C = X Y (fp64 result of fp32 operands), for the power products F Q of a
// refresh.
//
// Every row of X and every column of Y is scaled by a power of two so that its largest entry lies below 1, rounded to
// 54 bits and cut into seven signed 8-bit digits, most significant first: x = 2^(e - 6) sum_s 2^(-8 s) d_s.  (Splitting a
// product into exact low-precision ones is Ozaki, Ogita, Oishi and Rump's error-free transformation, Numer. Algorithms
// 2012; integer digits and integer accumulators for it: Ootomo, Ozaki and Yokota, 2023.)  The products of digits i and j
// with i + j = d share a scale, so one integer accumulator per d adds them up without rounding, and
//   C = 2^(ex + ey - 12) sum_{d < 7} 2^(-8 d) sum_{i + j = d} X_i Y_j,
// 28 products of the 49; those with i + j >= 7 lie below 2^-56 of the scale.  What is lost is the rounding of entries
// that are more than 2^30 smaller than the largest of their row (or column), at 2^-54 of that one, and the terms left
// out: of the size of the rounding of an fp64 sum.
//
// A CTA computes one 128 x 64 tile: seven 128 x 64 accumulators take 448 of the 512 columns of tensor memory, and 128 x 64
// is the widest tile for which they fit.  A stage holds all seven digit planes of both operands for 64 steps of the
// contraction (86 KB, one TMA load each), from which 28 x 2 instructions of 128 x 64 x 32 are issued.  Two products of order 1536
// take 327 us, 44 TFLOP/s of fp64-accurate arithmetic (the fp64 unit: 26 on the same operands), of order 1024 115 us; with
// consecutive instructions into different accumulators 356 and 126.
#include <cuda.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "br_internal.h"
#include "tc_ptx.h"

namespace br {
namespace {

constexpr int kS = 7;                             // digits
constexpr int kBM = 128, kBN = 64, kBK = 64;
constexpr int kPlaneA = kBM * kBK, kPlaneB = kBN * kBK;
constexpr int kStage = kS * (kPlaneA + kPlaneB), kStages = 2;
constexpr int kSmem = kStages * kStage + 1024;
constexpr int kThreads = 192;                     // warp 0: TMA, warp 1: MMA, warps 2..5: epilogue
constexpr int kGroup = 8;                         // products of one launch

inline size_t al256(size_t x) { return (x + 255) / 256 * 256; }
inline int64_t padk(int64_t K) { return (K + 15) / 16 * 16; }

// ---- digits ---------------------------------------------------------------------------------------------------------
// scale of a row (column) whose largest magnitude is m: x * up rounds to its 54-bit integer, down * (digit sums) is its
// value; entries that are not finite make the factor, and with it the row (column) of the product, NaN
__device__ __forceinline__ void scale_of(float m, double* up, double* down) {
  if (!(m < __int_as_float(0x7f800000))) { *up = 0.0; *down = __longlong_as_double(0x7ff8000000000000ll); return; }
  int e = 0;
  if (m > 0.f) frexpf(m, &e);                     // m < 2^e
  *up = scalbn(1.0, 8 * kS - 2 - e);
  *down = scalbn(1.0, e - 6);
}
// the larger magnitude, NaN if either is
__device__ __forceinline__ float max_or_nan(float a, float b) { return a != a || b != b ? __int_as_float(0x7fc00000) : fmaxf(a, b); }
__device__ __forceinline__ void digits(float x, double up, unsigned char (&d)[kS]) {
  long long v = __double2ll_rn((double)x * up);
#pragma unroll
  for (int s = kS - 1; s >= 0; --s) {
    const signed char c = (signed char)(v & 0xff);
    d[s] = (unsigned char)c;
    v = (v - c) >> 8;
  }
}

struct SplitJobs { const float* src[kGroup]; unsigned char* planes[kGroup]; double* factor[kGroup]; int R[kGroup], K[kGroup], begin[kGroup + 1], n; };

// Rows of a row-major matrix (R x K, leading dimension K): a warp per row, four entries per lane and step.
__global__ void __launch_bounds__(256) k_oz_rows(const __grid_constant__ SplitJobs g) {
  const int gw = (int)blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  int job = 0;
  while (job + 1 < g.n && g.begin[job + 1] <= gw) ++job;
  const int row = gw - g.begin[job], K = g.K[job], Kp = (K + 15) / 16 * 16;
  if (row >= g.R[job]) return;
  const float* x = g.src[job] + (int64_t)row * K;
  float m = 0.f;
#pragma unroll 8
  for (int k = lane; k < K; k += 32) m = max_or_nan(m, fabsf(x[k]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max_or_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
  double up, down;
  scale_of(m, &up, &down);
  if (lane == 0) g.factor[job][row] = down;
  const int64_t plane = (int64_t)g.R[job] * Kp;
  for (int k = 4 * lane; k < Kp; k += 128) {
    unsigned char d[4][kS];
#pragma unroll
    for (int u = 0; u < 4; ++u) digits(up != 0.0 && k + u < K ? x[k + u] : 0.f, up, d[u]);
#pragma unroll
    for (int s = 0; s < kS; ++s)
      *reinterpret_cast<uchar4*>(g.planes[job] + s * plane + (int64_t)row * Kp + k) = make_uchar4(d[0][s], d[1][s], d[2][s], d[3][s]);
  }
}

// Columns of a row-major matrix (K x R, leading dimension R), written with the contraction contiguous: a CTA of 1024 threads
// per 32 columns, transposed through shared memory 256 steps at a time (order 1536: 47 us on 256 threads, latency of its loads).
constexpr int kColThreads = 1024, kColStep = 256;
__global__ void __launch_bounds__(kColThreads) k_oz_cols(const __grid_constant__ SplitJobs g) {
  __shared__ float tile[kColStep][33];
  int job = 0;
  while (job + 1 < g.n && g.begin[job + 1] <= (int)blockIdx.x) ++job;
  const int R = g.R[job], K = g.K[job], Kp = (K + 15) / 16 * 16, c0 = ((int)blockIdx.x - g.begin[job]) * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const float* x = g.src[job];
  float m = 0.f;
  if (c0 + tx < R)
#pragma unroll 8
    for (int k = ty; k < K; k += 32) m = max_or_nan(m, fabsf(x[(int64_t)k * R + c0 + tx]));
  tile[ty][tx] = m;
  __syncthreads();
  // this thread's column when it writes: 32 threads to a column, 8 steps of the contraction each
  const int wc = threadIdx.x >> 5, wk = (threadIdx.x & 31) * 8;
  m = tile[threadIdx.x & 31][wc];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max_or_nan(m, __shfl_xor_sync(0xffffffffu, m, o));
  double up, down;
  scale_of(m, &up, &down);
  if (c0 + wc < R && wk == 0) g.factor[job][c0 + wc] = down;
  const int64_t plane = (int64_t)R * Kp;
  for (int k0 = 0; k0 < Kp; k0 += kColStep) {
    __syncthreads();
#pragma unroll
    for (int k = ty; k < kColStep; k += 32) tile[k][tx] = (k0 + k < K && c0 + tx < R) ? x[(int64_t)(k0 + k) * R + c0 + tx] : 0.f;
    __syncthreads();
    if (c0 + wc >= R || k0 + wk >= Kp) continue;  // (Kp is a multiple of 8)
    uint2 d[kS];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      unsigned char c[kS];
      digits(up != 0.0 ? tile[wk + u][wc] : 0.f, up, c);
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        uint32_t& w = u < 4 ? d[s].x : d[s].y;
        w = (u & 3) ? w | (uint32_t)c[s] << (8 * (u & 3)) : c[s];
      }
    }
#pragma unroll
    for (int s = 0; s < kS; ++s) *reinterpret_cast<uint2*>(g.planes[job] + s * plane + (int64_t)(c0 + wc) * Kp + k0 + wk) = d[s];
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
      if (lane == 0)
        for (int kb = 0; kb < nk; ++kb) {
          const int s = kb % kStages;
          if (!mbar_wait(empty(s), ((kb / kStages) & 1) ^ 1, abort_flag, g.status)) break;
          mbar_expect_tx(full(s), kStage);
          tma_load_3d(base + s * kStage, &p.a, full(s), kb * kBK, m0, 0);
          tma_load_3d(base + s * kStage + kS * kPlaneA, &p.b, full(s), kb * kBK, n0, 0);
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
#pragma unroll 1
          for (int d = 0; d < kS; ++d)
            for (int i = 0; i <= d; ++i)
#pragma unroll
              for (int k = 0; k < kBK / 32; ++k)
                umma_i8(tmem + d * kBN, a + (uint64_t)((i * kPlaneA + 32 * k) >> 4), b + (uint64_t)(((d - i) * kPlaneB + 32 * k) >> 4), idesc,
                        kb > 0 || i > 0 || k > 0);
          umma_commit(empty(s));
        }
        if (ok) umma_commit(done);
      }
    } else {
      // a thread per row, eight columns at a time: the seven sums in order of their weight, smallest first
      const int quad = warp & 3, row = m0 + quad * 32 + lane;
      if (mbar_wait(done, 0, abort_flag, g.status)) {
        tc_fence_after();
        const double fa = row < p.M ? p.fa[row] : 0.0;
        for (int c0 = 0; c0 < kBN && n0 + c0 < p.N; c0 += 8) {
          int acc[kS][8];
          __syncwarp();
#pragma unroll
          for (int d = 0; d < kS; ++d) tmem_ld8(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(d * kBN + c0), acc[d]);
          tmem_wait_ld();
          double* c = p.C + (int64_t)row * p.N + n0 + c0;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            double v = (double)acc[kS - 1][j];
#pragma unroll
            for (int d = kS - 2; d >= 0; --d) v = fma(v, 1.0 / 256.0, (double)acc[d][j]);
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

}  // namespace

size_t oz_scratch_bytes(int64_t M, int64_t N, int64_t K) { return operand_bytes(M, K) + operand_bytes(N, K); }

// The integer sums of a contraction of up to 2^14 steps cannot overflow (seven products of at most 2^14 each a step).
bool oz_eligible(int64_t M, int64_t N, int64_t K) { return M >= 1 && N >= 1 && K >= 1 && K <= (1 << 14) && M <= (1 << 14) && N <= (1 << 14); }

cudaError_t oz_product_group(const OzProduct* v, int n, char* scratch, size_t bytes, int* status, cudaStream_t s, int* launches) {
  static OncePerDevice once;
  cudaError_t e = once.run([] { return cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem); });
  if (e != cudaSuccess) return e;
  for (int first = 0; first < n;) {
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
      rows.src[i] = q.X; rows.planes[i] = A; rows.factor[i] = fa; rows.R[i] = (int)q.M; rows.K[i] = (int)q.K;
      rows.begin[i + 1] = rows.begin[i] + (int)((q.M + 7) / 8 * 8);
      cols.src[i] = q.Y; cols.planes[i] = B; cols.factor[i] = fb; cols.R[i] = (int)q.N; cols.K[i] = (int)q.K;
      cols.begin[i + 1] = cols.begin[i] + (int)((q.N + 31) / 32);
    }
    if (i == 0) return cudaErrorInvalidValue;     // (scratch smaller than one product)
    rows.n = cols.n = g.n = i;
    k_oz_rows<<<(unsigned)(rows.begin[i] / 8), 256, 0, s>>>(rows);
    k_oz_cols<<<(unsigned)cols.begin[i], kColThreads, 0, s>>>(cols);
    k_oz_gemm<<<(unsigned)tiles, kThreads, kSmem, s>>>(g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (launches) *launches += 3;
    first += i;
  }
  return cudaSuccess;
}

}  // namespace br
