// Orthonormalisation Q <- qr(A).Q (positive diagonal of R, fp64) by one thread-block cluster.
//
// The factorisation of qr.cu (recursive block Gram-Schmidt over panels that are orthonormalised by
// Cholesky-QR) is a chain of hundreds of short dependent steps: Gram matrix, Cholesky factor and its
// inverse, panel update, projection coefficients, projection.  As launches of their own they cost more
// in launch gaps than in work: at order 384, 248 launches of which 44 did something, 950 us a basis.
// Here one cluster of up to 16 CTAs walks the whole chain of a basis, or of a range of its columns, in one launch, and the
// steps are separated by the cluster's hardware barrier; the second sweep and the completion of a
// rank-deficient product are branches instead of cancelled launches.  Measured, one basis alone: order 64
// 32 us, 384 214 us, 1024 1.28 ms, 1536 3.6 ms; stand-alone Power() at order 384 1368 -> 242 us.
//
//  * Rows of A are dealt to the CTAs in contiguous chunks.  A CTA computes its rows' share of a panel's
//    Gram matrix and applies R^-1 and the projections to its own rows only, so these steps need no
//    barrier between them.  Only the Gram sums and the projection coefficients cross CTAs.
//  * The Gram shares stay in shared memory: every CTA adds up one slice of rows over all shares (fixed
//    order, through distributed shared memory) and writes it into every CTA, and after a second barrier each
//    computes the 64 x 64 Cholesky factor and its inverse for itself.  The redundant factorisation costs
//    nothing (the other CTAs would wait for it) and saves the broadcast, and since all of them see the
//    same bits, every decision (second pass, second sweep, completion) is taken alike without a word
//    exchanged.
//  * Projection coefficients Q_l^T A_r: one 64 x 64 tile per CTA, the contraction split over several CTAs
//    when there are fewer tiles than CTAs (partial sums through distributed shared memory, fixed order).
//
// Products run on the fp64 matrix unit (mma.sync.m8n8k4.f64): 64 x 64 tiles, a warp 16 rows x 32 columns,
// 16-deep stages, three of them in flight with cp.async.  95 KiB of shared memory and 128 registers, two CTAs
// per SM, so that the clusters of several bases share SMs and one cluster's barriers are another's work.
// Other CTAs write A and C while the kernel runs: plain loads are ordered by the acquire of the barrier
// behind those writes, and none goes through the read-only path.
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "br_internal.h"

namespace cg = cooperative_groups;

namespace br {
namespace {

constexpr int kT = 256;                       // threads per CTA
constexpr int kW = kOrthPanel;                // panel width
constexpr int kKs = 16;                       // contraction depth of a stage
// Leading dimensions of staged tiles, 4 mod 16 doubles: the fragment loads of a half-warp (4 x 4 or
// 4 contraction steps x 4 rows) then touch 16 different 8-byte banks.
constexpr int kLdK = 68;                      // [contraction][64]
constexpr int kLdI = 20;                      // [64][16 contraction steps]
constexpr int kOper = 64 * kLdI;              // doubles of a staged first operand (either layout)
constexpr int kOperB = kKs * kLdK;            // and of the second
constexpr int kStages = 3;
constexpr int kLdP = 72;                      // partial sums (16-byte stores of a quarter-warp: 8 different banks)
constexpr int kMaxCluster = 16;
constexpr int kStageD = kStages * (kOper + kOperB);   // operand stages; also one 64 x 64 tile of A (ld 68)
constexpr int kPartD = 64 * kLdP;             // partial sums of this CTA, later R^-T (ld 68)
// One shared-memory array, carved at compile time (pointers kept in a structure would make every access a
// generic one behind a reload of the pointer).
extern __shared__ double sm[];
constexpr int oStage = 0, oPart = oStage + kStageD, oDiag0 = oPart + kPartD, oFloor = oDiag0 + 64,
              oPiv = oFloor + 64, oN0 = oPiv + 64, kSmemD = oN0 + 64;
constexpr int kSmemBytes = kSmemD * (int)sizeof(double);
static_assert(kStageD >= 64 * kLdK && kOper >= kOperB, "staging area");

__device__ __forceinline__ void dmma(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(c0), "+d"(c1) : "d"(a), "d"(b));
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// A 64 x 64 tile on 8 warps, 16 rows x 32 columns each: entry e of a thread's accumulator (mi = e / 8,
// ni = e / 2 % 4) sits at row tile_row() + 8 mi, column tile_col() + 8 ni + e % 2 (8 x 64 per warp needs half
// as much again from shared memory).  The warps of a scheduler take different rows, so that a short tile still
// uses all four; with SYM only the 8 x 8 blocks on and above the diagonal are computed, and the warps are
// paired so that the schedulers get 8 to 10 of the 36 blocks.
template <bool SYM>
__device__ __forceinline__ int warp_m() {
  const int w = threadIdx.x >> 5;
  return SYM ? (0x31322010 >> (4 * w)) & 3 : w >> 1;       // per warp, from warp 0 up: 0 1 0 2 2 3 1 3
}
template <bool SYM>
__device__ __forceinline__ int warp_n() {
  const int w = threadIdx.x >> 5;
  return SYM ? (0x8B >> w) & 1 : w & 1;                    // 1 1 0 1 0 0 0 1
}
template <bool SYM> __device__ __forceinline__ int tile_row() { return 16 * warp_m<SYM>() + ((threadIdx.x & 31) >> 2); }
template <bool SYM> __device__ __forceinline__ int tile_col() { return 32 * warp_n<SYM>() + 2 * (threadIdx.x & 3); }

// One stage (16 contraction steps) of acc += (or -=, NEG) a b.  I: rows of the tile that exist.
// BT: the second operand is staged [64][contraction] like a first operand that is not DIRECT.
template <bool DIRECT, bool SYM, bool NEG, bool BT = false>
__device__ __forceinline__ void mma_stage(double (&acc)[16], const double* As, const double* Bs, int I) {
  const int lane = threadIdx.x & 31, g = lane >> 2, tig = lane & 3, wm = warp_m<SYM>(), wn = warp_n<SYM>();
  As += DIRECT ? tig * kLdK + 16 * wm + g : (16 * wm + g) * kLdI + tig;
  Bs += BT ? (32 * wn + g) * kLdI + tig : tig * kLdK + 32 * wn + g;
  if (16 * wm >= I || (SYM && 4 * wn + 3 < 2 * wm)) return;
  const bool two = 16 * wm + 8 < I;
#pragma unroll
  for (int k4 = 0; k4 < kKs; k4 += 4) {
    double a0 = As[DIRECT ? k4 * kLdK : k4], a1 = As[DIRECT ? k4 * kLdK + 8 : 8 * kLdI + k4];
    if (NEG) { a0 = -a0; a1 = -a1; }
    double b[4];
#pragma unroll
    for (int ni = 0; ni < 4; ++ni) b[ni] = Bs[BT ? 8 * ni * kLdI + k4 : k4 * kLdK + 8 * ni];
#pragma unroll
    for (int ni = 0; ni < 4; ++ni)
      if (!SYM || 4 * wn + ni >= 2 * wm) dmma(acc[2 * ni], acc[2 * ni + 1], a0, b[ni]);
    if (two) {
#pragma unroll
      for (int ni = 0; ni < 4; ++ni)
        if (!SYM || 4 * wn + ni >= 2 * wm + 1) dmma(acc[8 + 2 * ni], acc[9 + 2 * ni], a1, b[ni]);
    }
  }
}
// 16 or 8 bytes from global to shared memory, zero when !ok (the rows of an odd order are 8-byte aligned only)
template <bool VEC>
__device__ __forceinline__ void copy_async(double* dst, const double* src, bool ok) {
  if (VEC)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 16 : 0) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 8 : 0) : "memory");
}
// acc += sum over kk < K of a(i, kk) b(kk, j), i < I <= 64, j < J <= 64 (NEG: -=).
//   DIRECT: a(i, kk) = X[kk * lda + i]   otherwise a(i, kk) = X[i * lda + kk];   b(kk, j) = Y[kk * ldb + j].
//   BT: b(kk, j) = Y[j * ldb + kk].
// VEC: all dimensions and leading dimensions that a copy runs along are even, and X and Y 16-byte aligned.
template <bool VEC, bool DIRECT, bool SYM, bool NEG, bool BT = false>
__device__ __forceinline__ void mm64(double (&acc)[16], const double* X, int64_t lda, int I, const double* Y, int64_t ldb, int J, int K) {
  constexpr int V = VEC ? 2 : 1, N = 4 / V;                // doubles per copy; copies per thread, operand and stage
  const int t = threadIdx.x;
  // thread -> first element of an operand tile, and the distance of its next one
  constexpr int RK = kT / (64 / V), RI = kT / (kKs / V);   // rows of a [16][64] / [64][16] tile covered by one copy per thread
  constexpr int STAGE = kOper + (BT ? kOper : kOperB);
  const int dk = t / (64 / V), di = t % (64 / V) * V, sk = t % (kKs / V) * V, si = t / (kKs / V);   // [16][64] and [64][16] tiles
  const int ak = DIRECT ? dk : sk, ai = DIRECT ? di : si, bk = BT ? sk : dk, bj = BT ? si : di;
  const double* px = X + (DIRECT ? (int64_t)ak * lda + ai : (int64_t)ai * lda + ak);
  const double* py = Y + (BT ? (int64_t)bj * ldb + bk : (int64_t)bk * ldb + bj);
  const int64_t xq = (DIRECT ? RK : RI) * lda, xs = DIRECT ? kKs * lda : kKs, yq = (BT ? RI : RK) * ldb, ys = BT ? kKs : kKs * ldb;
  double* const dA = sm + oStage + (DIRECT ? ak * kLdK + ai : ai * kLdI + ak);
  double* const dB = sm + oStage + kOper + (BT ? bj * kLdI + bk : bk * kLdK + bj);
  const int nk = (K + kKs - 1) / kKs;
  auto fetch = [&](int s) {
    const int k0 = s * kKs, buf = (s % kStages) * STAGE;
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const bool ok = DIRECT ? (ai < I && k0 + ak + q * RK < K) : (ai + q * RI < I && k0 + ak < K);
      copy_async<VEC>(dA + buf + (DIRECT ? q * RK * kLdK : q * RI * kLdI), ok ? px + q * xq : X, ok);
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const bool ok = BT ? (bj + q * RI < J && k0 + bk < K) : (bj < J && k0 + bk + q * RK < K);
      copy_async<VEC>(dB + buf + (BT ? q * RI * kLdI : q * RK * kLdK), ok ? py + q * yq : Y, ok);
    }
    px += xs; py += ys;
  };
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < nk) fetch(s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int buf = 0;
  for (int s = 0; s < nk; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();                             // stage s is in place, and stage s - 1 has been read
    if (s + kStages - 1 < nk) fetch(s + kStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const double* st = sm + oStage + buf * STAGE;
    mma_stage<DIRECT, SYM, NEG, BT>(acc, st, st + kOper, I);
    if (++buf == kStages) buf = 0;
  }
  __syncthreads();
}
__device__ __forceinline__ void clear(double (&acc)[16]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) acc[i] = 0.0;
}
// the entries of a tile that exist: f(row, column, value)
template <typename FN>
__device__ __forceinline__ void each_entry(double (&acc)[16], int I, int J, FN f) {
  const int r = tile_row<false>(), c = tile_col<false>();
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const int row = r + 8 * (e >> 3), col = c + 8 * ((e >> 1) & 3) + (e & 1);
    if (row < I && col < J) f(row, col, acc[e]);
  }
}

// acc += sum over kk < K of x(i, kk) y(kk, j) on one tile, i < I, j < J, with X fp32 and Y fp32 or fp64, widened while
// they are staged through registers: x(i, kk) = X[kk * lda + i] (TRANS) or X[i * lda + kk], y(kk, j) = Y[kk * ldb + j].
// Two stages of loads are in flight; the tile ends behind a barrier, so the stages' memory is free again.
template <bool TRANS, typename TB>
__device__ __forceinline__ void product_tile(double (&acc)[16], const float* X, int64_t lda, int I, const TB* Y, int64_t ldb, int J, int K) {
  const int t = threadIdx.x;
  float ra[2][4];
  TB rb[2][4];
  auto load = [&](int k0, float (&a)[4], TB (&b)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = TRANS ? (t & 63) : (t >> 4) + 16 * q, ka = k0 + (TRANS ? (t >> 6) + 4 * q : (t & 15));
      const int j = t & 63, kb = k0 + (t >> 6) + 4 * q;
      a[q] = (i < I && ka < K) ? X[TRANS ? (int64_t)ka * lda + i : (int64_t)i * lda + ka] : 0.f;
      b[q] = (j < J && kb < K) ? Y[(int64_t)kb * ldb + j] : (TB)0;
    }
  };
  auto store = [&](int buf, const float (&a)[4], const TB (&b)[4]) {
    double* As = sm + oStage + buf * (kOper + kOperB);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      As[TRANS ? ((t >> 6) + 4 * q) * kLdK + (t & 63) : ((t >> 4) + 16 * q) * kLdI + (t & 15)] = (double)a[q];
      As[kOper + ((t >> 6) + 4 * q) * kLdK + (t & 63)] = (double)b[q];
    }
  };
  const int nk = (K + kKs - 1) / kKs;
  load(0, ra[0], rb[0]);
  load(kKs, ra[1], rb[1]);
  store(0, ra[0], rb[0]);
  __syncthreads();
  for (int s = 0; s < nk; s += 2) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (u && s + 1 >= nk) break;
      load((s + u + 2) * kKs, ra[u], rb[u]);
      const double* st = sm + oStage + u * (kOper + kOperB);
      mma_stage<TRANS, false, false>(acc, st, st + kOper, I);
      store(1 - u, ra[1 - u], rb[1 - u]);
      __syncthreads();
    }
  }
}
constexpr int kProductSmem = 2 * (kOper + kOperB) * (int)sizeof(double);

// C = alpha op(X) Y + beta C: one 64 x 64 tile per CTA, for the products of a refresh with an fp32 operand.  A refresh
// from the momentum (two such products), ms, with tiles of 128 x 128 on one CTA per SM and with these: 2048 x 2048 7.8 and
// 4.2, 4096 x 4096 27.2 and 20.9, 2560 x 6912 16.1 and 11.4, factorisation included.
template <bool TRANS, typename TB>
__global__ void __launch_bounds__(kT, 2)
k_product64(int M, int N, int K, double alpha, const float* __restrict__ X, int64_t lda, const TB* __restrict__ Y, int64_t ldb,
            double beta, double* __restrict__ C, int64_t ldc) {
  const int m0 = (int)blockIdx.y * 64, n0 = (int)blockIdx.x * 64;
  double acc[16];
  clear(acc);
  product_tile<TRANS>(acc, X + (TRANS ? m0 : (int64_t)m0 * lda), lda, M - m0, Y + n0, ldb, N - n0, K);
  each_entry(acc, M - m0, N - n0, [&](int i, int j, double v) {
    double* c = C + (int64_t)(m0 + i) * ldc + n0 + j;
    v *= alpha;
    *c = beta != 0.0 ? fma(beta, *c, v) : v;
  });
}

// A = F Q (fp32 in, fp64 out, k x k) for several bases in one launch, one tile per cluster of 1 to 8 CTAs that share its
// contraction: the partial sums are added through distributed shared memory in the order of the ranges.  One of order 384
// 15.4 us; 24 us as 36 CTAs with the whole contraction each.
template <int NJ> struct ProductGroup { const float *F[NJ], *Q[NJ]; double* A[NJ]; int k[NJ], tile0[NJ + 1], n; };
template <int NJ>
__global__ void __launch_bounds__(kT, 2) k_product_group(const __grid_constant__ ProductGroup<NJ> g) {
  cg::cluster_group cl = cg::this_cluster();
  const int zs = (int)cl.num_blocks(), z = (int)cl.block_rank(), tile = (int)blockIdx.x / zs;
  int p = 0;
  while (p + 1 < g.n && g.tile0[p + 1] <= tile) ++p;
  const int k = g.k[p], nt = (k + 63) / 64, m0 = (tile - g.tile0[p]) / nt * 64, n0 = (tile - g.tile0[p]) % nt * 64;
  const int kc = ((k + zs - 1) / zs + kKs - 1) / kKs * kKs, k0 = min(k, z * kc), K = min(kc, k - k0);
  const int I = min(64, k - m0), J = min(64, k - n0);
  double* const C = g.A[p] + (int64_t)m0 * k + n0;
  double acc[16];
  clear(acc);
  product_tile<false>(acc, g.F[p] + (int64_t)m0 * k + k0, k, I, g.Q[p] + (int64_t)k0 * k + n0, k, J, K);
  if (zs == 1) {
    each_entry(acc, I, J, [&](int i, int j, double v) { C[(int64_t)i * k + j] = v; });
    return;
  }
  each_entry(acc, 64, 64, [&](int i, int j, double v) { sm[i * kLdP + j] = v; });
  cluster_sync();
  const int rows = 64 / zs;
  for (int e = threadIdx.x; e < rows * 64; e += kT) {
    const int i = z * rows + (e >> 6), j = e & 63;
    double s = 0.0;
    for (int q = 0; q < zs; ++q) s += cl.map_shared_rank(sm, q)[i * kLdP + j];
    if (i < I && j < J) C[(int64_t)i * k + j] = s;
  }
  cluster_sync();                              // no CTA leaves while another may still read its partial sums
}
static_assert(64 * kLdP * (int)sizeof(double) <= kProductSmem, "the partial sums borrow the stages");

// C = alpha op(X) op(Y) + beta C in fp64, one 64 x 64 tile and a range of the contraction per CTA (split over
// blockIdx.z: partial sums, added by a second kernel).
template <bool VEC, bool TRANS, bool BT>
__global__ void __launch_bounds__(kT, 2)
k_dgemm64(int M, int N, int K, double alpha, const double* X, int64_t lda, const double* Y, int64_t ldb, double beta, double* C,
          int64_t ldc, int k_per_split, double* partial, const int* skip) {
  if (skip && *skip) return;            // uniform: a device-side flag cancels the whole launch
  const int m0 = (int)blockIdx.y * 64, n0 = (int)blockIdx.x * 64, k0 = (int)blockIdx.z * k_per_split;
  double acc[16];
  clear(acc);
  mm64<VEC, TRANS, false, false, BT>(acc, X + (TRANS ? (int64_t)k0 * lda + m0 : (int64_t)m0 * lda + k0), lda, min(64, M - m0),
                                     Y + (BT ? (int64_t)n0 * ldb + k0 : (int64_t)k0 * ldb + n0), ldb, min(64, N - n0), min(k_per_split, K - k0));
  const bool split = gridDim.z > 1;
  each_entry(acc, M - m0, N - n0, [&](int i, int j, double v) {
    if (split) { partial[((int64_t)blockIdx.z * M + m0 + i) * N + n0 + j] = v; return; }
    double* c = C + (int64_t)(m0 + i) * ldc + n0 + j;
    v *= alpha;
    *c = beta != 0.0 ? fma(beta, *c, v) : v;
  });
}
constexpr int kDgemmSmem = kStages * 2 * kOper * (int)sizeof(double);

template <bool VEC, bool TRANS, bool BT>
cudaError_t launch_dgemm(dim3 grid, int64_t M, int64_t N, int64_t K, double alpha, const double* A, int64_t lda, const double* B,
                         int64_t ldb, double beta, double* C, int64_t ldc, int64_t k_per_split, double* partial, const int* skip,
                         cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t e = once.run([] { return cudaFuncSetAttribute(k_dgemm64<VEC, TRANS, BT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kDgemmSmem); });
  if (e != cudaSuccess) return e;
  k_dgemm64<VEC, TRANS, BT><<<grid, kT, kDgemmSmem, s>>>((int)M, (int)N, (int)K, alpha, A, lda, B, ldb, beta, C, ldc, (int)k_per_split,
                                                        partial, skip);
  return cudaGetLastError();
}

template <typename TB>
cudaError_t launch_product(int ta, int64_t M, int64_t N, int64_t K, double alpha, const float* A, int64_t lda, const TB* B,
                           int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t s) {
  const dim3 grid((unsigned)((N + 63) / 64), (unsigned)((M + 63) / 64));
  const size_t bytes = kProductSmem;
  if (ta)
    k_product64<true, TB><<<grid, kT, bytes, s>>>((int)M, (int)N, (int)K, alpha, A, lda, B, ldb, beta, C, ldc);
  else
    k_product64<false, TB><<<grid, kT, bytes, s>>>((int)M, (int)N, (int)K, alpha, A, lda, B, ldb, beta, C, ldc);
  return cudaGetLastError();
}

struct PartArgs {                // columns [j0, j0 + w) of one sweep over the k x k matrix A, row-major
  double* A; int64_t k;
  int j0, w;
  int first;                     // this is the first sweep (watch the column norms)
  double ill_ratio;              // first: squared-norm ratio below which the second sweep has to run
  const double* norm0;           // first: squared norms of the columns before any projection
  double *C, *rdiag;             // projection coefficients; squared diagonal of R
  int* status; int* flags; const int* skip;
};
// The complete factorisations of several products: both sweeps, rank decision, completion, outputs.
template <int NJ> struct OrthGroup { OrthJob j[NJ]; int* status; };

struct Ctx {
  int64_t k;
  double* A;
  int rank, cs, r0, r1;
};

// Cholesky factor S = R^T R of the panel's Gram matrix (bw <= 64) and its inverse, as R^-T (ld 68), in the
// area of the partial sums.
//
// Blocks of 8 x 8 in shared memory; block row c of [S | I] is solved with R_cc (forward substitution, a column
// per thread) and subtracted, times R_ci^T, from the rows i below (matrix unit).  Column block j of S is dead
// once block row j is done, and column block j of the identity's part is still a unit block until then, so
// both share one 64 x 64 array.  The chain is bound by the 8 x 8 factorisations: warp 0 alone updates the
// next diagonal block and factors it in registers (every lane the same: no shuffles, 8 dependent square
// roots), while the other warps update the rest, all of a warp's blocks at once (a block row to a warp took as long as two
// factorisations).  Two barriers a block instead of one a pivot: 27 us with a barrier a pivot and the matrix in registers,
// 20 us with two pivots a barrier, 13.3 us with a block row to a warp.
// (Multiplying block row c by an explicit R_cc^-T instead loses the factorisation of a panel with a condition
// number of 1e6, such as a completed rank-deficient product has: its error, 1e-16 times the condition number,
// swamps pivots of 1e-12.  Substitution is backward stable like the unblocked elimination.)
// The pivots end up at oPiv, the Gram diagonal at oDiag0.
constexpr int oZ = oStage, oX = oZ + 64 * kLdK, oD = oX + 8 * kLdK;      // (in the operand stages)
static_assert(64 * kLdK + 8 * kLdK + 8 * 8 + 8 <= kStageD, "the factorisation borrows the operand stages");

// The blocks that step c updates with block row c - 1, its own diagonal block excepted: rows i >= c, columns j > i, j = i
// and (the identity's part) j < c.  Entries beyond the count are valid blocks whose result is dropped.
struct Updates { unsigned char ij[8][35]; unsigned char n[8]; };
constexpr Updates make_updates() {
  Updates u = {};
  for (int c = 1; c < 8; ++c)
    for (int i = c; i < 8; ++i)
      for (int j = 0; j < 8; ++j)
        if (j < c || j > i || (j == i && i > c)) u.ij[c][u.n[c]++] = (unsigned char)(8 * i + j);
  return u;
}
__constant__ const Updates kUpdates = make_updates();

// The diagonal block at Z (upper triangle) -> R_cc at oD (row-major 8 x 8), 1 / diagonal behind it, pivots at oPiv + 8 c
__device__ __forceinline__ void factor8(const double* Z, int c) {
  const int lane = threadIdx.x & 31;
  double u[8][8], inv[8], piv[8], fl[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) fl[i] = sm[oFloor + 8 * c + i];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = i; j < 8; ++j) u[i][j] = Z[i * kLdK + j];
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    piv[p] = u[p][p] > fl[p] ? u[p][p] : fl[p];
    inv[p] = rsqrt(piv[p]);
#pragma unroll
    for (int j = p + 1; j < 8; ++j) u[p][j] *= inv[p];
#pragma unroll
    for (int i = p + 1; i < 8; ++i)
#pragma unroll
      for (int j = i; j < 8; ++j) u[i][j] = fma(-u[p][i], u[p][j], u[i][j]);
  }
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
      for (int j = i + 1; j < 8; ++j) sm[oD + 8 * i + j] = u[i][j];
      sm[oD + 64 + i] = inv[i];
      sm[oPiv + 8 * c + i] = piv[i];
    }
  }
}

__device__ __noinline__ void chol64(int bw) {
  const int t = threadIdx.x, w = t >> 5, lane = t & 31, g = lane >> 2, tig = lane & 3;
  const int nb = (bw + 7) / 8;
  double* const Z = sm + oZ;
  double* const RT = sm + oPart;
  if (t < 64) {
    const double d = Z[t * kLdK + t], f = d * 1e-24;
    sm[oDiag0 + t] = d;
    sm[oFloor + t] = f > 1e-300 ? f : 1e-300;        // a pivot at or below this is clamped
  }
  __syncthreads();
#pragma unroll 1
  for (int c = 0; c < nb; ++c) {
    if (w == 0) {
      if (c > 0) {
        // block (c, c) <- itself - R_{c-1,c}^T R_{c-1,c}, and its factorisation
        double2* z = reinterpret_cast<double2*>(Z + (8 * c + g) * kLdK + 8 * c + 2 * tig);
        double2 d = *z;
#pragma unroll
        for (int k4 = 0; k4 < 8; k4 += 4) {
          const double x = sm[oX + (k4 + tig) * kLdK + g + 8 * c];
          dmma(d.x, d.y, -x, x);
        }
        *z = d;
        __syncwarp();
      }
      factor8(Z + 8 * c * kLdK + 8 * c, c);
    } else if (c > 0) {
      // the other blocks (i, j) of rows to come <- themselves - R_{c-1,i}^T X_j, with block row c - 1 of R | R^-T in oX:
      // at most 34, dealt to seven warps, all of a warp's in flight at once
      constexpr int U = 5;
      double2 d[U];
      int bi[U], bj[U];
      bool ok[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = w - 1 + 7 * u, ij = kUpdates.ij[c][e];
        bi[u] = ij >> 3; bj[u] = ij & 7;
        ok[u] = e < kUpdates.n[c] && max(bi[u], bj[u]) < nb;
        d[u] = *reinterpret_cast<const double2*>(Z + (8 * bi[u] + g) * kLdK + 8 * bj[u] + 2 * tig);
      }
#pragma unroll
      for (int k4 = 0; k4 < 8; k4 += 4)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const double* x = sm + oX + (k4 + tig) * kLdK + g;
          dmma(d[u].x, d[u].y, -x[8 * bi[u]], x[8 * bj[u]]);
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (ok[u]) *reinterpret_cast<double2*>(Z + (8 * bi[u] + g) * kLdK + 8 * bj[u] + 2 * tig) = d[u];
    }
    __syncthreads();
    // block row c: R right of the diagonal, R^-T up to it
    if (t < 8 * nb) {
      double x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = (t >> 3) == c ? ((t & 7) == i ? 1.0 : 0.0) : Z[(8 * c + i) * kLdK + t];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        x[i] *= sm[oD + 64 + i];
#pragma unroll
        for (int m = i + 1; m < 8; ++m) x[m] = fma(-sm[oD + 8 * i + m], x[i], x[m]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) sm[oX + i * kLdK + t] = x[i];
      if ((t >> 3) <= c) {
#pragma unroll
        for (int i = 0; i < 8; ++i) RT[(8 * c + i) * kLdK + t] = x[i];
      }
    }
    __syncthreads();
  }
}

// own rows of columns [j0, j0 + bw) <- own rows * R^-1 (upper triangular)
__device__ __noinline__ void apply_rinv(const Ctx q, int j0, int bw) {
  const int t = threadIdx.x, lane = t & 31, g = lane >> 2, tig = lane & 3;
  double pre[16];
  auto load = [&](int r) {
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int i = (t >> 6) + 4 * u, kk = t & 63;
      pre[u] = (r + i < q.r1 && kk < bw) ? __ldcg(q.A + (int64_t)(r + i) * q.k + j0 + kk) : 0.0;
    }
  };
  if (q.r0 < q.r1) load(q.r0);
  for (int r = q.r0; r < q.r1; r += 64) {
#pragma unroll
    for (int u = 0; u < 16; ++u) sm[oStage + ((t >> 6) + 4 * u) * kLdK + (t & 63)] = pre[u];
    __syncthreads();
    if (r + 64 < q.r1) load(r + 64);
    const int wm = warp_m<false>(), wn = warp_n<false>();
    if (r + 16 * wm < q.r1) {
      double acc[16];
      clear(acc);
      const double* As = sm + oStage + (16 * wm + g) * kLdK + tig;
      const double* Bs = sm + oPart + (32 * wn + g) * kLdK + tig;
#pragma unroll
      for (int k4 = 0; k4 < 64; k4 += 4) {
        if (k4 >= 32 && wn == 0) break;                // R^-1 is upper triangular
        const double a0 = As[k4], a1 = As[8 * kLdK + k4];
#pragma unroll
        for (int ni = 0; ni < 4; ++ni)
          if (k4 < 32 ? (wn == 1 || k4 <= 8 * ni + 7) : k4 - 32 <= 8 * ni + 7) {
            const double b = Bs[8 * ni * kLdK + k4];
            dmma(acc[2 * ni], acc[2 * ni + 1], a0, b);
            dmma(acc[8 + 2 * ni], acc[9 + 2 * ni], a1, b);
          }
      }
      each_entry(acc, q.r1 - r, bw, [&](int i, int j, double v) { q.A[(int64_t)(r + i) * q.k + j0 + j] = v; });
    }
    __syncthreads();
  }
}

// A[:, jt : jt + wt] -= Q (Q^T A[:, jt : jt + wt]), Q = A[:, jp : jp + wp] orthonormal, wp a multiple of 64.
template <bool VEC>
__device__ __noinline__ void project64(const Ctx q, double* C, int jp, int wp, int jt, int wt) {
  const int t = threadIdx.x;
  const int ntp = (wp + 63) / 64, ntt = (wt + 63) / 64, tiles = ntp * ntt;
  double acc[16];
  cluster_sync();                                       // every CTA's rows of both blocks are written
  // A tile per CTA while there are as many left; of fewer, as many as are a power of two at a time, their contractions
  // shared (nine tiles on 16 CTAs: eight on two CTAs each, then one on all, 9 / 16 of the time of one tile instead of all of it)
  for (int done = 0; done < tiles;) {
    const int left = tiles - done, n = left >= q.cs ? q.cs : 1 << (31 - __clz(left)), sp = q.cs / n;
    const int tile = done + q.rank / sp, split = q.rank % sp;
    const int i0 = (tile / ntt) * 64, c0 = (tile % ntt) * 64, I = min(64, wp - i0), J = min(64, wt - c0);
    const int kc = ((int)((q.k + sp - 1) / sp) + kKs - 1) / kKs * kKs, k0 = min((int)q.k, split * kc), kn = min(kc, (int)q.k - k0);
    clear(acc);
    mm64<VEC, true, false, false>(acc, q.A + (int64_t)k0 * q.k + jp + i0, q.k, I, q.A + (int64_t)k0 * q.k + jt + c0, q.k, J, kn);
    if (sp == 1) {
      each_entry(acc, I, J, [&](int i, int j, double v) { C[(int64_t)(i0 + i) * wt + c0 + j] = v; });
    } else {
      each_entry(acc, 64, 64, [&](int i, int j, double v) { sm[oPart + i * kLdP + j] = v; });
      cluster_sync();
      for (int e = split * kT + t; e < 64 * 64; e += sp * kT) {
        const int i = e >> 6, j = e & 63;
        double s = 0.0;
#pragma unroll 4
        for (int z = 0; z < sp; ++z) s += cg::this_cluster().map_shared_rank(sm + oPart, q.rank - split + z)[i * kLdP + j];
        if (i < I && j < J) C[(int64_t)(i0 + i) * wt + c0 + j] = s;
      }
      if (done + n < tiles) cluster_sync();             // before the partial sums are overwritten
    }
    done += n;
  }
  cluster_sync();
  for (int r = q.r0; r < q.r1; r += 64)
    for (int c0 = 0; c0 < wt; c0 += 64) {
      const int I = min(64, q.r1 - r), J = min(64, wt - c0);
      // the accumulator starts from A itself: its loads overlap the first copies
      double* p = q.A + (int64_t)r * q.k + jt + c0;
      clear(acc);
      each_entry(acc, I, J, [&](int i, int j, double& v) { v = __ldcg(p + (int64_t)i * q.k + j); });
      mm64<VEC, false, false, true>(acc, q.A + (int64_t)r * q.k + jp, q.k, I, C + c0, wt, J, wp);
      each_entry(acc, I, J, [&](int i, int j, double v) { p[(int64_t)i * q.k + j] = v; });
    }
  __syncthreads();
}

// What one sweep over the columns found (alike in every CTA).
struct SweepNotes { bool ill = false, tc_bad = false, clamped = false; };

// Cholesky-QR of the panel [j0, j0 + bw), repeated once unless every column kept kOrthPassRatio of its
// squared norm against the panel's columns before it.
template <bool VEC>
__device__ __forceinline__ void panel64(const Ctx& q, int j0, int bw, bool first, double ill_ratio, double* rdiag, bool rdiag_init,
                                        SweepNotes& notes) {
  const int t = threadIdx.x;
  for (int pass = 0; pass < 2; ++pass) {
    double acc[16];
    const double* P = q.A + (int64_t)q.r0 * q.k + j0;
    clear(acc);
    mm64<VEC, true, true, false>(acc, P, q.k, bw, P, q.k, bw, max(0, q.r1 - q.r0));
    {
      // (a warp whose blocks all lie below the diagonal writes zeros nobody reads)
      const int row = tile_row<true>(), col = tile_col<true>();
#pragma unroll
      for (int e = 0; e < 16; e += 2)
        *reinterpret_cast<double2*>(sm + oPart + (row + 8 * (e >> 3)) * kLdP + col + 8 * ((e >> 1) & 3)) = make_double2(acc[e], acc[e + 1]);
    }
    // the summed matrix at oZ of every CTA: its upper block triangle, the identity beyond the panel, zero elsewhere
    auto entry = [&](int i, int j, double v) { return max(i, j) >= bw ? (i == j ? 1.0 : 0.0) : j >= (i & ~7) ? v : 0.0; };
    if (q.cs > 1) {
      cluster_sync();
      const int rs = 64 / q.cs;
      for (int e = t; e < rs * 64; e += kT) {
        const int i = q.rank * rs + (e >> 6), j = e & 63;
        double s = 0.0;
#pragma unroll 8
        for (int z = 0; z < q.cs; ++z) s += cg::this_cluster().map_shared_rank(sm + oPart, z)[i * kLdP + j];
        s = entry(i, j, s);
#pragma unroll 8
        for (int z = 0; z < q.cs; ++z) cg::this_cluster().map_shared_rank(sm + oZ, z)[i * kLdK + j] = s;
      }
      cluster_sync();
    } else {
      __syncthreads();
      for (int e = t; e < 64 * 64; e += kT) sm[oZ + (e >> 6) * kLdK + (e & 63)] = entry(e >> 6, e & 63, sm[oPart + (e >> 6) * kLdP + (e & 63)]);
      __syncthreads();
    }
    chol64(bw);
    // what the pivots say: pivot / Gram diagonal is the squared sine of the angle between a column and the
    // span of the panel's columns before it
    bool low = false, ill = false, bad = false, cl = false;
    if (t < bw) {
      const double piv = sm[oPiv + t], d0 = sm[oDiag0 + t];
      low = !(d0 > 0.0 && piv >= kOrthPassRatio * d0);
      cl = !(piv > sm[oFloor + t]);
      if (first && pass == 0) { ill = d0 < ill_ratio * sm[oN0 + t]; bad = d0 < kOrthTcRatio * sm[oN0 + t]; }
      if (q.rank == 0 && rdiag) rdiag[j0 + t] = (rdiag_init && pass == 0) ? piv : __ldcg(rdiag + j0 + t) * piv;
    }
    low = __syncthreads_or(low); notes.ill |= __syncthreads_or(ill) != 0;
    notes.tc_bad |= __syncthreads_or(bad) != 0; notes.clamped |= __syncthreads_or(cl) != 0;
    apply_rinv(q, j0, bw);
    if (!low) break;
  }
}

// One sweep over the columns [j0, j0 + w): the recursion "orthonormalise the left half, project it out of
// the right half, orthonormalise the right half" in the order of its panels.  The node whose right part
// starts at panel l is projected right before that panel.
template <bool VEC>
__device__ __forceinline__ SweepNotes sweep64(const Ctx& q, double* C, int j0, int w, bool first, double ill_ratio, const double* norm0,
                                              int norm_parts, double* rdiag, bool rdiag_init) {
  SweepNotes notes;
  const int nl = (w + kW - 1) / kW;
  for (int l = 0; l < nl; ++l) {
    if (l > 0) {
      int lo = 0, n = nl, h;
      while (true) {
        h = (n + 1) / 2;
        if (l == lo + h) break;
        if (l < lo + h) n = h; else { lo += h; n -= h; }
      }
      project64<VEC>(q, C, j0 + lo * kW, h * kW, j0 + l * kW, min(n * kW, w - lo * kW) - h * kW);
    }
    const int c0 = j0 + l * kW, bw = min(kW, j0 + w - c0);
    if (first && (int)threadIdx.x < bw) {
      double s = 0.0;
      for (int z = 0; z < norm_parts; ++z) s += __ldcg(norm0 + (int64_t)z * q.k + c0 + threadIdx.x);
      sm[oN0 + threadIdx.x] = s;
    }
    panel64<VEC>(q, c0, bw, first, ill_ratio, rdiag, rdiag_init, notes);
  }
  return notes;
}

__device__ __forceinline__ Ctx context(double* A, int64_t k) {
  Ctx q;
  q.k = k; q.A = A;
  q.cs = (int)cg::this_cluster().num_blocks(); q.rank = (int)cg::this_cluster().block_rank();
  const int rc = (((int)k + q.cs - 1) / q.cs + 7) / 8 * 8;
  q.r0 = min((int)k, q.rank * rc); q.r1 = min((int)k, q.r0 + rc);
  return q;
}

template <bool VEC>
__global__ void __launch_bounds__(kT, 2) k_orth_part(PartArgs a) {
  if (a.skip && *a.skip) return;               // uniform: a device-side flag cancels the whole launch
  const Ctx q = context(a.A, a.k);
  const SweepNotes n = sweep64<VEC>(q, a.C, a.j0, a.w, a.first != 0, a.ill_ratio, a.norm0, 1, a.rdiag, false);
  if (q.rank == 0 && threadIdx.x == 0) {
    if (n.clamped) { atomicMax(a.status, (int)BR_WARN_RANK_DEFICIENT); a.flags[3] = 1; }
    if (a.first && n.ill) a.flags[1] = 0;
    if (a.first && n.tc_bad) a.flags[2] = 0;
  }
  cluster_sync();                              // no CTA leaves while another may still read its shared memory
}

// own rows of A <- own rows of F Qprev (a deficient product once more, before it is completed)
__device__ __noinline__ void own_product(const Ctx q, const float* F, const float* Q) {
  const int k = (int)q.k;
  for (int r = q.r0; r < q.r1; r += 64)
    for (int c = 0; c < k; c += 64) {
      double acc[16];
      clear(acc);
      product_tile<false>(acc, F + (int64_t)r * k, k, min(64, q.r1 - r), Q + c, k, min(64, k - c), k);
      each_entry(acc, min(64, q.r1 - r), min(64, k - c), [&](int i, int j, double v) { q.A[(int64_t)(r + i) * k + c + j] = v; });
    }
  __syncthreads();
}

template <bool VEC>
__device__ __forceinline__ void orth_whole_cluster(const OrthJob& a, int* status) {
  const Ctx q = context(a.A, a.k);
  const int k = (int)a.k, t = threadIdx.x;
  bool clamped = false, tc_bad = false, deficient = false;
  const bool fix = a.Qprev != nullptr && (a.Acopy != nullptr || a.F != nullptr) && !a.complete;
  for (int attempt = 0; attempt < 2; ++attempt) {
    double* normp = a.normp + (int64_t)attempt * q.cs * k;
    if (attempt && !a.complete && a.F) own_product(q, a.F, a.Qprev);
    const double* from = attempt && a.Acopy && !a.complete ? a.Acopy : q.A;
    for (int j = t; j < k; j += kT) {
      double s = 0.0;
      if (!attempt) {
        // (rows come in eights: eight loads in flight)
        for (int r = q.r0; r < q.r1; r += 8) {
          double v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] = r + u < q.r1 ? __ldcg(q.A + (int64_t)(r + u) * k + j) : 0.0;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (fix && a.Acopy && r + u < q.r1) a.Acopy[(int64_t)(r + u) * k + j] = v[u];
            s = fma(v[u], v[u], s);
          }
        }
      } else {
        // complete the product from the current basis: A_j + 1e-6 ||A_j|| Q_j (a zero column becomes Q_j)
        double n2 = 0.0;
        for (int z = 0; z < q.cs; ++z) n2 += __ldcg(a.normp + (int64_t)z * k + j);
        const double d = n2 > 0.0 ? kOrthCompletion * sqrt(n2) : 1.0;
        for (int r = q.r0; r < q.r1; ++r) {
          const int64_t i = (int64_t)r * k + j;
          const double v = fma(d, (double)a.Qprev[i], __ldcg(from + i));
          q.A[i] = v;
          s = fma(v, v, s);
        }
      }
      normp[(int64_t)q.rank * k + j] = s;
    }
    cluster_sync();
    if (a.complete && !attempt) continue;        // known to be short of rank: completed before the first sweep
    double* const rdiag = fix && !attempt ? a.rdiag : nullptr;
    SweepNotes n = sweep64<VEC>(q, a.C, 0, k, true, kOrthIllRatio, normp, q.cs, rdiag, true);
    clamped |= n.clamped;
    if (!attempt || a.complete) tc_bad = n.tc_bad;
    if (n.ill) {
      n = sweep64<VEC>(q, a.C, 0, k, false, 0.0, nullptr, 0, rdiag, false);
      clamped |= n.clamped;
    }
    if (!fix || attempt) break;
    // rank decision on the squared diagonal of R: deficient when some |R_jj| <= 1e-12 max |R_kk|
    cluster_sync();
    double lo = 1e300, hi = 0.0;
    for (int j = t; j < k; j += kT) {
      const double v = __ldcg(a.rdiag + j);
      lo = v > 0.0 ? fmin(lo, v) : 0.0; hi = fmax(hi, v);
    }
    sm[oStage + t] = lo; sm[oStage + kT + t] = hi;
    __syncthreads();
    for (int s = kT / 2; s > 0; s >>= 1) {
      if (t < s) {
        sm[oStage + t] = fmin(sm[oStage + t], sm[oStage + t + s]);
        sm[oStage + kT + t] = fmax(sm[oStage + kT + t], sm[oStage + kT + t + s]);
      }
      __syncthreads();
    }
    deficient = !(sm[oStage] > 1e-24 * sm[oStage + kT]);
    __syncthreads();
    if (!deficient) break;
  }
  // the result in fp32 and, for the tensor-core path, as a bf16 pair (own rows)
  for (int64_t i0 = (int64_t)q.r0 * k; i0 < (int64_t)q.r1 * k; i0 += 8 * kT) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) { const int64_t i = i0 + u * kT + t; x[u] = i < (int64_t)q.r1 * k ? (float)__ldcg(q.A + i) : 0.f; }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int64_t i = i0 + u * kT + t;
      if (i >= (int64_t)q.r1 * k) break;
      a.Qout[i] = x[u];
      if (a.Qh) {
        const __nv_bfloat16 h = __float2bfloat16_rn(x[u]);
        a.Qh[i] = h;
        a.Ql[i] = __float2bfloat16_rn(x[u] - __bfloat162float(h));
      }
    }
  }
  if (q.rank == 0 && t == 0) {
    if (clamped || deficient || a.complete) atomicMax(status, (int)BR_WARN_RANK_DEFICIENT);
    // bit 0: no column shrank below 1e-3 of its length; bit 1: numerically rank-deficient
    if (a.cond_out) *a.cond_out = (tc_bad ? 0 : 1) | (clamped || deficient ? 2 : 0);
  }
  cluster_sync();
}
template <int NJ>
__global__ void __launch_bounds__(kT, 2) k_orth_group(const __grid_constant__ OrthGroup<NJ> g) {
  const OrthJob& a = g.j[blockIdx.x / cg::this_cluster().num_blocks()];
  // 16-byte copies need even dimensions throughout (the buffers start on 256-byte boundaries)
  if (a.k % 2 == 0) orth_whole_cluster<true>(a, g.status); else orth_whole_cluster<false>(a, g.status);
}

// Largest cluster the device schedules for this kernel (16 needs the non-portable size), per device.
int max_cluster() {
  static int cap[64] = {};
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 0; }
  std::lock_guard<std::mutex> lock(mu);
  if (cap[dev]) return cap[dev];
  int best = kMaxCluster;
  const void* const kernels[] = {(const void*)k_orth_part<false>, (const void*)k_orth_part<true>, (const void*)k_orth_group<1>,
                                 (const void*)k_orth_group<kOrthGroup>};
  for (const void* kernel : kernels) {
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes) != cudaSuccess) { cudaGetLastError(); return 0; }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kMaxCluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kMaxCluster); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kSmemBytes; cfg.attrs = at; cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n < 1)
      best = 8;
  }
  cudaGetLastError();
  return cap[dev] = best;
}

// CTAs for order k: at least 32 rows each, a power of two.
int cluster_for(int64_t k) {
  int cs = 1;
  while (cs < kMaxCluster && 32 * cs < k) cs *= 2;
  return cs;
}

// One cluster of `cs` CTAs for each of n jobs.
template <typename KERNEL, typename ARGS>
cudaError_t launch(KERNEL kernel, const ARGS& a, int cs, int n, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(cs * n)); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kSmemBytes; cfg.stream = s;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

inline int64_t pad32(int64_t doubles) { return (doubles + 31) / 32 * 32; }
// The largest coefficient block: the root's is at most (k / 2)^2, a node of the left half (which may be
// the larger one when the last panel is ragged) at most that or one panel squared.
int64_t coef_doubles(int64_t k) { return pad32(std::max<int64_t>(((k + 1) / 2) * ((k + 1) / 2), kW * kW)); }

}  // namespace

static int64_t norm_doubles(int64_t k, bool grouped) { return pad32(2 * (grouped ? kMaxCluster : cluster_for(k)) * k); }
size_t orth_work_doubles(int64_t k, bool grouped) { return (size_t)(coef_doubles(k) + norm_doubles(k, grouped) + pad32(k)); }
void orth_job_work(OrthJob* j, double* work, bool grouped) {
  j->C = work; j->normp = j->C + coef_doubles(j->k); j->rdiag = j->normp + norm_doubles(j->k, grouped);
}

template <int NJ>
static cudaError_t orth_launch(const OrthJob* jobs, int n, int cs, int* status, cudaStream_t s) {
  OrthGroup<NJ> g;
  for (int i = 0; i < n; ++i) g.j[i] = jobs[i];
  g.status = status;
  return launch(k_orth_group<NJ>, g, cs, n, s);
}
cudaError_t orth_group(const OrthJob* jobs, int n, int* status, cudaStream_t s) {
  const int cap = max_cluster();
  if (cap == 0) return cudaErrorInvalidConfiguration;
  int64_t k = 1;
  for (int i = 0; i < n; ++i) k = std::max(k, jobs[i].k);
  const int cs = std::min(cap, cluster_for(k));
  for (int i = 0; i < n; i += kOrthGroup) {
    const int m = std::min(kOrthGroup, n - i);
    const cudaError_t e = m == 1 ? orth_launch<1>(jobs + i, 1, cs, status, s) : orth_launch<kOrthGroup>(jobs + i, m, cs, status, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t orth_part(double* A, int64_t k, int64_t j0, int64_t w, double* C, int first, double ill_ratio, const double* norm0,
                      double* rdiag, int* status, int* flags, const int* skip, cudaStream_t s) {
  const int cap = max_cluster();
  if (cap == 0) return cudaErrorInvalidConfiguration;
  PartArgs a = {};
  a.A = A; a.k = k; a.j0 = (int)j0; a.w = (int)w; a.first = first; a.ill_ratio = ill_ratio; a.norm0 = norm0;
  a.C = C; a.rdiag = rdiag; a.status = status; a.flags = flags; a.skip = skip;
  const int cs = std::min(cap, cluster_for(k));
  return k % 2 == 0 ? launch(k_orth_part<true>, a, cs, 1, s) : launch(k_orth_part<false>, a, cs, 1, s);
}

template <int NJ>
static cudaError_t product_launch(const OrthJob* jobs, int n, int zs, cudaStream_t s) {
  ProductGroup<NJ> g;
  g.n = n;
  g.tile0[0] = 0;
  for (int i = 0; i < n; ++i) {
    const int nt = (int)((jobs[i].k + 63) / 64);
    g.F[i] = jobs[i].F; g.Q[i] = jobs[i].Qprev; g.A[i] = jobs[i].A; g.k[i] = (int)jobs[i].k;
    g.tile0[i + 1] = g.tile0[i] + nt * nt;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)zs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(g.tile0[n] * zs)); cfg.blockDim = dim3(kT); cfg.dynamicSmemBytes = kProductSmem; cfg.stream = s;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_product_group<NJ>, g);
}
cudaError_t product_group(const OrthJob* jobs, int n, cudaStream_t s) {
  for (int i = 0; i < n; i += kOrthGroup) {
    const int m = std::min(kOrthGroup, n - i);
    int64_t tiles = 0, k = 0;
    for (int q = i; q < i + m; ++q) { const int64_t nt = (jobs[q].k + 63) / 64; tiles += nt * nt; k = std::max(k, jobs[q].k); }
    // fewer tiles than two CTAs per SM can hold: share their contractions, down to three stages each (at most 1, 2, 4 and 8 ways, refresh of
    // one basis of order 256 169, 166, 157, 158 us, of 384 269, 259, 254, 256, of 768 808, 797, 796, 797; four of 200 155, 153, 148, 147)
    int zs = 1;
    while (zs < 8 && 2 * zs * tiles <= 296 && 2 * zs * 3 * kKs <= k) zs *= 2;
    const cudaError_t e = m == 1 ? product_launch<1>(jobs + i, 1, zs, s) : product_launch<kOrthGroup>(jobs + i, m, zs, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t product64(int ta, int64_t M, int64_t N, int64_t K, double alpha, const float* A, int64_t lda, const float* B,
                      int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t s) {
  return launch_product(ta, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s);
}
cudaError_t product64(int ta, int64_t M, int64_t N, int64_t K, double alpha, const float* A, int64_t lda, const double* B,
                      int64_t ldb, double beta, double* C, int64_t ldc, cudaStream_t s) {
  return launch_product(ta, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, s);
}

cudaError_t dgemm64(int ta, int tb, int64_t M, int64_t N, int64_t K, double alpha, const double* A, int64_t lda, const double* B,
                    int64_t ldb, double beta, double* C, int64_t ldc, int nsplit, int64_t k_per_split, double* partial, const int* skip,
                    cudaStream_t s) {
  const dim3 grid((unsigned)((N + 63) / 64), (unsigned)((M + 63) / 64), (unsigned)nsplit);
  const bool vec = ((M | N | K | lda | ldb) & 1) == 0 && ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
#define BR_DGEMM64(T, B_) \
  return vec ? launch_dgemm<true, T, B_>(grid, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, k_per_split, partial, skip, s) \
             : launch_dgemm<false, T, B_>(grid, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, k_per_split, partial, skip, s)
  if (ta) { if (tb) BR_DGEMM64(true, true); BR_DGEMM64(true, false); }
  if (tb) BR_DGEMM64(false, true);
  BR_DGEMM64(false, false);
#undef BR_DGEMM64
}

}  // namespace br
