// Grouped fp32 (FFMA) contractions: the accurate path.  Used for BR_GEMM_FP32 and for layers whose
// shapes the tensor-core tiles do not take.  (The fp64 contractions of the basis refresh live in
// dgemm.cu and orth.cu.)
//
//   C = alpha * op(A) op(B) + beta * C, all row-major, op(A) M x K, op(B) K x N
//
// or, DUAL, two products with the same shapes whose tiles meet in one epilogue (the rotated gradient and
// the rotated momentum, see SimtProblem).  One launch covers the same phase of every layer of a handle: the
// matrices of this path are small, and a launch of their own for each product left most SMs idle and cost
// 40 us for what a CTA computes in 10 (four ragged layers of 37 x 53 to 333 x 257: 1.1 ms an update as 40
// launches, of which 1.0 ms in the products).
//
// A CTA computes one tile; the next 16 steps of the contraction are fetched into registers while the
// current ones are multiplied out of shared memory.  The tile follows from the size of the launch's results (launch_sized):
// 32 x 32 on 64 threads while those tiles fit on the GPU at once (the time is then that of one tile's chain, and a small
// tile's step is the shortest), 64 x 64 up to a few waves, 128 x 128 (8 x 8 per thread, half the shared-memory
// reads per multiply-add) above.  With at most four tiles of 32 x 32 per SM a step is bound by the latency of
// its loads, and four groups of 64 threads take a quarter of the contraction each: the dual launch of the four
// ragged layers 54 -> 30 us, the others 30 -> 16 us.  The orientations of the operands are compile-time values (four bodies a
// kernel): factors and first sides of those layers 36.7 -> 26 us, back rotation 11 -> 8.7, weight write 21 -> 16.5.
#include "br_internal.h"

namespace br {
namespace {

constexpr int BK = 16;
constexpr int kMaxProblems = 32;      // by value: 3.2 KB of launch parameters

struct GroupArgs {
  SimtProblem p[kMaxProblems];
  int tile_begin[kMaxProblems + 1];
  int n;
};

// A thread's share of an operand tile of BX rows (columns) by BK steps of the contraction.  T: the tile index is the
// contiguous one, x(i, kk) = X[kk * ld + i]; otherwise x(i, kk) = X[i * ld + kk].  Everything that does not change from stage to
// stage is worked out once (with the orientation a runtime value and the address formed per entry, index arithmetic
// was half of all instructions).
template <bool T, int BX, int NT>
struct Operand {
  static constexpr int L = BX * BK / NT, DI = T ? 0 : NT / BK, DK = T ? NT / BX : 0;
  static_assert(NT % BX == 0 && NT % BK == 0, "a thread's entries differ in one index only");
  const float* at;
  int64_t step, next;
  int i, k;
  unsigned rows;                        // bit u: entry u lies inside the matrix
  __device__ __forceinline__ Operand(const float* X, int64_t ld, int t, int x0, int extent, int kbeg) {
    i = T ? t % BX : t / BK; k = T ? t / BX : t % BK;
    at = X + (T ? (int64_t)(kbeg + k) * ld + x0 + i : (int64_t)(x0 + i) * ld + kbeg + k);
    step = T ? DK * ld : DI * ld; next = T ? BK * ld : BK;
    rows = 0;
#pragma unroll
    for (int u = 0; u < L; ++u) rows |= (unsigned)(x0 + i + u * DI < extent) << u;
  }
  __device__ __forceinline__ void fetch(float (&v)[L], int left) {      // left: steps of the contraction from here on
#pragma unroll
    for (int u = 0; u < L; ++u) v[u] = ((rows >> u) & 1) && k + u * DK < left ? at[u * step] : 0.f;
    at += next;
  }
  template <typename S> __device__ __forceinline__ void put(S& s, const float (&v)[L]) const {
#pragma unroll
    for (int u = 0; u < L; ++u) s[k + u * DK][i + u * DI] = v[u];
  }
};

template <int BM, int BN, bool DUAL, int KS> struct Area {
  static constexpr int FA = BK * (BM + 4), FB = BK * (BN + 4);
  __align__(16) float v[KS][(DUAL ? 2 : 1) * (FA + FB)];
};

// KS groups of NT threads share one tile's contraction (a range of it each) and add up their sums at the end.
template <int BM, int BN, int TM, int TN, bool DUAL, int KS, bool TA, bool TB>
__device__ __forceinline__ void simt_tile(const SimtProblem& p, int tile, Area<BM, BN, DUAL, KS>& area_) {
  constexpr int NT = (BM / TM) * (BN / TN), NP = DUAL ? 2 : 1;
  constexpr int FA = Area<BM, BN, DUAL, KS>::FA, FB = Area<BM, BN, DUAL, KS>::FB;
  static_assert(KS == 1 || (TM == 4 && TN == 4 && KS == TM && NP * TM * NT * 4 <= NP * (FA + FB)), "partial sums fit the operand area");
  auto& area = area_.v;
  const int group = KS == 1 ? 0 : (int)threadIdx.x / NT;
  float(*As)[BK][BM + 4] = reinterpret_cast<float(*)[BK][BM + 4]>(area[group]);
  float(*Bs)[BK][BN + 4] = reinterpret_cast<float(*)[BK][BN + 4]>(area[group] + NP * FA);
  auto sync = [&] {      // the groups run at their own pace
    if (KS == 1) __syncthreads(); else asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(NT) : "memory");
  };
  const int tiles_n = (p.N + BN - 1) / BN;
  const int m0 = tile / tiles_n * BM, n0 = tile % tiles_n * BN;
  const int M = p.M, N = p.N;
  const int kc = KS == 1 ? p.K : (p.K + KS * BK - 1) / (KS * BK) * BK, kbeg = min(p.K, group * kc), K = min(p.K, kbeg + kc);
  const int t = threadIdx.x % NT, tx = t % (BN / TN), ty = t / (BN / TN);

  typedef Operand<TA, BM, NT> OpA;
  typedef Operand<!TB, BN, NT> OpB;
  OpA a0(p.A[0], p.lda, t, m0, M, kbeg), a1(p.A[NP - 1], p.lda, t, m0, M, kbeg);
  OpB b0(p.B[0], p.ldb, t, n0, N, kbeg), b1(p.B[NP - 1], p.ldb, t, n0, N, kbeg);
  float ra[NP][OpA::L], rb[NP][OpB::L];
  auto fetch = [&](int left) {
    a0.fetch(ra[0], left); b0.fetch(rb[0], left);
    if (DUAL) { a1.fetch(ra[NP - 1], left); b1.fetch(rb[NP - 1], left); }
  };
  float acc[NP][TM][TN];
#pragma unroll
  for (int z = 0; z < NP; ++z)
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j) acc[z][i][j] = 0.f;
  // thread rows ty * 4 + i % 4 (+ BM / 2 for i >= 4), columns likewise: 16-byte reads, neighbours adjacent
  auto sub = [](int base, int i, int half) { return (i < 4 ? 0 : half) + base * 4 + (i & 3); };
  if (kbeg < K) fetch(K - kbeg);
  for (int k0 = kbeg; k0 < K; k0 += BK) {
    a0.put(As[0], ra[0]); b0.put(Bs[0], rb[0]);
    if (DUAL) { a1.put(As[NP - 1], ra[NP - 1]); b1.put(Bs[NP - 1], rb[NP - 1]); }
    sync();
    if (k0 + BK < K) fetch(K - k0 - BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk)
#pragma unroll
      for (int z = 0; z < NP; ++z) {
        float a[TM], b[TN];
#pragma unroll
        for (int i = 0; i < TM; i += 4) *reinterpret_cast<float4*>(a + i) = *reinterpret_cast<const float4*>(&As[z][kk][sub(ty, i, BM / 2)]);
#pragma unroll
        for (int j = 0; j < TN; j += 4) *reinterpret_cast<float4*>(b + j) = *reinterpret_cast<const float4*>(&Bs[z][kk][sub(tx, j, BN / 2)]);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) acc[z][i][j] = fmaf(a[i], b[j], acc[z][i][j]);
      }
    sync();
  }
  if (KS > 1) {
    // [product][row of the thread's tile][thread], four columns each; group g then finishes row g of every tile
    float4* mine = reinterpret_cast<float4*>(area[group]);
#pragma unroll
    for (int z = 0; z < NP; ++z)
#pragma unroll
      for (int i = 0; i < TM; ++i) mine[(z * TM + i) * NT + t] = make_float4(acc[z][i][0], acc[z][i][1], acc[z][i][2], acc[z][i][3]);
    __syncthreads();
#pragma unroll
    for (int z = 0; z < NP; ++z) {
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int g = 0; g < KS; ++g) {
        const float4 o = reinterpret_cast<const float4*>(area[g])[(z * TM + group) * NT + t];
        s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
      }
      acc[z][0][0] = s.x; acc[z][0][1] = s.y; acc[z][0][2] = s.z; acc[z][0][3] = s.w;
    }
  }
  constexpr int ROWS = KS > 1 ? 1 : TM;
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const int gm = m0 + sub(ty, KS > 1 ? group : i, BM / 2);
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gn = n0 + sub(tx, j, BN / 2);
      if (gn >= N) continue;
      const int64_t at = (int64_t)gm * p.ldc + gn;
      if (DUAL) {
        const float g = acc[0][i][j], v2 = p.beta * p.V2[at] + p.alpha * g * g;
        p.V2[at] = v2;
        p.C[at] = acc[NP - 1][i][j] / sqrtf(v2 + p.eps);
      } else {
        float v = p.alpha * acc[0][i][j];
        if (p.beta != 0.f) v = fmaf(p.beta, p.C[at], v);
        p.C[at] = v;
      }
    }
  }
}

template <int BM, int BN, int TM, int TN, bool DUAL, int KS>
__global__ void __launch_bounds__(KS * (BM / TM) * (BN / TN))
k_simt_group(const __grid_constant__ GroupArgs ga) {
  __shared__ Area<BM, BN, DUAL, KS> area;
  int pi = 0;
  while (pi + 1 < ga.n && (int)blockIdx.x >= ga.tile_begin[pi + 1]) ++pi;
  const SimtProblem& p = ga.p[pi];
  const int tile = (int)blockIdx.x - ga.tile_begin[pi];
  if (p.ta) {
    if (p.tb) simt_tile<BM, BN, TM, TN, DUAL, KS, true, true>(p, tile, area); else simt_tile<BM, BN, TM, TN, DUAL, KS, true, false>(p, tile, area);
  } else {
    if (p.tb) simt_tile<BM, BN, TM, TN, DUAL, KS, false, true>(p, tile, area); else simt_tile<BM, BN, TM, TN, DUAL, KS, false, false>(p, tile, area);
  }
}

template <int BM, int BN, int TM, int TN, bool DUAL, int KS = 1>
cudaError_t launch(GroupArgs& ga, cudaStream_t s) {
  int64_t tiles = 0;
  for (int i = 0; i < ga.n; ++i) {
    ga.tile_begin[i] = (int)tiles;
    tiles += (int64_t)((ga.p[i].M + BM - 1) / BM) * ((ga.p[i].N + BN - 1) / BN);
  }
  ga.tile_begin[ga.n] = (int)tiles;
  if (tiles > 0x7fffffff) return cudaErrorInvalidConfiguration;
  k_simt_group<BM, BN, TM, TN, DUAL, KS><<<(unsigned)tiles, KS * (BM / TM) * (BN / TN), 0, s>>>(ga);
  return cudaGetLastError();
}

// The lines, in result tiles of 32 x 32, measured on updates of one k x k matrix rotated on one side (us, the form below
// the line and the one above): 592: k = 640 (400 tiles) 110 and 134, 900 (841) 281 and 249.  1776: 1400 (1936) 789 and
// 711; 64 x 64 is the faster one already at 1000 (1024) with 343 and 282 and at 1300 (1681) with 639 and 524.  9472: level
// within 2 % from 2800 to 4200.  How long the contraction is does not enter: a result of few tiles with a contraction of
// tens of thousands is one chain per tile.
template <bool DUAL>
cudaError_t launch_sized(GroupArgs& ga, cudaStream_t s) {
  double area = 0.0;                                       // in tiles of 32 x 32
  for (int i = 0; i < ga.n; ++i) area += (double)((ga.p[i].M + 31) / 32) * ((ga.p[i].N + 31) / 32);
  if (area <= 148 * 4) return launch<32, 32, 4, 4, DUAL, 4>(ga, s);
  if (area <= 148 * 12) return launch<32, 32, 4, 4, DUAL>(ga, s);
  if (DUAL || area <= 148 * 64) return launch<64, 64, 4, 4, DUAL>(ga, s);
  return launch<128, 128, 8, 8, false>(ga, s);
}

}  // namespace

cudaError_t simt_group(const SimtProblem* problems, int n, bool dual, cudaStream_t s) {
  GroupArgs ga;
  for (int at = 0; at < n; at += kMaxProblems) {
    ga.n = 0;
    for (int i = at; i < n && i < at + kMaxProblems; ++i)
      if (problems[i].M > 0 && problems[i].N > 0) ga.p[ga.n++] = problems[i];
    if (ga.n == 0) continue;
    const cudaError_t e = dual ? launch_sized<true>(ga, s) : launch_sized<false>(ga, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

SimtProblem simt_problem(int ta, int tb, int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda, const float* B,
                         int64_t ldb, float beta, float* C, int64_t ldc) {
  SimtProblem p = {};
  p.A[0] = p.A[1] = A; p.B[0] = p.B[1] = B; p.C = C;
  p.M = (int)M; p.N = (int)N; p.K = (int)K; p.lda = (int)lda; p.ldb = (int)ldb; p.ldc = (int)ldc;
  p.ta = ta; p.tb = tb; p.alpha = alpha; p.beta = beta;
  return p;
}

cudaError_t sgemm(int ta, int tb, int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t lda, const float* B,
                  int64_t ldb, float beta, float* C, int64_t ldc, cudaStream_t s) {
  const SimtProblem p = simt_problem(ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
  return simt_group(&p, 1, false, s);
}

}  // namespace br
