// One rotated-Adam update of small weight matrices in a single launch, a cluster of up to four CTAs per matrix:
// Alg. 1 (momentum, rotation, second moment, weight update) and the factor EMAs of Alg. 2, with every operand
// staged in shared memory and fp32 FFMA dot products.  A matrix of this size is bound by launch latency, not by
// arithmetic: the grouped launches of the general fp32 path are five per update, this kernel is one.  The
// refresh of the bases (Alg. 1 (periodic refresh)) is not part of it: a call on which a refresh is due goes
// through the general path.
//
// Every CTA stages all operands and computes its share of the rows of every result; only X crosses CTAs (each
// writes its rows of X into all of them before the back rotation U X).  A thread computes 2 x 4 tiles from
// operands whose contraction index is the slow one (an 8- and a 16-byte read per step for 8 multiply-adds; the
// rotation of G and of M shares the basis' read).  That takes G, U and V in both orientations; T, X and Y are
// written in the one the next product reads.  Bound by the shared-memory reads of one SM, hence the cluster:
// a 64 x 32 matrix took 33 us with a dot product per thread, 18 us with 4 x 4 tiles on one CTA, 13 us now.  Matrices
// of a few hundred entries keep the dot product per thread (k_tiny_step).
#include <cooperative_groups.h>

#include <algorithm>

#include "br_internal.h"

namespace cg = cooperative_groups;

namespace br {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxSmem = 220 * 1024;

// NJ: 1 or kSmallJobs (3 KB of parameters make a launch longer on the host)
template <int NJ> struct SmallGroup { SmallJob j[NJ]; float lr, beta1, beta2, eps, decay, beta_factor; };

__host__ __device__ inline int up4(int x) { return (x + 3) & ~3; }
// leading dimension of a staged matrix with `cols` columns (16-byte rows; the rows that a thread writes transposed
// fall into two groups of banks instead of one)
__host__ __device__ inline int ldp(int cols) { return up4(cols) + 4; }

struct Acc { float v[2][4]; };
__device__ __forceinline__ void fma8(Acc& c, float2 x, float4 y) {
  c.v[0][0] = fmaf(x.x, y.x, c.v[0][0]); c.v[0][1] = fmaf(x.x, y.y, c.v[0][1]);
  c.v[0][2] = fmaf(x.x, y.z, c.v[0][2]); c.v[0][3] = fmaf(x.x, y.w, c.v[0][3]);
  c.v[1][0] = fmaf(x.y, y.x, c.v[1][0]); c.v[1][1] = fmaf(x.y, y.y, c.v[1][1]);
  c.v[1][2] = fmaf(x.y, y.z, c.v[1][2]); c.v[1][3] = fmaf(x.y, y.w, c.v[1][3]);
}
__device__ __forceinline__ float2 f2(const float* p) { return *reinterpret_cast<const float2*>(p); }
__device__ __forceinline__ float4 f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
// acc[a][b] = sum_k A[k * lda + a] B[k * ldb + b]
__device__ __forceinline__ void tile(Acc& c, const float* A, int lda, const float* B, int ldb, int K) {
  c = Acc{};
#pragma unroll 8
  for (int k = 0; k < K; ++k) fma8(c, f2(A + k * lda), f4(B + k * ldb));
}
// two products with a common first (A) or second (B) operand
__device__ __forceinline__ void tile_a(Acc& c, Acc& d, const float* A, int lda, const float* B0, const float* B1, int ldb, int K) {
  c = Acc{}; d = Acc{};
#pragma unroll 8
  for (int k = 0; k < K; ++k) { const float2 x = f2(A + k * lda); fma8(c, x, f4(B0 + k * ldb)); fma8(d, x, f4(B1 + k * ldb)); }
}
__device__ __forceinline__ void tile_b(Acc& c, Acc& d, const float* A0, const float* A1, int lda, const float* B, int ldb, int K) {
  c = Acc{}; d = Acc{};
#pragma unroll 8
  for (int k = 0; k < K; ++k) { const float4 y = f4(B + k * ldb); fma8(c, f2(A0 + k * lda), y); fma8(d, f2(A1 + k * lda), y); }
}
// P[(i + a) * cols + j + b] = f(old, a, b) on the part of the tile that exists
template <typename FN>
__device__ __forceinline__ void rmw(float* P, int rows, int cols, int i, int j, FN f) {
  if (i + 2 <= rows && (cols & 3) == 0) {
    const float4 o0 = f4(P + i * cols + j), o1 = f4(P + (i + 1) * cols + j);
    *reinterpret_cast<float4*>(P + i * cols + j) = make_float4(f(o0.x, 0, 0), f(o0.y, 0, 1), f(o0.z, 0, 2), f(o0.w, 0, 3));
    *reinterpret_cast<float4*>(P + (i + 1) * cols + j) = make_float4(f(o1.x, 1, 0), f(o1.y, 1, 1), f(o1.z, 1, 2), f(o1.w, 1, 3));
    return;
  }
  float o[2][4];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) o[a][b] = (i + a < rows && j + b < cols) ? P[(i + a) * cols + j + b] : 0.f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (i + a < rows && j + b < cols) P[(i + a) * cols + j + b] = f(o[a][b], a, b);
}
// tile -> S row-major [i][j], or transposed [j][i]
__device__ __forceinline__ void put(float* S, int ld, int i, int j, const Acc& c) {
#pragma unroll
  for (int a = 0; a < 2; ++a) *reinterpret_cast<float4*>(S + (i + a) * ld + j) = make_float4(c.v[a][0], c.v[a][1], c.v[a][2], c.v[a][3]);
}
__device__ __forceinline__ void put_t(float* S, int ld, int i, int j, const Acc& c) {
#pragma unroll
  for (int b = 0; b < 4; ++b) *reinterpret_cast<float2*>(S + (j + b) * ld + i) = make_float2(c.v[0][b], c.v[1][b]);
}

// Walks the entries t, t + kThreads, ... of a matrix with `cols` columns without a division per entry.
struct Walk {
  int r, c, dr, dc, cols;
  __device__ __forceinline__ Walk(int cols_) : cols(cols_) {
    r = (int)threadIdx.x / cols; c = (int)threadIdx.x % cols; dr = kThreads / cols; dc = kThreads % cols;
  }
  __device__ __forceinline__ void next() { r += dr; c += dc; if (c >= cols) { c -= cols; ++r; } }
};

// S[r][c] and St[c][r] (both ld) <- the k x k matrix P, zero-padded to a multiple of four; eight loads in flight
__device__ __forceinline__ void stage_both(const float* __restrict__ P, int k, float* S, float* St, int ld) {
  const int kp = up4(k);
  Walk ld_at(kp), st_at(kp);
  while (ld_at.r < kp) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      v[u] = (ld_at.r < k && ld_at.c < k) ? __ldg(P + ld_at.r * k + ld_at.c) : 0.f;
      ld_at.next();
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (st_at.r < kp) { S[st_at.r * ld + st_at.c] = v[u]; St[st_at.c * ld + st_at.r] = v[u]; }
      st_at.next();
    }
  }
}

// This call's gradient into the ring slot that every reader of it in the launch has passed: item `at` of the copy's
// 16-byte pieces (2-byte units where its size is no multiple of them), then every `step`-th.  (As a copy behind the kernel it
// took 2.3 us of the 16.6 of a call on one 64 x 32 matrix.)
struct RingCopy {
  int units, vec;
  uint4 first;
  __device__ __forceinline__ void load(const SmallJob& a, int at) {
    const int bytes = a.ring ? a.m * a.n * (a.g_is_bf16 ? 2 : 4) : 0;
    vec = bytes % 16 == 0 ? 1 : 0;
    units = bytes / (vec ? 16 : 2);
    if (at < units) { if (vec) first = reinterpret_cast<const uint4*>(a.grad)[at]; else first.x = reinterpret_cast<const uint16_t*>(a.grad)[at]; }
  }
  __device__ __forceinline__ void store(const SmallJob& a, int at, int step) const {
    if (vec) {
      uint4* r = reinterpret_cast<uint4*>(a.ring);
      if (at < units) r[at] = first;
      for (int i = at + step; i < units; i += step) r[i] = reinterpret_cast<const uint4*>(a.grad)[i];
    } else {
      uint16_t* r = reinterpret_cast<uint16_t*>(a.ring);
      if (at < units) r[at] = (uint16_t)first.x;
      for (int i = at + step; i < units; i += step) r[i] = reinterpret_cast<const uint16_t*>(a.grad)[i];
    }
  }
};

template <int NJ>
__global__ void __launch_bounds__(kThreads) k_small_step(const __grid_constant__ SmallGroup<NJ> grp) {
  extern __shared__ __align__(16) float sm[];
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const SmallJob& a = grp.j[blockIdx.x / cs];
  const int m = a.m, n = a.n, t = threadIdx.x;
  const int mp = up4(m), np = up4(n), lm = ldp(m), ln = ldp(n);
  const bool L = a.left != 0, R = a.right != 0;
  // staged matrices; padding rows and columns are zero
  float* G = sm;                          // [m][n]
  float* Gt = G + mp * ln;                // [n][m]
  float* Mx = Gt + np * lm;               // [m][n], or [n][m] when only the right side is rotated
  float* X = Mx + (L ? mp * ln : np * lm);    // [m][n]; [n][m] when only the right side is rotated
  float* T1 = X + (L ? mp * ln : np * lm);    // first-side products, transposed [n][m]; later Y^T (both sides rotated)
  float* T2 = T1 + (L && R ? np * lm : 0);
  float* U = T2 + (L && R ? np * lm : 0); // [m][m] and transposed
  float* Ut = U + (L ? mp * lm : 0);
  float* V = Ut + (L ? mp * lm : 0);      // [n][n] and transposed
  float* Vt = V + (R ? np * ln : 0);
  // this CTA's rows of results with m and with n rows
  const int mr = up4((m + cs - 1) / cs), m0 = min(mp, rank * mr), m1 = min(mp, m0 + mr);
  const int nr = up4((n + cs - 1) / cs), n0 = min(np, rank * nr), n1 = min(np, n0 + nr);
  const float gs = a.gscale ? *a.gscale : 1.0f;
  RingCopy copy;
  copy.load(a, rank * kThreads + t);
  if (L) stage_both(a.U, m, U, Ut, lm);
  if (R) stage_both(a.V, n, V, Vt, ln);
  // Alg. 1 (momentum update): M <- beta1 M + (1 - beta1) G
  Walk ld_at(np), st_at(np);
  while (ld_at.r < mp) {
    float g[4], mo[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const bool ok = ld_at.r < m && ld_at.c < n;
      const int i = ok ? ld_at.r * n + ld_at.c : 0;
      g[u] = !ok ? 0.f : a.g_is_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a.G)[i]) : reinterpret_cast<const float*>(a.G)[i];
      mo[u] = ok ? a.M[i] : 0.f;
      ld_at.next();
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = st_at.r, c = st_at.c;
      if (r < mp) {
        g[u] *= gs;
        mo[u] = grp.beta1 * mo[u] + (1.0f - grp.beta1) * g[u];
        G[r * ln + c] = g[u]; Gt[c * lm + r] = g[u];
        if (L) Mx[r * ln + c] = mo[u]; else Mx[c * lm + r] = mo[u];
      }
      st_at.next();
    }
  }
  // every CTA has read all of M and G (and none has left before another writes to its shared memory)
  if (cs > 1) cl.sync(); else __syncthreads();
  copy.store(a, rank * kThreads + t, cs * kThreads);
  for (int e = t; e < (min(m, m1) - m0) * n; e += kThreads) {
    const int r = m0 + e / n, c = e % n;
    a.M[r * n + c] = L ? Mx[r * ln + c] : Mx[c * lm + r];
  }
  // V~ <- beta2 V~ + (1 - beta2) G~^2 ; X = M~ / sqrt(V~ + eps)   (Alg. 1 (second-moment update and scaling))
  auto scale = [&](int i, int j, const Acc& g, Acc& x) {
    Acc v2 = {};
    rmw(a.V2, m, n, i, j, [&](float o, int p, int q) { return v2.v[p][q] = grp.beta2 * o + (1.0f - grp.beta2) * g.v[p][q] * g.v[p][q]; });
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) x.v[p][q] = (i + p < m && j + q < n) ? x.v[p][q] / sqrtf(v2.v[p][q] + grp.eps) : 0.f;
    // the back rotation needs all rows of X in every CTA
    if (!L) put_t(X, lm, i, j, x);
    else if (cs == 1) put(X, ln, i, j, x);
    else
      for (int z = 0; z < cs; ++z) put(cl.map_shared_rank(X, z), ln, i, j, x);
  };
  // independent work of the first phase, dealt to the threads as one list: the rotation (the longest) first
  const int n4 = np / 4, mh = max(0, m1 - m0) / 2, nT = mh * n4;
  const int nL = a.accumulate && a.L ? mh * (mp / 4) : 0, nR = a.accumulate && a.R ? max(0, n1 - n0) / 2 * n4 : 0;
  Acc c, d;
  const float b = grp.beta_factor, ob = 1.0f - grp.beta_factor;
  for (int e = t; e < nT + nL + nR; e += kThreads) {
    if (e < nT) {
      const int i = m0 + e / n4 * 2, j = e % n4 * 4;
      if (L) tile_a(c, d, U + i, lm, G + j, Mx + j, ln, m);         // U^T G, U^T M
      else tile_b(c, d, Gt + i, Mx + i, lm, V + j, ln, n);          // G V, M V
      if (L && R) { put_t(T1, lm, i, j, c); put_t(T2, lm, i, j, d); } else scale(i, j, c, d);
    } else if (e < nT + nL) {             // L <- b L + (1 - b) G G^T
      const int m4 = mp / 4, i = m0 + (e - nT) / m4 * 2, j = (e - nT) % m4 * 4;
      tile(c, Gt + i, lm, Gt + j, lm, n);
      rmw(a.L, m, m, i, j, [&](float o, int p, int q) { return b * o + ob * c.v[p][q]; });
    } else {                              // R <- b R + (1 - b) G^T G
      const int i = n0 + (e - nT - nL) / n4 * 2, j = (e - nT - nL) % n4 * 4;
      tile(c, G + i, ln, G + j, ln, m);
      rmw(a.R, n, n, i, j, [&](float o, int p, int q) { return b * o + ob * c.v[p][q]; });
    }
  }
  if (L && R) {
    __syncthreads();
    for (int e = t; e < nT; e += kThreads) {           // G~ = T1 V, M~ = T2 V
      const int i = m0 + e / n4 * 2, j = e % n4 * 4;
      tile_b(c, d, T1 + i, T2 + i, lm, V + j, ln, n);
      scale(i, j, c, d);
    }
  }
  if (L && cs > 1) cl.sync(); else __syncthreads();
  // weight update: W <- decay W - eta U X V^T
  const float* Yt = X;
  if (L) {
    for (int e = t; e < nT; e += kThreads) {
      const int i = m0 + e / n4 * 2, j = e % n4 * 4;
      tile(c, Ut + i, lm, X + j, ln, m);
      if (R) put_t(T1, lm, i, j, c);
      else rmw(a.W, m, n, i, j, [&](float o, int p, int q) { return grp.decay * o - grp.lr * c.v[p][q]; });
    }
    if (!R) return;
    Yt = T1;
    __syncthreads();
  }
  for (int e = t; e < nT; e += kThreads) {
    const int i = m0 + e / n4 * 2, j = e % n4 * 4;
    tile(c, Yt + i, lm, Vt + j, ln, n);
    rmw(a.W, m, n, i, j, [&](float o, int p, int q) { return grp.decay * o - grp.lr * c.v[p][q]; });
  }
}

// The same update for launches of tiny matrices only (tiny_eligible), a CTA each and a dot product per thread.  Such a
// matrix is bound by the latency of its loads and barriers: the form above stages more copies, zero-padded, behind
// index arithmetic and a second set of barriers.  Kernel time on one matrix, here and above, us: 8 x 8 4.8 and 7.4,
// 16 x 16 5.7 and 7.2, 32 x 4 6.3 and 9.0, 40 x 8 rotated on the right only 4.4 and 6.0.
constexpr int kTinyThreads = 512, kTinySmem = 80 * 1024;
template <int NJ>
__global__ void __launch_bounds__(kTinyThreads) k_tiny_step(const __grid_constant__ SmallGroup<NJ> grp) {
  extern __shared__ __align__(16) float sm[];
  const SmallJob& a = grp.j[blockIdx.x];
  const int m = a.m, n = a.n, mn = m * n, t = threadIdx.x;
  const int ln = n | 1, lm = m | 1;           // odd: a walk along a column touches different banks
  float* sG = sm;                             // G, later X
  float* sM = sG + m * ln;                    // M, later Y
  float* sT1 = sM + m * ln;                   // first-side products of G and of M
  float* sT2 = sT1 + m * ln;
  float* sU = sT2 + m * ln;                   // m x m (left side rotated)
  float* sV = sU + (a.left ? m * lm : 0);     // n x n (right side rotated)
  const float gs = a.gscale ? *a.gscale : 1.0f;
  RingCopy copy;
  copy.load(a, t);
  for (int e = t; e < mn; e += kTinyThreads) {
    const float g = gs * (a.g_is_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(a.G)[e]) : reinterpret_cast<const float*>(a.G)[e]);
    const float mo = grp.beta1 * a.M[e] + (1.0f - grp.beta1) * g;
    const int at = e / n * ln + e % n;
    sG[at] = g; sM[at] = mo; a.M[e] = mo;
  }
  if (a.left) for (int e = t; e < m * m; e += kTinyThreads) sU[e / m * lm + e % m] = a.U[e];
  if (a.right) for (int e = t; e < n * n; e += kTinyThreads) sV[e / n * ln + e % n] = a.V[e];
  __syncthreads();
  copy.store(a, t, kTinyThreads);
  if (a.accumulate) {                         // L <- b L + (1 - b) G G^T ; R <- b R + (1 - b) G^T G
    const float b = grp.beta_factor, ob = 1.0f - grp.beta_factor;
    if (a.L)
      for (int e = t; e < m * m; e += kTinyThreads) {
        const int i = e / m, j = e % m;
        float s = 0.f;
        for (int k = 0; k < n; ++k) s = fmaf(sG[i * ln + k], sG[j * ln + k], s);
        a.L[e] = b * a.L[e] + ob * s;
      }
    if (a.R)
      for (int e = t; e < n * n; e += kTinyThreads) {
        const int i = e / n, j = e % n;
        float s = 0.f;
        for (int k = 0; k < m; ++k) s = fmaf(sG[k * ln + i], sG[k * ln + j], s);
        a.R[e] = b * a.R[e] + ob * s;
      }
  }
  for (int e = t; e < mn; e += kTinyThreads) {           // T1 = U^T G, T2 = U^T M
    const int i = e / n, j = e % n;
    float s1 = sG[i * ln + j], s2 = sM[i * ln + j];
    if (a.left) {
      s1 = 0.f; s2 = 0.f;
      for (int k = 0; k < m; ++k) { const float u = sU[k * lm + i]; s1 = fmaf(u, sG[k * ln + j], s1); s2 = fmaf(u, sM[k * ln + j], s2); }
    }
    sT1[i * ln + j] = s1; sT2[i * ln + j] = s2;
  }
  __syncthreads();
  for (int e = t; e < mn; e += kTinyThreads) {           // G~ = T1 V, M~ = T2 V, second moment, X
    const int i = e / n, j = e % n;
    float gt = sT1[i * ln + j], mt = sT2[i * ln + j];
    if (a.right) {
      gt = 0.f; mt = 0.f;
      for (int k = 0; k < n; ++k) { const float v = sV[k * ln + j]; gt = fmaf(sT1[i * ln + k], v, gt); mt = fmaf(sT2[i * ln + k], v, mt); }
    }
    const float v2 = grp.beta2 * a.V2[e] + (1.0f - grp.beta2) * gt * gt;
    a.V2[e] = v2;
    sG[i * ln + j] = mt / sqrtf(v2 + grp.eps);
  }
  __syncthreads();
  for (int e = t; e < mn; e += kTinyThreads) {           // Y = U X
    const int i = e / n, j = e % n;
    float y = sG[i * ln + j];
    if (a.left) {
      y = 0.f;
      for (int k = 0; k < m; ++k) y = fmaf(sU[i * lm + k], sG[k * ln + j], y);
    }
    sM[i * ln + j] = y;
  }
  __syncthreads();
  for (int e = t; e < mn; e += kTinyThreads) {           // W <- decay W - eta Y V^T
    const int i = e / n, j = e % n;
    float d = sM[i * ln + j];
    if (a.right) {
      d = 0.f;
      for (int k = 0; k < n; ++k) d = fmaf(sM[i * ln + k], sV[j * ln + k], d);
    }
    a.W[e] = grp.decay * a.W[e] - grp.lr * d;
  }
}

size_t tiny_bytes(int64_t m, int64_t n, bool left, bool right) {
  return sizeof(float) * (size_t)(4 * m * (n | 1) + (left ? m * (m | 1) : 0) + (right ? n * (n | 1) : 0));
}
// In this range the form above takes about as long for every size, and this one as many steps as its phases have
// passes over their entries times terms of a dot product: 264 steps are 9 to 11 us either way while a pass covers the
// matrix, and beyond that the lines are where a sweep of 259 shapes, each with one and with two rotated sides, with
// and without factors, has the two level (the worst of the 1036 is 14 % above what the one form alone took before the
// other existed, 24 are more than 3 %).
bool tiny_eligible(const SmallJob& j) {
  const int m = j.m, n = j.n;
  auto passes = [](int entries) { return (entries + kTinyThreads - 1) / kTinyThreads; };
  int steps = 2 * passes(m * n) * ((j.left ? m : 0) + (j.right ? n : 0));
  if (j.accumulate) steps += (j.L ? passes(m * m) * n : 0) + (j.R ? passes(n * n) * m : 0);
  return m * n < 1024 && steps <= (m * n <= kTinyThreads ? 264 : j.left && j.right ? 240 : 136) &&
         tiny_bytes(m, n, j.left != 0, j.right != 0) <= (size_t)kTinySmem;
}

size_t small_bytes(int64_t m64, int64_t n64, bool left, bool right) {
  const int m = (int)m64, n = (int)n64, mp = up4(m), np = up4(n), lm = ldp(m), ln = ldp(n);
  size_t f = (size_t)mp * ln + (size_t)np * lm + 2 * (left ? (size_t)mp * ln : (size_t)np * lm);
  f += (left && right) ? 2 * (size_t)np * lm : 0;
  f += (left ? 2 * (size_t)mp * lm : 0) + (right ? 2 * (size_t)np * ln : 0);
  return sizeof(float) * f;
}

}  // namespace

// What does not fit in shared memory goes through the grouped launches, which are as fast from about 72 x 72 on (an
// update of 80 x 80 on both sides 27 us either way, 128 x 128 31 us; 64 x 32 14 us here, 21 there).
bool small_step_eligible(int64_t m, int64_t n, bool left, bool right) {
  return (left || right) && m <= 128 && n <= 128 && small_bytes(m, n, left, right) <= kMaxSmem;
}

namespace {
template <int NJ>
SmallGroup<NJ> group(const SmallJob* jobs, int n, float lr, float beta1, float beta2, float eps, float weight_decay, float beta_factor) {
  SmallGroup<NJ> g;
  g.lr = lr; g.beta1 = beta1; g.beta2 = beta2; g.eps = eps; g.decay = 1.0f - lr * weight_decay; g.beta_factor = beta_factor;
  for (int i = 0; i < n; ++i) g.j[i] = jobs[i];
  return g;
}
template <int NJ>
cudaError_t launch_tiny(const SmallJob* jobs, int n, float lr, float beta1, float beta2, float eps, float weight_decay, float beta_factor,
                        cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t e = once.run([] { return cudaFuncSetAttribute(k_tiny_step<NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTinySmem); });
  if (e != cudaSuccess) return e;
  size_t bytes = 0;
  for (int i = 0; i < n; ++i) bytes = std::max(bytes, tiny_bytes(jobs[i].m, jobs[i].n, jobs[i].left != 0, jobs[i].right != 0));
  k_tiny_step<NJ><<<n, kTinyThreads, bytes, s>>>(group<NJ>(jobs, n, lr, beta1, beta2, eps, weight_decay, beta_factor));
  return cudaGetLastError();
}
template <int NJ>
cudaError_t launch(const SmallJob* jobs, int n, float lr, float beta1, float beta2, float eps, float weight_decay, float beta_factor,
                   cudaStream_t s) {
  static OncePerDevice once;
  const cudaError_t e = once.run([] { return cudaFuncSetAttribute(k_small_step<NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem); });
  if (e != cudaSuccess) return e;
  size_t bytes = 0;
  int rows = 0;
  for (int i = 0; i < n; ++i) {
    const size_t need = small_bytes(jobs[i].m, jobs[i].n, jobs[i].left != 0, jobs[i].right != 0);
    if (need > bytes) bytes = need;
    if (jobs[i].m > rows) rows = jobs[i].m;
    if (jobs[i].n > rows) rows = jobs[i].n;
  }
  const int cs = rows >= 32 ? 4 : 1;       // (below 32 rows the cluster's barriers cost more than its SMs give)
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(n * cs)); cfg.blockDim = dim3(kThreads); cfg.dynamicSmemBytes = bytes; cfg.stream = s;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_small_step<NJ>, group<NJ>(jobs, n, lr, beta1, beta2, eps, weight_decay, beta_factor));
}
}  // namespace

bool tiny_step_eligible(const SmallJob& j) { return tiny_eligible(j); }

cudaError_t small_step(const SmallJob* jobs, int n, bool tiny, float lr, float beta1, float beta2, float eps, float weight_decay,
                       float beta_factor, cudaStream_t s) {
  if (n < 1 || n > kSmallJobs) return cudaErrorInvalidValue;
  if (tiny)
    return n == 1 ? launch_tiny<1>(jobs, 1, lr, beta1, beta2, eps, weight_decay, beta_factor, s)
                  : launch_tiny<kSmallJobs>(jobs, n, lr, beta1, beta2, eps, weight_decay, beta_factor, s);
  return n == 1 ? launch<1>(jobs, 1, lr, beta1, beta2, eps, weight_decay, beta_factor, s)
                : launch<kSmallJobs>(jobs, n, lr, beta1, beta2, eps, weight_decay, beta_factor, s);
}

}  // namespace br
