// Fused element-wise kernels of the rotated Adam step.  All are HBM-bound: one pass over the
// data, 128-bit accesses on the aligned body, grid-stride loops on a grid sized as a multiple of
// the SM count.
#include <algorithm>

#include "br_internal.h"

namespace br {

namespace {

constexpr int kThreads = 256;

template <int NSEG>
struct ClipSegs {                 // passed by value: one launch covers up to NSEG gradients
  const void* ptr[NSEG];
  long long begin[NSEG + 1];      // element offsets in the concatenation
  int bf16[NSEG];
};

inline int grid_for(int64_t n_vec) {
  // 148 SMs on a B200, 8 resident CTAs of 256 threads each.
  int64_t want = (n_vec + kThreads - 1) / kThreads;
  int64_t cap = 148 * 8;
  if (want < 1) want = 1;
  return (int)(want < cap ? want : cap);
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }

__device__ __forceinline__ float4 ld4_bf16(const __nv_bfloat16* p) {
  uint2 raw = *reinterpret_cast<const uint2*>(p);
  float4 r;
  r.x = __uint_as_float(raw.x << 16);
  r.y = __uint_as_float(raw.x & 0xFFFF0000u);
  r.z = __uint_as_float(raw.y << 16);
  r.w = __uint_as_float(raw.y & 0xFFFF0000u);
  return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ void st4_bf16(__nv_bfloat16* p, float4 v) {
  uint2 raw;
  raw.x = pack_bf16(v.x, v.y);
  raw.y = pack_bf16(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = raw;
}

__device__ __forceinline__ float bf16_round(float x) {
  return __bfloat162float(__float2bfloat16_rn(x));
}

template <bool G_BF16>
__device__ __forceinline__ float4 load_grad4(const void* G, int64_t i) {
  if (G_BF16) return ld4_bf16(reinterpret_cast<const __nv_bfloat16*>(G) + i);
  return ld4(reinterpret_cast<const float*>(G) + i);
}
template <bool G_BF16>
__device__ __forceinline__ float load_grad1(const void* G, int64_t i) {
  if (G_BF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(G)[i]);
  return reinterpret_cast<const float*>(G)[i];
}

__global__ void k_set_identity(float* Q, int64_t k) {
  int64_t n = k * k;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    Q[i] = (i / k == i % k) ? 1.0f : 0.0f;
  }
}

constexpr int kMaxEmaJobs = 32;
struct EmaArgs {                  // passed by value
  EmaJob j[kMaxEmaJobs];
  int block_begin[kMaxEmaJobs + 1];
  int n;
};

template <bool G_BF16>
__device__ __forceinline__ void ema_one(const EmaJob& j, int block, int blocks, float beta1) {
  const float gs = j.gscale ? *j.gscale : 1.0f;     // clipping factor of the call this gradient came with
  const float omb = 1.0f - beta1;
  const int64_t nvec = j.numel >> 2, stride = (int64_t)blocks * kThreads;
  for (int64_t v = block * (int64_t)kThreads + threadIdx.x; v < nvec; v += stride) {
    const int64_t i = v << 2;
    float4 g = load_grad4<G_BF16>(j.G, i);
    g.x *= gs; g.y *= gs; g.z *= gs; g.w *= gs;
    float4 m = ld4(j.M + i);
    m.x = beta1 * m.x + omb * g.x;
    m.y = beta1 * m.y + omb * g.y;
    m.z = beta1 * m.z + omb * g.z;
    m.w = beta1 * m.w + omb * g.w;
    st4(j.M + i, m);
    if (j.Gf32) st4(j.Gf32 + i, g);
  }
  // ragged tail (numel not a multiple of 4)
  for (int64_t i = (nvec << 2) + block * (int64_t)kThreads + threadIdx.x; i < j.numel; i += stride) {
    const float g = gs * load_grad1<G_BF16>(j.G, i);
    j.M[i] = beta1 * j.M[i] + omb * g;
    if (j.Gf32) j.Gf32[i] = g;
  }
}

// The momentum EMA of every layer of the fp32 path: blocks are dealt to the layers in proportion to their size.
__global__ void __launch_bounds__(kThreads) k_ema_momentum(const __grid_constant__ EmaArgs a, float beta1) {
  int i = 0;
  while (i + 1 < a.n && (int)blockIdx.x >= a.block_begin[i + 1]) ++i;
  const int block = (int)blockIdx.x - a.block_begin[i], blocks = a.block_begin[i + 1] - a.block_begin[i];
  if (a.j[i].g_is_bf16) ema_one<true>(a.j[i], block, blocks, beta1); else ema_one<false>(a.j[i], block, blocks, beta1);
}

template <bool G_BF16>
__global__ void __launch_bounds__(kThreads)
k_plain_adam(float* __restrict__ W, float* __restrict__ M, float* __restrict__ V,
             const void* __restrict__ G, int64_t numel, float lr, float beta1, float beta2,
             float eps, float decay, const float* __restrict__ gscale) {
  const float gs = gscale ? *gscale : 1.0f;
  const float omb1 = 1.0f - beta1, omb2 = 1.0f - beta2;
  const int64_t nvec = numel >> 2;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nvec; v += stride) {
    const int64_t i = v << 2;
    float4 g = load_grad4<G_BF16>(G, i);
    g.x *= gs; g.y *= gs; g.z *= gs; g.w *= gs;
    float4 m = ld4(M + i), s = ld4(V + i), w = ld4(W + i);
#define BR_ADAM1(c)                                   \
  m.c = beta1 * m.c + omb1 * g.c;                     \
  s.c = beta2 * s.c + omb2 * g.c * g.c;               \
  w.c = decay * w.c - lr * (m.c / sqrtf(s.c + eps));
    BR_ADAM1(x) BR_ADAM1(y) BR_ADAM1(z) BR_ADAM1(w)
#undef BR_ADAM1
    st4(M + i, m);
    st4(V + i, s);
    st4(W + i, w);
  }
  for (int64_t i = (nvec << 2) + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < numel;
       i += stride) {
    float g = gs * load_grad1<G_BF16>(G, i);
    float m = beta1 * M[i] + omb1 * g;
    float s = beta2 * V[i] + omb2 * g * g;
    M[i] = m;
    V[i] = s;
    W[i] = decay * W[i] - lr * (m / sqrtf(s + eps));
  }
}

// One 32 x 32 block pair per CTA of 32 x 8 threads, through a padded shared-memory tile.  Blocks are numbered along
// the columns of the strict upper block triangle (block b of column c, b < c, is number c (c - 1) / 2 + b).  Bound by memory, 8 bytes per pair of entries.
struct MirrorArgs { float* F[kElemGroup]; int k[kElemGroup], begin[kElemGroup + 1], n; };
__global__ void __launch_bounds__(256) k_mirror_lower(const __grid_constant__ MirrorArgs a) {
  __shared__ float tile[32][33];
  int job = 0;
  while (job + 1 < a.n && a.begin[job + 1] <= (int)blockIdx.x) ++job;
  float* const F = a.F[job];
  const int64_t k = a.k[job];
  const int id = (int)blockIdx.x - a.begin[job];
  int c = (int)((sqrtf(8.0f * (float)id + 1.0f) + 1.0f) * 0.5f);
  while (c * (c - 1) / 2 > id) --c;
  while (c * (c + 1) / 2 <= id) ++c;
  const int b = id - c * (c - 1) / 2;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t r0 = 32 * (int64_t)b, c0 = 32 * (int64_t)c;
#pragma unroll
  for (int i = ty; i < 32; i += 8)
    if (c0 + tx < k) tile[i][tx] = F[(r0 + i) * k + c0 + tx];
  __syncthreads();
#pragma unroll
  for (int i = ty; i < 32; i += 8)
    if (c0 + i < k) F[(c0 + i) * k + r0 + tx] = tile[tx][i];
}

struct SplitArgs { SplitJob j[kElemGroup]; int begin[kElemGroup + 1], n; };
__global__ void __launch_bounds__(kThreads)
k_split_bf16(const __grid_constant__ SplitArgs a) {
  int job = 0;
  while (job + 1 < a.n && a.begin[job + 1] <= (int)blockIdx.x) ++job;
  const float* const X = a.j[job].X;
  __nv_bfloat16 *const hi = a.j[job].hi, *const lo = a.j[job].lo;
  const int64_t numel = a.j[job].numel, block = (int)blockIdx.x - a.begin[job];
  const int64_t nvec = numel >> 2;
  const int64_t stride = (int64_t)(a.begin[job + 1] - a.begin[job]) * blockDim.x;
  for (int64_t v = block * blockDim.x + threadIdx.x; v < nvec; v += stride) {
    const int64_t i = v << 2;
    float4 x = ld4(X + i);
    float4 h = make_float4(bf16_round(x.x), bf16_round(x.y), bf16_round(x.z), bf16_round(x.w));
    st4_bf16(hi + i, h);
    if (lo) st4_bf16(lo + i, make_float4(x.x - h.x, x.y - h.y, x.z - h.z, x.w - h.w));
  }
  for (int64_t i = (nvec << 2) + block * blockDim.x + threadIdx.x; i < numel; i += stride) {
    float x = X[i], h = bf16_round(x);
    hi[i] = __float2bfloat16_rn(x);
    if (lo) lo[i] = __float2bfloat16_rn(x - h);
  }
}

__global__ void __launch_bounds__(kThreads)
k_widen_bf16(const __nv_bfloat16* __restrict__ X, float* __restrict__ out, int64_t numel) {
  const int64_t nvec = numel >> 2;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nvec; v += stride) {
    const int64_t i = v << 2;
    st4(out + i, ld4_bf16(X + i));
  }
  for (int64_t i = (nvec << 2) + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < numel;
       i += stride)
    out[i] = __bfloat162float(X[i]);
}

// out <- beta1 M + (1-beta1) G, M untouched (M_t for a refresh that reads the momentum)
template <bool G_BF16>
__global__ void __launch_bounds__(kThreads)
k_ema_out(float* __restrict__ out, const float* __restrict__ M, const void* __restrict__ G, int64_t numel,
          float beta1, const float* __restrict__ gscale) {
  const float omb = (1.0f - beta1) * (gscale ? *gscale : 1.0f);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nvec = numel >> 2;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nvec; v += stride) {
    const int64_t i = v << 2;
    const float4 g = load_grad4<G_BF16>(G, i);
    float4 m = ld4(M + i);
    m.x = beta1 * m.x + omb * g.x; m.y = beta1 * m.y + omb * g.y;
    m.z = beta1 * m.z + omb * g.z; m.w = beta1 * m.w + omb * g.w;
    st4(out + i, m);
  }
  for (int64_t i = (nvec << 2) + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < numel; i += stride)
    out[i] = beta1 * M[i] + omb * load_grad1<G_BF16>(G, i);
}

// Global-norm clipping factor of one call (App. D.2): sum of squares over all layers' gradients in a
// fixed order (each CTA a contiguous share of the concatenated gradients, tree inside the CTA, then one
// CTA over the CTAs' sums), then factor = min(1, clip / norm).  Bound by the read of the gradients: 16-byte loads,
// four in flight per thread; a share that does not start on a 16-byte boundary begins and ends with single elements.
// The four matrices of a d = 1024 block (25 MB): 12.5 us and 2.3 us for the two launches; 22.6 and 10.9 with loads of two
// bytes and one thread over the CTAs.
__device__ __forceinline__ double tree_sum(double* sh, double v) {
  sh[threadIdx.x] = v;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  return sh[0];
}
template <bool BF16>
__device__ __forceinline__ double sum_squares(const void* ptr, long long a, long long b) {
  constexpr int V = BF16 ? 8 : 4;              // elements of a 16-byte load
  constexpr int U = 4;
  auto one = [&](long long i) { return (double)(BF16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(ptr)[i]) : reinterpret_cast<const float*>(ptr)[i]); };
  double acc[2] = {0.0, 0.0};
  const long long off = (long long)((reinterpret_cast<uintptr_t>(ptr) + (uintptr_t)a * (BF16 ? 2 : 4)) % 16) / (BF16 ? 2 : 4);
  const long long head = min(b, a + (off ? V - off : 0)), nv = (b - head) / V;
  if (a + threadIdx.x < head) { const double v = one(a + threadIdx.x); acc[0] = v * v; }
  const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const char*>(ptr) + head * (BF16 ? 2 : 4));
  for (long long i = threadIdx.x; i < nv; i += U * kThreads) {
    uint4 q[U];
#pragma unroll
    for (int u = 0; u < U; ++u) q[u] = i + u * kThreads < nv ? __ldg(p + i + u * kThreads) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const uint32_t w = c == 0 ? q[u].x : c == 1 ? q[u].y : c == 2 ? q[u].z : q[u].w;
        if (BF16) {
          const double lo = (double)__uint_as_float(w << 16), hi = (double)__uint_as_float(w & 0xffff0000u);
          acc[0] = fma(lo, lo, acc[0]); acc[1] = fma(hi, hi, acc[1]);
        } else {
          const double v = (double)__uint_as_float(w);
          acc[c & 1] = fma(v, v, acc[c & 1]);
        }
      }
  }
  const long long tail = head + nv * V + threadIdx.x;
  if (tail < b) { const double v = one(tail); acc[1] = fma(v, v, acc[1]); }
  return acc[0] + acc[1];
}
template <int NSEG>
__global__ void __launch_bounds__(kThreads)
k_clip_partial(ClipSegs<NSEG> segs, int nseg, double* __restrict__ part) {
  __shared__ double sh[kThreads];
  const long long total = segs.begin[nseg];
  const long long chunk = (total + gridDim.x - 1) / gridDim.x;
  const long long lo = (long long)blockIdx.x * chunk;
  const long long hi = lo + chunk < total ? lo + chunk : total;
  double acc = 0.0;
  int sg = 0;
  while (sg < nseg && segs.begin[sg + 1] <= lo) ++sg;
  for (; sg < nseg && segs.begin[sg] < hi; ++sg) {
    const long long a = (lo > segs.begin[sg] ? lo : segs.begin[sg]) - segs.begin[sg];
    const long long b = (hi < segs.begin[sg + 1] ? hi : segs.begin[sg + 1]) - segs.begin[sg];
    acc += segs.bf16[sg] ? sum_squares<true>(segs.ptr[sg], a, b) : sum_squares<false>(segs.ptr[sg], a, b);
  }
  acc = tree_sum(sh, acc);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}
__global__ void __launch_bounds__(kThreads) k_clip_final(const double* __restrict__ part, int n, float clip, float* __restrict__ out) {
  __shared__ double sh[kThreads];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += kThreads) s += part[i];
  const double nrm = sqrt(tree_sum(sh, s));
  if (threadIdx.x) return;
  *out = (nrm > (double)clip) ? (float)((double)clip / nrm) : 1.0f;
}

// Copies (a call's gradients into the ring) that run beside the last contraction launches of a step: one CTA of 256 threads and
// 40 registers per SM is what fits next to one of those.  One cudaMemcpyAsync per gradient takes 2.7 us each at the sizes of a
// d = 384 layer, 43 us a step.
constexpr int kCopyThreads = 256, kCopyLoads = 4;
struct CopyArgs { CopyJob j[kElemGroup]; long long begin[kElemGroup + 1]; int n; };     // begin: in 16-byte pieces
__global__ void __launch_bounds__(kCopyThreads, 6) k_ring_copy(const __grid_constant__ CopyArgs a) {
  const long long total = a.begin[a.n], stride = (long long)gridDim.x * kCopyThreads;
  int job = 0;
  for (long long i = (long long)blockIdx.x * kCopyThreads + threadIdx.x; i < total; i += kCopyLoads * stride) {
    uint4 v[kCopyLoads];
    uint4* d[kCopyLoads];
#pragma unroll
    for (int u = 0; u < kCopyLoads; ++u) {
      const long long at = i + u * stride;
      d[u] = nullptr;
      if (at >= total) continue;
      while (a.begin[job + 1] <= at) ++job;
      const CopyJob& j = a.j[job];
      const size_t off = (size_t)(at - a.begin[job]) * 16;
      const char* s = static_cast<const char*>(j.src) + off;
      if (off + 16 <= j.bytes) {
        v[u] = __ldg(reinterpret_cast<const uint4*>(s));
        d[u] = reinterpret_cast<uint4*>(static_cast<char*>(j.dst) + off);
      } else {                                 // the last piece (gradients start on 16-byte boundaries, slots on 256-byte ones)
        for (size_t b = off; b < off + 16 && b < j.bytes; b += 2)
          *reinterpret_cast<uint16_t*>(static_cast<char*>(j.dst) + b) = *reinterpret_cast<const uint16_t*>(static_cast<const char*>(j.src) + b);
      }
    }
#pragma unroll
    for (int u = 0; u < kCopyLoads; ++u) if (d[u]) *d[u] = v[u];
  }
}

// x (rounded to fp32) = p1 + p2 + p3 with three bf16 terms: all 24 significant bits survive.
__device__ __forceinline__ void split3(float f, __nv_bfloat16& p1, __nv_bfloat16& p2, __nv_bfloat16& p3) {
  const float h1 = bf16_round(f);
  const float r1 = f - h1;
  const float h2 = bf16_round(r1);
  const float r2 = r1 - h2;
  p1 = __float2bfloat16_rn(h1); p2 = __float2bfloat16_rn(h2); p3 = __float2bfloat16_rn(r2);
}

// Four columns per thread (widths are multiples of 8 and rows start on 16-byte boundaries), 32-bit index arithmetic.
// SUB: A -= D first (D fp32, compact); SPLIT: the three planes (compact).  Both in one pass between the two passes of a projection.
struct alignas(8) bf16x4 { __nv_bfloat16 v[4]; };
__device__ __forceinline__ void split3x4(const float (&x)[4], int64_t i, __nv_bfloat16* p1, __nv_bfloat16* p2, __nv_bfloat16* p3) {
  bf16x4 a, b, c;
#pragma unroll
  for (int u = 0; u < 4; ++u) split3(x[u], a.v[u], b.v[u], c.v[u]);
  *reinterpret_cast<bf16x4*>(p1 + i) = a;
  *reinterpret_cast<bf16x4*>(p2 + i) = b;
  *reinterpret_cast<bf16x4*>(p3 + i) = c;
}
template <bool SUB, bool SPLIT>
__global__ void __launch_bounds__(kThreads)
k_sub_split3(double* __restrict__ A, int64_t ld, unsigned groups, unsigned per_row, const float* __restrict__ D,
             __nv_bfloat16* __restrict__ p1, __nv_bfloat16* __restrict__ p2, __nv_bfloat16* __restrict__ p3) {
  for (unsigned g = blockIdx.x * kThreads + threadIdx.x; g < groups; g += gridDim.x * kThreads) {
    const unsigned r = g / per_row, c = 4 * (g - r * per_row);
    double2* const at = reinterpret_cast<double2*>(A + (int64_t)r * ld + c);
    double2 lo = at[0], hi = at[1];
    if (SUB) {
      const float4 d = *reinterpret_cast<const float4*>(D + 4 * (int64_t)g);
      lo.x -= (double)d.x; lo.y -= (double)d.y; hi.x -= (double)d.z; hi.y -= (double)d.w;
      at[0] = lo; at[1] = hi;
    }
    if (SPLIT) {
      const float x[4] = {(float)lo.x, (float)lo.y, (float)hi.x, (float)hi.y};
      split3x4(x, 4 * (int64_t)g, p1, p2, p3);
    }
  }
}
// the sum of `parts` compact arrays (4 * groups entries each) into planes; summed in fp64
__global__ void __launch_bounds__(kThreads)
k_split3_f32(const float* __restrict__ X, unsigned groups, int parts, __nv_bfloat16* __restrict__ p1,
             __nv_bfloat16* __restrict__ p2, __nv_bfloat16* __restrict__ p3) {
  for (unsigned g = blockIdx.x * kThreads + threadIdx.x; g < groups; g += gridDim.x * kThreads) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int z = 0; z < parts; ++z) {
      const float4 v = *reinterpret_cast<const float4*>(X + 4 * ((int64_t)z * groups + g));
      s[0] += (double)v.x; s[1] += (double)v.y; s[2] += (double)v.z; s[3] += (double)v.w;
    }
    const float x[4] = {(float)s[0], (float)s[1], (float)s[2], (float)s[3]};
    split3x4(x, 4 * (int64_t)g, p1, p2, p3);
  }
}

__global__ void __launch_bounds__(kThreads)
k_f32_to_f64(const float* __restrict__ X, double* __restrict__ out, int64_t numel) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < numel; i += stride)
    out[i] = (double)X[i];
}

__global__ void __launch_bounds__(kThreads)
k_f64_to_f32(const double* __restrict__ X, float* __restrict__ out, int64_t numel) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < numel; i += stride)
    out[i] = (float)X[i];
}

}  // namespace

cudaError_t set_identity(float* Q, int64_t k, cudaStream_t s) {
  k_set_identity<<<grid_for(k * k), kThreads, 0, s>>>(Q, k);
  return cudaGetLastError();
}

cudaError_t ring_copy(const CopyJob* jobs, int n, bool beside, cudaStream_t s) {
  for (int first = 0; first < n; first += kElemGroup) {
    CopyArgs a;
    a.n = std::min(kElemGroup, n - first);
    a.begin[0] = 0;
    for (int i = 0; i < a.n; ++i) {
      a.j[i] = jobs[first + i];
      a.begin[i + 1] = a.begin[i] + (long long)((a.j[i].bytes + 15) / 16);
    }
    const long long want = (a.begin[a.n] + kCopyThreads - 1) / kCopyThreads;
    k_ring_copy<<<(unsigned)std::min<long long>(want, 148 * (beside ? 1 : 6)), kCopyThreads, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t mirror_lower(const MirrorJob* jobs, int n, cudaStream_t s) {
  for (int first = 0; first < n; first += kElemGroup) {
    MirrorArgs a;
    a.n = std::min(kElemGroup, n - first);
    a.begin[0] = 0;
    for (int i = 0; i < a.n; ++i) {
      const int nb = (int)((jobs[first + i].k + 31) / 32);
      a.F[i] = jobs[first + i].F; a.k[i] = (int)jobs[first + i].k;
      a.begin[i + 1] = a.begin[i] + nb * (nb - 1) / 2;
    }
    if (a.begin[a.n]) k_mirror_lower<<<(unsigned)a.begin[a.n], 256, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t ema_momentum(const EmaJob* jobs, int n, float beta1, cudaStream_t s) {
  EmaArgs a;
  for (int at = 0; at < n; at += kMaxEmaJobs) {
    a.n = n - at < kMaxEmaJobs ? n - at : kMaxEmaJobs;
    int blocks = 0;
    for (int i = 0; i < a.n; ++i) {
      a.j[i] = jobs[at + i];
      a.block_begin[i] = blocks;
      blocks += grid_for((a.j[i].numel + 3) / 4);
    }
    a.block_begin[a.n] = blocks;
    k_ema_momentum<<<blocks, kThreads, 0, s>>>(a, beta1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t plain_adam(float* W, float* M, float* V, const void* G, int g_is_bf16, int64_t numel,
                       float lr, float beta1, float beta2, float eps, float wd, const float* gscale, cudaStream_t s) {
  int grid = grid_for((numel + 3) / 4);
  float decay = 1.0f - lr * wd;
  if (g_is_bf16)
    k_plain_adam<true><<<grid, kThreads, 0, s>>>(W, M, V, G, numel, lr, beta1, beta2, eps, decay, gscale);
  else
    k_plain_adam<false><<<grid, kThreads, 0, s>>>(W, M, V, G, numel, lr, beta1, beta2, eps, decay, gscale);
  return cudaGetLastError();
}

cudaError_t split_bf16(const SplitJob* jobs, int n, cudaStream_t s) {
  for (int first = 0; first < n; first += kElemGroup) {
    SplitArgs a;
    a.n = std::min(kElemGroup, n - first);
    a.begin[0] = 0;
    for (int i = 0; i < a.n; ++i) {
      a.j[i] = jobs[first + i];
      a.begin[i + 1] = a.begin[i] + grid_for((a.j[i].numel + 3) / 4);
    }
    k_split_bf16<<<(unsigned)a.begin[a.n], kThreads, 0, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t widen_bf16(const __nv_bfloat16* X, float* out, int64_t numel, cudaStream_t s) {
  k_widen_bf16<<<grid_for((numel + 3) / 4), kThreads, 0, s>>>(X, out, numel);
  return cudaGetLastError();
}

cudaError_t ema_out(float* out, const float* M, const void* G, int g_is_bf16, int64_t numel, float beta1,
                    const float* gscale, cudaStream_t s) {
  const int grid = grid_for((numel + 3) / 4);
  if (g_is_bf16) k_ema_out<true><<<grid, kThreads, 0, s>>>(out, M, G, numel, beta1, gscale);
  else k_ema_out<false><<<grid, kThreads, 0, s>>>(out, M, G, numel, beta1, gscale);
  return cudaGetLastError();
}

cudaError_t clip_factor(const void* const* grads, const int64_t* numel, const int* is_bf16, int n, float clip,
                        double* part, float* out, cudaStream_t s) {
  constexpr int NSEG = 64, GRID = 296;
  int launches = 0;
  for (int first = 0; first < n; first += NSEG, ++launches) {
    ClipSegs<NSEG> segs;
    const int cnt = (n - first < NSEG) ? n - first : NSEG;
    segs.begin[0] = 0;
    for (int i = 0; i < cnt; ++i) {
      segs.ptr[i] = grads[first + i];
      segs.bf16[i] = is_bf16[first + i];
      segs.begin[i + 1] = segs.begin[i] + numel[first + i];
    }
    k_clip_partial<NSEG><<<GRID, kThreads, 0, s>>>(segs, cnt, part + (size_t)launches * GRID);
  }
  k_clip_final<<<1, kThreads, 0, s>>>(part, launches * GRID, clip, out);
  return cudaGetLastError();
}

cudaError_t sub_split3(double* A, int64_t ld, int64_t rows, int64_t cols, const float* D, __nv_bfloat16* p1, __nv_bfloat16* p2,
                       __nv_bfloat16* p3, cudaStream_t s) {
  if (cols % 4 || ld % 2 || rows * cols / 4 > 0xffffffffll - (1 << 22)) return cudaErrorInvalidValue;
  const unsigned groups = (unsigned)(rows * cols / 4), per_row = (unsigned)(cols / 4);
  const int grid = grid_for(groups);
  if (D && p1) k_sub_split3<true, true><<<grid, kThreads, 0, s>>>(A, ld, groups, per_row, D, p1, p2, p3);
  else if (D) k_sub_split3<true, false><<<grid, kThreads, 0, s>>>(A, ld, groups, per_row, D, p1, p2, p3);
  else k_sub_split3<false, true><<<grid, kThreads, 0, s>>>(A, ld, groups, per_row, D, p1, p2, p3);
  return cudaGetLastError();
}
cudaError_t split3_f32(const float* X, int64_t numel, int parts, __nv_bfloat16* p1, __nv_bfloat16* p2, __nv_bfloat16* p3,
                       cudaStream_t s) {
  if (numel % 4 || numel / 4 > 0xffffffffll - (1 << 22)) return cudaErrorInvalidValue;
  k_split3_f32<<<grid_for(numel / 4), kThreads, 0, s>>>(X, (unsigned)(numel / 4), parts, p1, p2, p3);
  return cudaGetLastError();
}

cudaError_t f32_to_f64(const float* X, double* out, int64_t numel, cudaStream_t s) {
  k_f32_to_f64<<<grid_for(numel), kThreads, 0, s>>>(X, out, numel);
  return cudaGetLastError();
}

cudaError_t f64_to_f32(const double* X, float* out, int64_t numel, cudaStream_t s) {
  k_f64_to_f32<<<grid_for(numel), kThreads, 0, s>>>(X, out, numel);
  return cudaGetLastError();
}

// ---- debug canaries: 256-byte guard words behind every piece of the handle's slab ----
namespace {
constexpr unsigned int kGuardWord = 0xC5C5C5C5u;
__global__ void k_guard_fill(char* slab, const unsigned long long* offs, int n) {
  const int g = blockIdx.x;
  if (g < n) reinterpret_cast<unsigned int*>(slab + offs[g])[threadIdx.x] = kGuardWord;
}
__global__ void k_guard_check(const char* slab, const unsigned long long* offs, int n, int* first_bad) {
  const int g = blockIdx.x;
  if (g < n && reinterpret_cast<const unsigned int*>(slab + offs[g])[threadIdx.x] != kGuardWord) atomicMin(first_bad, g);
}
}  // namespace

cudaError_t guard_fill(char* slab, const unsigned long long* offs, int n, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_guard_fill<<<n, 64, 0, s>>>(slab, offs, n);
  return cudaGetLastError();
}
cudaError_t guard_check(const char* slab, const unsigned long long* offs, int n, int* first_bad, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_guard_check<<<n, 64, 0, s>>>(slab, offs, n, first_bad);
  return cudaGetLastError();
}

}  // namespace br
