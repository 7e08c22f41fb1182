// Grouped bf16 contraction on the 5th-generation tensor cores (sm_100a):
//   D_tile = sum over operand pairs p and k-blocks of A_p[128 x 64] * B_p[256 x 64]^T
// TMA (cp.async.bulk.tensor, 128-byte swizzle) stages operand tiles in shared memory, one elected
// thread issues tcgen05.mma (kind::f16, bf16 operands, fp32 accumulation) into tensor memory,
// eight epilogue warps read the accumulator back with tcgen05.ld, turn it through shared memory so
// that global memory is accessed along rows, and apply a fused epilogue
// (factor EMA, bf16 hi/lo split, second-moment update, Adam scaling, weight write).
//
// A problem may sum several operand pairs into one tile (the bf16 hi/lo products of an fp32
// operand).  When the pairs are combinations of at most two distinct A and two distinct B operands
// (hi*hi + lo*hi + hi*lo), the kernel runs in its shared-operand form: a stage holds one k-block of
// every distinct operand (2 x 16 KiB + 2 x 32 KiB) and all combinations are issued from it, so each
// operand tile is fetched from L2 once per k-block instead of once per pair.
//
// One persistent CTA per SM walks a static tile list that spans every problem of a launch
// (all layers of one phase of the step), so small and large matrices share one launch; the lists are made on
// the host, longest tiles first (make_schedule).
// Two 256-column accumulators in tensor memory let the epilogue of a tile overlap the main
// loop of the next one.
//
// Operands may be K-major (K contiguous) or MN-major (M / N contiguous); the latter is how the
// row-major G, U, V enter products that contract over their row index (G^T G, U^T G, T V).
// Every tensor map is 3-D; the third coordinate selects a ring slot for operands that live in
// the stale-gradient ring and is 0 otherwise.
//
// Paired form (cta_group::2).  Two CTAs of a cluster, on neighbouring SMs, work on one 256 x 256
// tile: each stages its own 128 rows of A and only half of B (128 of the 256 result columns), the
// leader (cluster rank 0) issues tcgen05.mma.cta_group::2 of shape 256 x 256 x 16, which reads both
// halves of B from the two shared memories and leaves rows 0..127 of the accumulator in the leader's
// tensor memory and rows 128..255 in the peer's.  Per flop this takes two thirds of the L2 -> shared
// memory traffic and half of the shared-memory reads of B, which is what bounds the unpaired form.
// Barriers: both CTAs' TMA transactions complete on the leader's "full" barrier; the leader's
// commits arrive on the "empty" and "accumulator full" barriers of both CTAs (one commit per CTA, the
// peer's barrier addressed through mapa); the epilogue warps of both CTAs arrive on the leader's
// "accumulator empty" barrier.  Both CTAs meet at a cluster barrier after set-up and before they free
// their tensor memory, so neither exits while the other can still signal it.
//
// Folded form (factor products G G^T, G^T G).  The tensor core truncates its fp32 accumulator once
// per instruction (16-deep slice of the contraction), a one-sided error that grows with the length of
// the chain and with the size of the partial sums: 0.3 (K / 16) 2^-24 relative for contraction length
// K, 3e-6 at K = 2560.  The factors feed Power(), whose trailing basis vectors come out of a
// cancellation against eigenvalues 1e5 times larger, and an error of that size moves them by 1e-2.
// In this form the contraction is cut into chunks of a few k-blocks; the chunks are accumulated from
// zero, alternately in the two tensor-memory buffers, and eight epilogue warps (two per lane quadrant,
// 128 result columns each) add every finished chunk, round to nearest on the CUDA cores, to a running
// sum they keep in registers, while the tensor core is already working on the next chunk.  Chains
// are 8 to 16 instructions on partial sums a tenth the size: the error drops by the number of chunks.
// The final epilogue (factor EMA) runs from the registers while the first two chunks of the next tile
// accumulate.  It is bound by the traffic between L2 and the SMs, which all of them cause at the same time:
// 19 to 25 thousand cycles a tile when it wrote the mirror image of every block as well, against 26 thousand
// for the chunks of a tile of K = 2560.
//
// Every wait on an mbarrier is bounded: when a wait gives up the CTA raises an abort flag,
// records BR_ERR_TIMEOUT in the status word, leaves its loops, outlasts its copies in flight, frees its
// tensor memory and returns; later launches return at once while the status word is negative.
#include <cuda.h>

#include <cstdlib>
#include <algorithm>
#include <cstring>
#include <functional>
#include <mutex>
#include <queue>
#include <string>
#include <vector>

#include "br_internal.h"
#include "tc_ptx.h"

namespace br {

namespace {

constexpr int BM = 128, BN = 256, BK = 64;       // tile (elements); BK*2 bytes = one 128-byte swizzle row
constexpr int UMMA_K = 16;
constexpr int A_BYTES = BM * BK * 2;             // 16 KiB
// Steps with four epilogue warps of 256 columns each: one block of d = 1024 745 us instead of 602, four of d = 384 402 and 324, one of
// d = 2048 with its embedding 4.05 and 3.59 ms, four of d = 2560 22.1 and 20.4 ms.
constexpr int EPI_WARPS = 8;
constexpr int EPI_BYTES = EPI_WARPS * 32 * 32 * 4;   // one 32 x 32 fp32 block per epilogue warp
constexpr int OPERAND_BYTES = 192 * 1024;            // operand stages in the shared-operand form
// 160 KiB in the others.  A sixth stage in the plain form: four blocks of d = 2560 0.7 % shorter, four of d = 384 1.1 % longer, one of d = 2048
// 0.6 % longer; unpaired, three stages against four: d = 1024 0.9 % longer, d = 384 1.0 % shorter, d = 2048 the same.  With a limit of 128
// registers (launch bounds of 512 threads; no rotated Adam, whose problems always sum operand pairs) the plain form also leaves a
// quarter of each sub-partition's registers: the copies of the gradients into the ring run beside the last two phases of a step.
// At 168 registers three warps fill a sub-partition, and the copies kept the weight-write launch waiting (four blocks of
// d = 2560: 21.4 ms a step instead of 20.1).
constexpr int PLAIN_OPERAND_BYTES = 160 * 1024;
constexpr int SMEM_BYTES = OPERAND_BYTES + EPI_BYTES + 1024;          // + slack to align the tiles to 1 KiB
constexpr int SMEM_BYTES_PLAIN = PLAIN_OPERAND_BYTES + EPI_BYTES + 1024;
constexpr int MAX_STAGES = 5;
// Per-form geometry.  PAIR: the CTA pair owns a 256-row tile, each CTA stages 128 columns of B.
template <bool SHARED, bool PAIR>
struct Form {
  static constexpr int TM = PAIR ? 2 * BM : BM;                 // rows of a tile
  static constexpr int BNC = PAIR ? BN / 2 : BN;                // result columns whose B rows this CTA stages
  static constexpr int BB = BNC * BK * 2;                       // bytes of one staged B tile
  static constexpr int STAGE = SHARED ? 2 * A_BYTES + 2 * BB : A_BYTES + BB;
  static constexpr int OPERANDS = SHARED ? OPERAND_BYTES : PLAIN_OPERAND_BYTES;
  static constexpr int NST = OPERANDS / STAGE;                  // 3 / 2 unpaired, 5 / 3 paired
  static_assert(NST <= MAX_STAGES, "barriers");
};
constexpr int TMEM_COLS = 512;
constexpr int NUM_THREADS = 64 + 32 * EPI_WARPS; // warp 0: TMA, warp 1: MMA, warps 2..9: epilogue (two per lane quadrant)
// folded form: two blocks of 32 x 32 floats for each of its eight epilogue warps
constexpr int FOLD_BLOCK = 32 * 32;
constexpr int SMEM_BYTES_FOLD = PLAIN_OPERAND_BYTES + EPI_WARPS * 2 * FOLD_BLOCK * 4 + 1024;
constexpr int MAX_PAIRS = 3;
// Fixed part of a tile's cost in the schedule (see make_schedule), plain and folded form.  Steady steps with 6 and 24, 3 and 24, 12 and 24,
// 6 and 12, 6 and 48: one block of d = 1024 602 to 604 us, four of d = 384 324 to 325 us, one of d = 2048 with its embedding 3.58 to 3.60 ms, four
// of d = 2560 20.3 to 20.5 ms, in no order (0 and 0, with an epilogue of four warps: 2 to 6 % longer).
constexpr int kTileCost = 6, kFoldTileCost = 24;
// Tile rasterisation: a group of row-blocks (or, transposed, of column-blocks) is swept across the
// other dimension, so that the group's operand panel stays in L2 while the other operand streams
// through once per group.  The host picks orientation and group size per problem (see plan creation).
constexpr double kL2PanelBytes = 40e6;           // what one resident operand panel may take of the 126 MB L2

struct alignas(128) DevProblem {
  CUtensorMap mapA[MAX_PAIRS];
  CUtensorMap mapB[MAX_PAIRS];
  int32_t Md, Nd, K, n_pairs;
  int32_t a_mn, b_mn, epilogue, tiles_m;
  int32_t tiles_n, tile_begin, tile_count, tau_max;
  int32_t ring_slots, a_ring_mask, b_ring_mask, dyn_scalars;
  float alpha, beta, eps, beta1;
  float* D;
  long long ldd;
  __nv_bfloat16* Dh;
  __nv_bfloat16* Dl;
  long long ldh;
  float* D2;
  // shared-operand form: mapA[0..nA) / mapB[0..nB) are the distinct operands, `combos` lists the
  // products to issue per k-block: bits 8.. = count, bits 2c, 2c+1 = (A index, B index) of product c
  int32_t symmetric, nA, nB, combos;
  int32_t group, raster_n;        // blocks per group; 0: groups of row-blocks, 1: groups of column-blocks
  int32_t tri;                    // symmetric product with square tiles: the tile list holds the upper triangle only
  const float* clip;              // clipping factors by call (see TcProblem::clip_mode), or null
  int32_t clip_slots, clip_mode;
  int32_t fold_kb;                // folded form: k-blocks per chunk
};

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// paired form: `bar` is a shared::cluster address (this CTA's barrier or the peer's)
__device__ __forceinline__ void umma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
// Shared-memory matrix descriptor, 128-byte swizzle.  lbo / sbo in bytes.
//   K-major : rows of 128 bytes (64 elements of K); 8-row groups 1024 bytes apart (sbo); lbo unused.
//   MN-major: rows of 128 bytes (64 elements of M/N), one row per k; 8-k groups sbo apart,
//             64-element M/N blocks lbo apart.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;     // descriptor version of this architecture
  d |= 2ull << 61;     // 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, M = 128, N = 256.
__device__ __forceinline__ uint32_t make_idesc(int a_mn, int b_mn, int rows = BM) {
  uint32_t d = 0;
  d |= 1u << 4;                       // accumulator format: fp32
  d |= 1u << 7;                       // A format: bf16
  d |= 1u << 10;                      // B format: bf16
  d |= (uint32_t)(a_mn ? 1 : 0) << 15;
  d |= (uint32_t)(b_mn ? 1 : 0) << 16;
  d |= (uint32_t)(BN >> 3) << 17;
  d |= (uint32_t)(rows >> 4) << 24;
  return d;
}

__device__ __forceinline__ uint32_t pack2_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}

struct TileInfo {
  const DevProblem* p;
  int m0, n0, z;
  bool active;
};

// tile index -> problem (`problem`, or where that is negative by a binary search over tile_begin) and block coordinates
template <int TM>
__device__ __forceinline__ TileInfo locate_tile(const DevProblem* probs, int n_probs, int tile, int problem,
                                                long long calls, int tau) {
  int lo = problem, hi = problem;
  if (problem < 0) { lo = 0; hi = n_probs - 1; }
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (probs[mid].tile_begin <= tile) lo = mid; else hi = mid - 1;
  }
  const DevProblem* p = probs + lo;
  TileInfo ti;
  ti.p = p;
  const int local = tile - p->tile_begin;
  if (p->tri) {
    // upper triangle, column by column: column c holds the row-blocks 0..c at positions c (c + 1) / 2 + r
    int c = (int)((sqrtf(8.0f * (float)local + 1.0f) - 1.0f) * 0.5f);
    while ((c + 1) * (c + 2) / 2 <= local) ++c;
    while (c * (c + 1) / 2 > local) --c;
    ti.m0 = (local - c * (c + 1) / 2) * TM;
    ti.n0 = c * BN;
    const int tl = tau < 0 ? p->tau_max : tau;
    ti.active = (calls - tl >= 1);
    ti.z = 0;
    if (p->ring_slots > 0 && ti.active) ti.z = (int)((calls - 1 - tl) % p->ring_slots);
    return ti;
  }
  const int g = p->group;
  const int across = p->raster_n ? p->tiles_m : p->tiles_n;      // blocks of the swept dimension
  const int along = p->raster_n ? p->tiles_n : p->tiles_m;       // blocks of the grouped dimension
  const int per_group = g * across;
  const int group = local / per_group;
  const int first = group * g;
  const int gsz = min(along - first, g);
  const int in_group = local - group * per_group;
  const int blk_g = first + in_group % gsz, blk_s = in_group / gsz;
  ti.m0 = (p->raster_n ? blk_s : blk_g) * TM;
  ti.n0 = (p->raster_n ? blk_g : blk_s) * BN;
  // delayed-gradient bookkeeping: the layer is active once call - tau >= 1; the gradient to
  // apply sits in ring slot (calls - 1 - tau) mod slots
  const int tl = tau < 0 ? p->tau_max : tau;
  ti.active = (calls - tl >= 1);
  // a symmetric product is computed on the tiles that touch the upper triangle only
  if (p->symmetric && ti.m0 >= ti.n0 + BN) ti.active = false;
  ti.z = 0;
  if (p->ring_slots > 0 && ti.active) ti.z = (int)((calls - 1 - tl) % p->ring_slots);
  return ti;
}

// ---------------------------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------------------------
template <bool SHARED, bool PAIR, bool FOLD = false>
__global__ void __launch_bounds__(SHARED || FOLD ? NUM_THREADS : 512, 1)
k_tc_gemm(const DevProblem* __restrict__ probs, int n_probs, int first_tile, int total_tiles, const int* __restrict__ schedule,
          long long calls, int tau, float dyn_alpha, float dyn_beta, int* status) {
  using F = Form<SHARED, PAIR>;
  constexpr int NST = F::NST;
  constexpr int TM = F::TM;
  extern __shared__ uint8_t smem_raw[];
  __shared__ alignas(8) uint64_t bars[2 * MAX_STAGES + 4];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  __shared__ uint32_t dead_word;
  volatile int* abort_flag = &abort_word;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;        // 0: leader of the pair
  const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;      // index of this CTA (pair) in the tile walk
  const int n_units = PAIR ? (int)(gridDim.x >> 1) : (int)gridDim.x;
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  // operand slot i of stage s
  auto sA = [&](int s, int i) {
    return SHARED ? tiles_base + (uint32_t)s * F::STAGE + (uint32_t)i * A_BYTES
                  : tiles_base + (uint32_t)s * A_BYTES;
  };
  auto sB = [&](int s, int i) {
    return SHARED ? tiles_base + (uint32_t)s * F::STAGE + 2u * A_BYTES + (uint32_t)i * F::BB
                  : tiles_base + (uint32_t)NST * A_BYTES + (uint32_t)s * F::BB;
  };
  float* epi_tiles = reinterpret_cast<float*>(smem_raw + ((tiles_base - smem_u32(smem_raw)) + (uint32_t)F::OPERANDS));
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (MAX_STAGES + s); };
  auto tfull_bar = [&](int a) { return bar0 + 8u * (2 * MAX_STAGES + a); };
  auto tempty_bar = [&](int a) { return bar0 + 8u * (2 * MAX_STAGES + 2 + a); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    // accumulator hand-back: every epilogue warp, of both CTAs in the paired form
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), (PAIR ? 2 : 1) * EPI_WARPS); }
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if (PAIR) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(TMEM_COLS) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  // an earlier launch failed: nothing to do
  if (threadIdx.x == 0) dead_word = (*reinterpret_cast<volatile int*>(status) < 0) ? 1u : 0u;
  tc_fence_before();
  __syncthreads();
  bool dead = dead_word != 0u;
  if (PAIR) {
    // both CTAs have initialised their barriers before either signals the other; the pair skips its
    // work together when the leader saw a failed status word
    cluster_barrier();
    dead = ld_cluster_u32(map_to_cta(smem_u32(&dead_word), 0)) != 0u;
  }
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&tmem_slot);
  // this unit's tiles: entries [walk_begin, walk_end) of the schedule's list behind its n_units + 1 offsets, with their problems
  // in a second list behind that, or, without a schedule, every n_units-th tile of the range.  A dead pair finds an empty list in every role.
  const int walk_begin = schedule ? schedule[unit] : first_tile + unit, walk_step = schedule ? 1 : n_units;
  const int walk_end = dead ? walk_begin : schedule ? schedule[unit + 1] : total_tiles;
  auto tile_at = [&](int i) {
    const int* at = schedule + n_units + 1 + i;
    return locate_tile<TM>(probs, n_probs, schedule ? at[0] : i, schedule ? at[total_tiles] : -1, calls, tau);
  };

  if (warp == 0) {
    // ======================= TMA producer =======================
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      // paired form: the CTA's own rows of A and its half of the rows of B; every transaction of
      // the pair completes on the leader's barrier, on which only the leader posts the byte count
      const int row_off = (int)rank * BM, col_off = (int)rank * F::BNC;
      auto load = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y, int z) {
        if (PAIR) tma_load_3d_pair(dst, map, bar, x, y, z); else tma_load_3d(dst, map, bar, x, y, z);
      };
      for (int wi = walk_begin; wi < walk_end && !*abort_flag; wi += walk_step) {
        const TileInfo ti = tile_at(wi);
        if (!ti.active) continue;
        const DevProblem* p = ti.p;
        // (copies: the barriers' memory clobbers would have every use in the loops read the problem again, out of L2 since
        // the operand stages leave three KB of L1; the first-side launch of four d = 2560 blocks 4.75 -> 4.5 ms)
        const int nkb = (p->K + BK - 1) / BK, nA = p->nA, nB = p->nB, n_pairs = p->n_pairs;
        const int a_mn = p->a_mn, b_mn = p->b_mn, a_ring = p->a_ring_mask, b_ring = p->b_ring_mask;
        bool ok = true;
        auto load_a = [&](uint32_t dst, const CUtensorMap* ma, int k0, int za, uint32_t bar) {
          if (a_mn) {
#pragma unroll
            for (int j = 0; j < BM / 64; ++j) load(dst + j * (BK * 128), ma, bar, ti.m0 + row_off + 64 * j, k0, za);
          } else {
            load(dst, ma, bar, k0, ti.m0 + row_off, za);
          }
        };
        auto load_b = [&](uint32_t dst, const CUtensorMap* mb, int k0, int zb, uint32_t bar) {
          if (b_mn) {
#pragma unroll
            for (int j = 0; j < F::BNC / 64; ++j) load(dst + j * (BK * 128), mb, bar, ti.n0 + col_off + 64 * j, k0, zb);
          } else {
            load(dst, mb, bar, k0, ti.n0 + col_off, zb);
          }
        };
        const uint32_t copies = PAIR ? 2u : 1u;
        if (SHARED) {
          for (int kb = 0; kb < nkb; ++kb) {
            if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, status)) { ok = false; break; }
            const uint32_t fb = PAIR ? map_to_cta(full_bar(stage), 0) : full_bar(stage);
            if (rank == 0) mbar_expect_tx(full_bar(stage), copies * (uint32_t)(nA * A_BYTES + nB * F::BB));
            for (int i = 0; i < nA; ++i) load_a(sA(stage, i), &p->mapA[i], kb * BK, ((a_ring >> i) & 1) ? ti.z : 0, fb);
            for (int i = 0; i < nB; ++i) load_b(sB(stage, i), &p->mapB[i], kb * BK, ((b_ring >> i) & 1) ? ti.z : 0, fb);
            if (++stage == NST) { stage = 0; phase ^= 1u; }
          }
        } else {
          for (int pr = 0; pr < n_pairs && ok; ++pr) {
            const int za = ((a_ring >> pr) & 1) ? ti.z : 0;
            const int zb = ((b_ring >> pr) & 1) ? ti.z : 0;
            for (int kb = 0; kb < nkb; ++kb) {
              if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, status)) { ok = false; break; }
              const uint32_t fb = PAIR ? map_to_cta(full_bar(stage), 0) : full_bar(stage);
              if (rank == 0) mbar_expect_tx(full_bar(stage), copies * (uint32_t)F::STAGE);
              load_a(sA(stage, 0), &p->mapA[pr], kb * BK, za, fb);
              load_b(sB(stage, 0), &p->mapB[pr], kb * BK, zb, fb);
              if (++stage == NST) { stage = 0; phase ^= 1u; }
            }
          }
        }
        if (!ok) break;
      }
      outlast_copies(abort_flag);
    }
  } else if (warp == 1) {
    // ======================= MMA issuer =======================
    // (paired form: the leader issues for both CTAs; the peer's warp only owns the tensor-memory allocation)
    if (lane == 0 && rank == 0) {
      int stage = 0; uint32_t phase = 0;
      int acc = 0; uint32_t acc_phase = 0;
      uint32_t fold_seq = 0;                      // folded form: chunks handed over so far (buffer = seq & 1)
      // a commit arrives on this CTA's barrier and, in the paired form, on the peer's as well
      auto commit = [&](uint32_t bar) {
        if (PAIR) { umma_commit_pair(bar); umma_commit_pair(map_to_cta(bar, 1)); } else { umma_commit(bar); }
      };
      for (int wi = walk_begin; wi < walk_end && !*abort_flag; wi += walk_step) {
        const TileInfo ti = tile_at(wi);
        if (!ti.active) continue;
        const DevProblem* p = ti.p;
        const int nkb = (p->K + BK - 1) / BK;
        const int combos = p->combos, fold_kb = p->fold_kb;      // (copies: see the producer)
        const uint32_t idesc = make_idesc(p->a_mn, p->b_mn, TM);
        // K-major: advance 32 bytes per 16-element k step inside the swizzle row;
        // MN-major: 16 k rows = two 8-row groups of 1024 bytes.
        const uint32_t a_lbo = p->a_mn ? BK * 128 : 0, a_adv = p->a_mn ? 2048 : 32;
        const uint32_t b_lbo = p->b_mn ? BK * 128 : 0, b_adv = p->b_mn ? 2048 : 32;
        if (FOLD) {
          // chunks of fold_kb k-blocks, each accumulated from zero, alternately in the two buffers, and
          // handed to the epilogue warps, which add it to the running sum in their registers
          bool ok = true;
          for (int kb0 = 0; kb0 < nkb && ok; kb0 += fold_kb) {
            const int buf = (int)(fold_seq & 1u);
            if (!mbar_wait<PAIR>(tempty_bar(buf), ((fold_seq >> 1) & 1u) ^ 1u, abort_flag, status)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d_chunk = tmem_base + (uint32_t)buf * BN;
            uint32_t accumulate = 0;
            const int kb1 = min(nkb, kb0 + fold_kb);
            for (int kb = kb0; kb < kb1; ++kb) {
              if (!mbar_wait(full_bar(stage), phase, abort_flag, status)) { ok = false; break; }
              tc_fence_after();
              const uint64_t adesc = make_smem_desc(sA(stage, 0), a_lbo, 1024);
              const uint64_t bdesc = make_smem_desc(sB(stage, 0), b_lbo, 1024);
#pragma unroll
              for (int k = 0; k < BK / UMMA_K; ++k) {
                if (PAIR)
                  umma_bf16_pair(d_chunk, adesc + (uint64_t)((k * a_adv) >> 4), bdesc + (uint64_t)((k * b_adv) >> 4),
                                 idesc, accumulate);
                else
                  umma_bf16(d_chunk, adesc + (uint64_t)((k * a_adv) >> 4), bdesc + (uint64_t)((k * b_adv) >> 4),
                            idesc, accumulate);
                accumulate = 1;
              }
              commit(empty_bar(stage));
              if (++stage == NST) { stage = 0; phase ^= 1u; }
            }
            if (!ok) break;
            commit(tfull_bar(buf));
            ++fold_seq;
          }
          if (!ok) break;
          continue;
        }
        if (!mbar_wait<PAIR>(tempty_bar(acc), acc_phase ^ 1u, abort_flag, status)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)acc * BN;
        uint32_t accumulate = 0;
        bool ok = true;
        const int n_steps = SHARED ? nkb : p->n_pairs * nkb;
        const int n_combo = SHARED ? (combos >> 8) : 1;
        for (int it = 0; it < n_steps; ++it) {
          if (!mbar_wait(full_bar(stage), phase, abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          for (int c = 0; c < n_combo; ++c) {
            const int ai = SHARED ? ((combos >> (2 * c)) & 1) : 0;
            const int bi = SHARED ? ((combos >> (2 * c + 1)) & 1) : 0;
            const uint64_t adesc = make_smem_desc(sA(stage, ai), a_lbo, 1024);
            const uint64_t bdesc = make_smem_desc(sB(stage, bi), b_lbo, 1024);
#pragma unroll
            for (int k = 0; k < BK / UMMA_K; ++k) {
              if (PAIR)
                umma_bf16_pair(d_tmem, adesc + (uint64_t)((k * a_adv) >> 4), bdesc + (uint64_t)((k * b_adv) >> 4),
                               idesc, accumulate);
              else
                umma_bf16(d_tmem, adesc + (uint64_t)((k * a_adv) >> 4), bdesc + (uint64_t)((k * b_adv) >> 4),
                          idesc, accumulate);
              accumulate = 1;
            }
          }
          commit(empty_bar(stage));               // frees the stage once these MMAs have read it
          if (++stage == NST) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        commit(tfull_bar(acc));                   // accumulator complete
        acc ^= 1;
        if (acc == 0) acc_phase ^= 1u;
      }
    }
  } else {
    // ======================= epilogue warps =======================
    // A warp may read only its own quadrant of tensor memory, where lane = accumulator row: a
    // 32 x 32 block arrives with one row per lane.  It is turned through a swizzled shared-memory
    // block so that global memory is accessed along rows: 8 lanes cover 128 contiguous bytes of one
    // row, a warp instruction four whole rows.  The values a read-modify-write epilogue needs are
    // prefetched into L2 while the main loop of the tile is still running; those of a warp's first block are loaded
    // before it waits for the accumulator, those of the next one in place of the ones just used.  (Four warps, one
    // block's loads behind the other's stores and IEEE division and square root: 34 us for a tile of the rotated Adam
    // at d = 1024, three times its main loop.)  A symmetric product (the factor EMAs) computes and writes only
    // the 32 x 32 blocks on and above the diagonal (see TcProblem::symmetric).
    const int quad = warp & 3;                    // tensor-memory lane quadrant this warp may read
    const int half = (warp - 2) >> 2;             // and its half of the result columns
    float* const block = epi_tiles + (warp - 2) * (32 * 32);
    // 16-byte piece c of row r of the warp's block: a thread's own row and a row by eight lanes are both conflict-free
    auto piece = [&](int r, int c) { return block + r * 32 + ((c ^ (r & 7)) * 4); };
    const int sub_r = lane >> 3, sub_c = (lane & 7) * 4;
    int acc = 0; uint32_t acc_phase = 0;
    uint32_t fold_seq = 0;
    for (int wi = walk_begin; wi < walk_end && !*abort_flag; wi += walk_step) {
      const TileInfo ti = tile_at(wi);
      if (!ti.active) continue;
      const DevProblem* p = ti.p;
      float alpha = p->dyn_scalars ? dyn_alpha : p->alpha;
      const float beta = p->dyn_scalars ? dyn_beta : p->beta;
      const float eps = p->eps;
      const int epi = p->epilogue;
      // clipping factor of the call whose gradient this accumulator was built from
      float gclip = 1.0f;
      if (p->clip) {
        const int tl = tau < 0 ? p->tau_max : tau;
        gclip = p->clip[(int)((calls - 1 - tl) % p->clip_slots)];
        if (p->clip_mode == 2) alpha *= gclip * gclip;
      }
      const int row_base = ti.m0 + (int)rank * BM + quad * 32;
      const int col_base = ti.n0 + half * (BN / 2);
      const bool quad_ok = row_base < p->Md;      // uniform across the warp
      const bool reads_d = (epi == EPI_AXPBY_F32 && beta != 0.0f) || epi == EPI_ROTATED_ADAM;
      if (!FOLD && reads_d && row_base + lane < p->Md) {
        const long long at = (long long)(row_base + lane) * p->ldd + col_base;
#pragma unroll
        for (int q = 0; q < BN / 64; ++q)
          if (col_base + 32 * q < p->Nd) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p->D + at + 32 * q));
            if (epi == EPI_ROTATED_ADAM) asm volatile("prefetch.global.L2 [%0];" ::"l"(p->D2 + at + 32 * q));
          }
      }
      if constexpr (FOLD) {
        // ---- folded form: this warp owns 32 rows (its lane quadrant) x 128 columns (its half) ----
        float* const fbuf = epi_tiles + (warp - 2) * (2 * FOLD_BLOCK);
        const int nkb = (p->K + BK - 1) / BK, fold_kb = p->fold_kb;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(half * 128);
        // which of the four 32-column blocks are written at all (uniform across the warp)
        uint32_t need = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int col0 = col_base + 32 * b;
          if (col0 < p->Nd && quad_ok && !(p->symmetric && row_base >= col0 + 32)) need |= 1u << b;
        }
        // The old values of D are copied to shared memory asynchronously, two of the four blocks while the chunks
        // of the tile accumulate and the others as soon as a buffer is free: 16-byte pieces, piece c of row r at
        // c ^ (r % 8), so that both the copies (a row's 128 bytes by eight lanes) and a thread's walk along its own
        // row are free of bank conflicts.  (Loaded into registers beside the 128 running sums they were spilled, or
        // exposed the latency of memory once per half block.)
        auto piece2 = [&](int buf, int r, int c) { return fbuf + buf * FOLD_BLOCK + r * 32 + ((c ^ (r & 7)) * 4); };
        const int cp_r = sub_r, cp_c = lane & 7;
        float* const d0 = p->D + (long long)(row_base + cp_r) * p->ldd + col_base + cp_c * 4;
        const long long step = 4 * p->ldd;
        auto rows_of = [&](int b) {                // groups of four rows of block b that exist in this lane's columns
          if (!((need >> b) & 1u) || col_base + 32 * b + cp_c * 4 >= p->Nd) return 0;
          const int n_it = (p->Md - row_base - cp_r + 3) >> 2;
          return n_it > 8 ? 8 : n_it;
        };
        auto fetch_old = [&](int b) {
          const int n_it = beta != 0.0f ? rows_of(b) : 0;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i < n_it)
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(piece2(b & 1, 4 * i + cp_r, cp_c))),
                           "l"(d0 + 32 * b + i * step) : "memory");
          asm volatile("cp.async.commit_group;" ::: "memory");
        };
        fetch_old(0);
        fetch_old(1);
        // The running sum of this thread: its row, its warp's 128 columns.  The first chunk is loaded
        // straight into these registers; every later one is added with packed fp32 adds, one 32-column
        // block at a time (the other warp of the quadrant covers the load latency).
        uint32_t sum[4][32];
        bool ok = true;
        for (int kb0 = 0; kb0 < nkb; kb0 += fold_kb) {
          const int buf = (int)(fold_seq & 1u);
          if (!mbar_wait(tfull_bar(buf), (fold_seq >> 1) & 1u, abort_flag, status)) { ok = false; break; }
          tc_fence_after();
          const uint32_t src = lane_base + (uint32_t)(buf * BN);
          if (kb0 == 0) {
#pragma unroll
            for (int b = 0; b < 4; ++b)
              if ((need >> b) & 1u) tmem_ld32_issue(src + 32 * b, sum[b]);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              if (!((need >> b) & 1u)) continue;
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t t[16];
                tmem_ld16_issue(src + 32 * b + 16 * h, t);
                tmem_wait_ld();
#pragma unroll
                for (int j = 0; j < 16; j += 2) {
                  const float2 r = __fadd2_rn(make_float2(__uint_as_float(sum[b][16 * h + j]), __uint_as_float(sum[b][16 * h + j + 1])),
                                              make_float2(__uint_as_float(t[j]), __uint_as_float(t[j + 1])));
                  sum[b][16 * h + j] = __float_as_uint(r.x); sum[b][16 * h + j + 1] = __float_as_uint(r.y);
                }
              }
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (PAIR) mbar_arrive_cluster(map_to_cta(tempty_bar(buf), 0)); else mbar_arrive(tempty_bar(buf));
          }
          ++fold_seq;
        }
        if (!ok) break;
        // ---- factor EMA D <- alpha sum + beta D on the blocks that touch the upper triangle ----
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          asm volatile("cp.async.wait_group 1;" ::: "memory");
          __syncwarp();
          if ((need >> b) & 1u) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              float4* q = reinterpret_cast<float4*>(piece2(b & 1, lane, c));
              float4 r = make_float4(alpha * __uint_as_float(sum[b][4 * c]), alpha * __uint_as_float(sum[b][4 * c + 1]),
                                     alpha * __uint_as_float(sum[b][4 * c + 2]), alpha * __uint_as_float(sum[b][4 * c + 3]));
              if (beta != 0.0f) {
                const float4 o = *q;
                r.x = fmaf(beta, o.x, r.x); r.y = fmaf(beta, o.y, r.y); r.z = fmaf(beta, o.z, r.z); r.w = fmaf(beta, o.w, r.w);
              }
              *q = r;
            }
          }
          __syncwarp();
          const int n_it = rows_of(b);
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i < n_it) *reinterpret_cast<float4*>(d0 + 32 * b + i * step) = *reinterpret_cast<const float4*>(piece2(b & 1, 4 * i + cp_r, cp_c));
          __syncwarp();
          if (b < 2) fetch_old(b + 2); else asm volatile("cp.async.commit_group;" ::: "memory");
        }
        continue;
      }
      // The blocks of 32 columns that this warp writes (uniform across it), and the groups of four rows of block b that
      // exist in this lane's columns (columns come in multiples of 8: a group of four is all in or all out).
      auto writes = [&](int b) {
        const int col0 = col_base + 32 * b;
        return quad_ok && b < BN / 64 && col0 < p->Nd && !(p->symmetric && row_base >= col0 + 32);
      };
      auto rows_of = [&](int b) {
        if (!writes(b) || col_base + 32 * b + sub_c >= p->Nd) return 0;
        const int n_it = (p->Md - row_base - sub_r + 3) >> 2;
        return n_it > 8 ? 8 : n_it;
      };
      const long long at_d = (long long)(row_base + sub_r) * p->ldd + col_base + sub_c, step_d = 4 * p->ldd;
      const long long at_h = (long long)(row_base + sub_r) * p->ldh + col_base + sub_c, step_h = 4 * p->ldh;
      // block b of the accumulator, turned: entry `it` of this lane is row 4 it + sub_r, columns sub_c .. sub_c + 3
      auto turn = [&](int b) {
        float v[32];
        tmem_ld32(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * BN + half * (BN / 2) + 32 * b), v);
#pragma unroll
        for (int c = 0; c < 8; ++c) *reinterpret_cast<float4*>(piece(lane, c)) = make_float4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
        __syncwarp();
      };
      auto turned = [&](int it) { return *reinterpret_cast<const float4*>(piece(4 * it + sub_r, lane & 7)); };
      if (SHARED && epi == EPI_ROTATED_ADAM) {
        const float b1 = p->beta1, ob1 = 1.0f - p->beta1;
        float* const pv = p->D + at_d;                 // V~
        float* const pm = p->D2 + at_d;                // M~
        float4 mm[8], ss[8];
        int n_it = rows_of(0);
#pragma unroll
        for (int it = 0; it < 8; ++it)
          if (it < n_it) {
            mm[it] = *reinterpret_cast<const float4*>(pm + it * step_d);
            ss[it] = *reinterpret_cast<const float4*>(pv + it * step_d);
          }
        if (!mbar_wait(tfull_bar(acc), acc_phase, abort_flag, status)) break;
        tc_fence_after();
#pragma unroll 1
        for (int b = 0; b < BN / 64; ++b) {
          if (!writes(b)) break;
          turn(b);
          const int n_next = rows_of(b + 1);
          float *const dv = pv + 32 * b, *const dm = pm + 32 * b;
          __nv_bfloat16* const xh = p->Dh + at_h + 32 * b;
#pragma unroll
          for (int it = 0; it < 8; ++it) {
            if (it < n_it) {
              const float4 x = turned(it);
              const float4 g = make_float4(gclip * x.x, gclip * x.y, gclip * x.z, gclip * x.w);
              float4 m = mm[it], q = ss[it];
              m.x = b1 * m.x + ob1 * g.x; m.y = b1 * m.y + ob1 * g.y;
              m.z = b1 * m.z + ob1 * g.z; m.w = b1 * m.w + ob1 * g.w;
              q.x = fmaf(beta, q.x, alpha * g.x * g.x); q.y = fmaf(beta, q.y, alpha * g.y * g.y);
              q.z = fmaf(beta, q.z, alpha * g.z * g.z); q.w = fmaf(beta, q.w, alpha * g.w * g.w);
              *reinterpret_cast<float4*>(dm + it * step_d) = m;
              *reinterpret_cast<float4*>(dv + it * step_d) = q;
              uint2 o;
              o.x = pack2_bf16(m.x / sqrtf(q.x + eps), m.y / sqrtf(q.y + eps));
              o.y = pack2_bf16(m.z / sqrtf(q.z + eps), m.w / sqrtf(q.w + eps));
              *reinterpret_cast<uint2*>(xh + it * step_h) = o;
            }
            if (it < n_next) {
              mm[it] = *reinterpret_cast<const float4*>(dm + 32 + it * step_d);
              ss[it] = *reinterpret_cast<const float4*>(dv + 32 + it * step_d);
            }
          }
          n_it = n_next;
          __syncwarp();                           // the block's buffer is rewritten by the next one
        }
      } else if (epi == EPI_AXPBY_F32) {
        float* const pd = p->D + at_d;
        float4 old[8];
        const bool rd = beta != 0.0f;
        int n_it = rows_of(0);
#pragma unroll
        for (int it = 0; it < 8; ++it)
          if (rd && it < n_it) old[it] = *reinterpret_cast<const float4*>(pd + it * step_d);
        if (!mbar_wait(tfull_bar(acc), acc_phase, abort_flag, status)) break;
        tc_fence_after();
#pragma unroll 1
        for (int b = 0; b < BN / 64; ++b) {
          const int n_next = rows_of(b + 1);
          float* const d = pd + 32 * b;
          if (writes(b)) turn(b);
#pragma unroll
          for (int it = 0; it < 8; ++it) {
            if (it < n_it) {
              const float4 x = turned(it);
              float4 o = make_float4(alpha * x.x, alpha * x.y, alpha * x.z, alpha * x.w);
              if (rd) {
                o.x = fmaf(beta, old[it].x, o.x); o.y = fmaf(beta, old[it].y, o.y);
                o.z = fmaf(beta, old[it].z, o.z); o.w = fmaf(beta, old[it].w, o.w);
              }
              *reinterpret_cast<float4*>(d + it * step_d) = o;
            }
            if (rd && it < n_next) old[it] = *reinterpret_cast<const float4*>(d + 32 + it * step_d);
          }
          n_it = n_next;
          __syncwarp();
        }
      } else {  // EPI_SPLIT_BF16
        if (!mbar_wait(tfull_bar(acc), acc_phase, abort_flag, status)) break;
        tc_fence_after();
#pragma unroll 1
        for (int b = 0; b < BN / 64; ++b) {
          if (!writes(b)) break;
          turn(b);
          const int n_it = rows_of(b);
          __nv_bfloat16* const dh = p->Dh + at_h + 32 * b;
          __nv_bfloat16* const dl = p->Dl ? p->Dl + at_h + 32 * b : nullptr;
#pragma unroll
          for (int it = 0; it < 8; ++it)
            if (it < n_it) {
              const float4 g = turned(it);
              const float h0 = __bfloat162float(__float2bfloat16_rn(g.x)), h1 = __bfloat162float(__float2bfloat16_rn(g.y));
              const float h2 = __bfloat162float(__float2bfloat16_rn(g.z)), h3 = __bfloat162float(__float2bfloat16_rn(g.w));
              uint2 o;
              o.x = pack2_bf16(h0, h1); o.y = pack2_bf16(h2, h3);
              *reinterpret_cast<uint2*>(dh + it * step_h) = o;
              if (dl) {
                uint2 l;
                l.x = pack2_bf16(g.x - h0, g.y - h1); l.y = pack2_bf16(g.z - h2, g.w - h3);
                *reinterpret_cast<uint2*>(dl + it * step_h) = l;
              }
            }
          __syncwarp();
        }
      }
      // all tcgen05.ld of this warp have completed (wait::ld): hand the accumulator back
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (PAIR) mbar_arrive_cluster(map_to_cta(tempty_bar(acc), 0)); else mbar_arrive(tempty_bar(acc));
      }
      acc ^= 1;
      if (acc == 0) acc_phase ^= 1u;
    }
  }

  // teardown: every role has left its loop (all waits are bounded)
  // (paired form: neither CTA frees its tensor memory or exits while the other may still signal it)
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_barrier();
  if (warp == 1) {
    tc_fence_after();
    if (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// One warp waits, with the kernel's own bounded wait, on an mbarrier that nothing ever arrives on: the
// wait must give up after limit_ns, leave BR_ERR_TIMEOUT in the status word and return.
__global__ void __launch_bounds__(32) k_wait_probe(uint64_t limit_ns, int* status) {
  __shared__ alignas(8) uint64_t bar;
  __shared__ int abort_word;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (threadIdx.x == 0) mbar_wait(smem_u32(&bar), 0u, &abort_word, status, limit_ns);
}

// ---------------------------------------------------------------------------------------------
// Host side: tensor-map encoding and plans
// ---------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// rows = extent of the M / N index, K = contraction extent.
bool encode_operand(CUtensorMap* map, const TcOperand& op, int64_t rows, int64_t K, int box_rows,
                    std::string* err) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) { *err = "cuTensorMapEncodeTiled is not available from the driver"; return false; }
  const int64_t inner = op.mn_major ? rows : K;
  const int64_t outer = op.mn_major ? K : rows;
  const int slots = op.ring_slots > 0 ? op.ring_slots : 1;
  const uint64_t slot_stride = op.ring_slots > 0 ? (uint64_t)op.slot_stride_bytes
                                                 : (uint64_t)op.ld * 2ull * (uint64_t)outer;
  if ((reinterpret_cast<uintptr_t>(op.ptr) & 15) || (op.ld % 8) || (slot_stride % 16)) {
    *err = "tensor-core operand is not 16-byte aligned (pointer, leading dimension or slot stride)";
    return false;
  }
  cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)outer, (cuuint64_t)slots};
  cuuint64_t strides[2] = {(cuuint64_t)op.ld * 2ull, (cuuint64_t)slot_stride};
  cuuint32_t box[3] = {64u, (cuuint32_t)(op.mn_major ? BK : box_rows), 1u};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(op.ptr), dims, strides, box,
                   estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    *err = "cuTensorMapEncodeTiled failed with code " + std::to_string((int)r);
    return false;
  }
  return true;
}

typedef void (*TcKernel)(const DevProblem*, int, int, int, const int*, long long, int, float, float, int*);
TcKernel kernel_of(bool shared, bool pair, bool fold = false) {
  if (fold) return pair ? k_tc_gemm<false, true, true> : k_tc_gemm<false, false, true>;
  if (pair) return shared ? k_tc_gemm<true, true> : k_tc_gemm<false, true>;
  return shared ? k_tc_gemm<true, false> : k_tc_gemm<false, false>;
}

// Number of CTA pairs (clusters of two) of the paired form that fit on the current device at once;
// 0 when that form is switched off (environment BR_TC_PAIR=0) or cannot be launched.
int pair_capacity(bool shared) {
  static int cap[2] = {-1, -1};
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  int& c = cap[shared ? 1 : 0];
  if (c >= 0) return c;
  c = 0;
  const char* env = std::getenv("BR_TC_PAIR");
  if (env && env[0] == '0') return c;
  TcKernel kernel = kernel_of(shared, true);
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES) != cudaSuccess) {
    cudaGetLastError();
    return c;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(2u * (unsigned)(sms / 2));
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.attrs = attr; cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return c; }
  c = clusters < sms / 2 ? clusters : sms / 2;
  return c;
}

// Longest tiles first, each to the unit with the least work so far.  The round-robin walk of the plan's order
// leaves units idle at the end when a launch mixes contraction lengths (the factor products of a decoder layer with
// its embedding: 55 tiles of 500 k-blocks behind 1739 of 40 to 108) or has few tiles per unit.  Tiles of equal
// length keep their order, so that neighbours in the walk still run at the same time and share operands in L2.
// A tile costs its k-blocks plus `fixed` (the part of its epilogue that the next tile's main loop does not
// cover, in k-blocks).  Layout: units + 1 offsets, then the tiles, then their problems.
std::vector<int> make_schedule(const std::vector<DevProblem>& probs, int total, int units, int fixed) {
  struct Tile { int cost, index, problem; };
  std::vector<Tile> tiles;
  tiles.reserve((size_t)total);
  for (size_t p = 0; p < probs.size(); ++p)
    for (int i = 0; i < probs[p].tile_count; ++i)
      tiles.push_back({probs[p].n_pairs * ((probs[p].K + BK - 1) / BK) + fixed, probs[p].tile_begin + i, (int)p});
  std::stable_sort(tiles.begin(), tiles.end(), [](const Tile& a, const Tile& b) { return a.cost > b.cost; });
  typedef std::pair<long long, int> Load;                     // (work so far, unit)
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> heap;
  for (int u = 0; u < units; ++u) heap.push({0, u});
  std::vector<std::vector<Tile>> list((size_t)units);
  for (const Tile& t : tiles) {
    Load l = heap.top();
    heap.pop();
    list[(size_t)l.second].push_back(t);
    l.first += t.cost;
    heap.push(l);
  }
  std::vector<int> out;
  out.reserve((size_t)(units + 1 + 2 * total));
  int at = 0;
  for (int u = 0; u < units; ++u) { out.push_back(at); at += (int)list[(size_t)u].size(); }
  out.push_back(at);
  for (const auto& l : list) for (const Tile& t : l) out.push_back(t.index);
  for (const auto& l : list) for (const Tile& t : l) out.push_back(t.problem);
  return out;
}

}  // namespace

struct TcPlan {
  bool fold = false;            // launches the folded form (chunked accumulation, running sum in registers)
  bool shared = false;          // launches the shared-operand form of the kernel
  bool pair = false;            // launches the paired form (clusters of two CTAs, 256-row tiles)
  int max_pairs = 0;            // CTA pairs that can be resident at once
  std::vector<int> tile_begin;  // per problem, plus the total at the end
  std::vector<double> prob_flops;
  DevProblem* d_probs = nullptr;
  int* d_schedule = nullptr;    // tile lists of the whole plan's units (see make_schedule), or null
  int units = 0;                // CTA pairs (or CTAs) of a launch of the whole plan
  int n = 0;
  int total_tiles = 0;
  double flops = 0.0;
  int sm_count = 148;
  std::string err;
};

int tc_supported(int device) {
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return 0;
  return prop.major == 10 && get_encode_fn() != nullptr;
}

void* tensor_map_encoder() { return reinterpret_cast<void*>(get_encode_fn()); }

TcPlan* tc_plan_create(const TcProblem* problems, int n, int device, cudaStream_t s, const char** err) {
  static thread_local std::string last;
  auto fail = [&](const std::string& m) -> TcPlan* { last = m; if (err) *err = last.c_str(); return nullptr; };
  if (n <= 0) return fail("empty plan");
  // The shared-operand form pays off when some problem sums several pairs, and applies when every
  // problem combines at most two distinct A and two distinct B operands.
  auto same_operand = [](const TcOperand& x, const TcOperand& y) {
    return x.ptr == y.ptr && x.ld == y.ld && x.mn_major == y.mn_major && x.ring_slots == y.ring_slots &&
           x.slot_stride_bytes == y.slot_stride_bytes;
  };
  bool shared = false, eligible = true;
  for (int i = 0; i < n; ++i) {
    const TcProblem& q = problems[i];
    if (q.n_pairs < 1 || q.n_pairs > MAX_PAIRS) return fail("tensor-core problem: 1 to 3 operand pairs");
    if (q.n_pairs > 1) shared = true;
    int nA = 0, nB = 0;
    for (int p = 0; p < q.n_pairs; ++p) {
      bool newa = true, newb = true;
      for (int u = 0; u < p; ++u) {
        if (same_operand(q.A[u], q.A[p])) newa = false;
        if (same_operand(q.B[u], q.B[p])) newb = false;
      }
      nA += newa; nB += newb;
    }
    if (nA > 2 || nB > 2) eligible = false;
  }
  shared = shared && eligible;
  // the folded form: every problem asks for it, and none sums several operand pairs
  bool fold = !shared;
  for (int i = 0; i < n; ++i) fold = fold && problems[i].fold_kb > 0 && problems[i].n_pairs == 1;
  if (const char* env = std::getenv("BR_TC_FOLD")) { if (env[0] == '0') fold = false; }      // tuning aid
  int fold_override = 0;
  if (const char* env = std::getenv("BR_TC_FOLD_KB")) { const int v = std::atoi(env); if (v >= 1 && v <= 1024) fold_override = v; }
  const int pairs = pair_capacity(shared);
  const bool pair = pairs > 0;
  const int TM = pair ? 2 * BM : BM;            // rows of a tile
  const int b_box = pair ? BN / 2 : BN;         // rows of B one CTA stages per k-block
  double panel_bytes = kL2PanelBytes;
  if (const char* env = std::getenv("BR_TC_L2_PANEL_MB")) {        // tuning aid
    const double v = std::atof(env);
    if (v >= 1.0 && v <= 512.0) panel_bytes = v * 1e6;
  }
  std::vector<DevProblem> host(n);
  std::vector<int> tile_starts;
  std::vector<double> prob_flops;
  int tile_begin = 0;
  double flops = 0.0;
  for (int i = 0; i < n; ++i) {
    const TcProblem& q = problems[i];
    DevProblem& d = host[i];
    std::memset(&d, 0, sizeof d);
    if (q.n_pairs < 1 || q.n_pairs > MAX_PAIRS || q.Md < 1 || q.Nd < 1 || q.K < 1 ||
        (q.Md % 8) || (q.Nd % 8) || (q.K % 8) || q.Md > (1ll << 30) || q.Nd > (1ll << 30) || q.K > (1ll << 30))
      return fail("tensor-core problem: dimensions must be positive multiples of 8");
    std::string e;
    for (int p = 0; p < q.n_pairs; ++p)
      if (q.A[p].mn_major != q.A[0].mn_major || q.B[p].mn_major != q.B[0].mn_major)
        return fail("tensor-core problem: all pairs must share operand majors");
    if (shared) {
      // distinct operands and the list of products
      int ua[MAX_PAIRS], ub[MAX_PAIRS], nA = 0, nB = 0, combos = 0;
      for (int p = 0; p < q.n_pairs; ++p) {
        int ia = -1, ib = -1;
        for (int u = 0; u < nA; ++u) if (same_operand(q.A[ua[u]], q.A[p])) ia = u;
        for (int u = 0; u < nB; ++u) if (same_operand(q.B[ub[u]], q.B[p])) ib = u;
        if (ia < 0) { ia = nA; ua[nA++] = p; }
        if (ib < 0) { ib = nB; ub[nB++] = p; }
        combos |= (ia | (ib << 1)) << (2 * p);
      }
      for (int u = 0; u < nA; ++u) {
        if (!encode_operand(&d.mapA[u], q.A[ua[u]], q.Md, q.K, BM, &e)) return fail(e);
        if (q.A[ua[u]].ring_slots > 0) { d.a_ring_mask |= 1 << u; d.ring_slots = q.A[ua[u]].ring_slots; }
      }
      for (int u = 0; u < nB; ++u) {
        if (!encode_operand(&d.mapB[u], q.B[ub[u]], q.Nd, q.K, b_box, &e)) return fail(e);
        if (q.B[ub[u]].ring_slots > 0) { d.b_ring_mask |= 1 << u; d.ring_slots = q.B[ub[u]].ring_slots; }
      }
      d.nA = nA; d.nB = nB; d.combos = combos | (q.n_pairs << 8);
    } else {
      for (int p = 0; p < q.n_pairs; ++p) {
        if (!encode_operand(&d.mapA[p], q.A[p], q.Md, q.K, BM, &e)) return fail(e);
        if (!encode_operand(&d.mapB[p], q.B[p], q.Nd, q.K, b_box, &e)) return fail(e);
        if (q.A[p].ring_slots > 0) { d.a_ring_mask |= 1 << p; d.ring_slots = q.A[p].ring_slots; }
        if (q.B[p].ring_slots > 0) { d.b_ring_mask |= 1 << p; d.ring_slots = q.B[p].ring_slots; }
      }
    }
    d.Md = (int32_t)q.Md; d.Nd = (int32_t)q.Nd; d.K = (int32_t)q.K; d.n_pairs = q.n_pairs;
    d.a_mn = q.A[0].mn_major; d.b_mn = q.B[0].mn_major; d.epilogue = q.epilogue;
    d.tiles_m = (int32_t)((q.Md + TM - 1) / TM);
    d.tiles_n = (int32_t)((q.Nd + BN - 1) / BN);
    d.tile_begin = tile_begin;
    d.tile_count = d.tiles_m * d.tiles_n;
    // A symmetric product on square tiles lists only the tiles of the upper triangle, so that no CTA pair is dealt
    // tiles it then skips.  (The unpaired form's tiles are 128 x 256: it lists and skips them.)
    d.tri = (q.symmetric && TM == BN && d.tiles_m == d.tiles_n) ? 1 : 0;
    if (d.tri) d.tile_count = d.tiles_m * (d.tiles_m + 1) / 2;
    {
      // Estimated DRAM reads of the two walks: the resident panel's operand once, the other once per
      // group.  Group = as many blocks as keep the panel within its share of L2.
      int nA = 0, nB = 0;
      for (int p = 0; p < q.n_pairs; ++p) {
        bool newa = true, newb = true;
        for (int u = 0; u < p; ++u) {
          if (same_operand(q.A[u], q.A[p])) newa = false;
          if (same_operand(q.B[u], q.B[p])) newb = false;
        }
        nA += newa; nB += newb;
      }
      const double stripeA = (double)TM * (double)q.K * 2.0 * nA, stripeB = (double)BN * (double)q.K * 2.0 * nB;
      const double totalA = stripeA * d.tiles_m, totalB = stripeB * d.tiles_n;
      auto clampi = [](double v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : (int)v); };
      const int gM = clampi(panel_bytes / stripeA, 1, d.tiles_m), gN = clampi(panel_bytes / stripeB, 1, d.tiles_n);
      const double trafficM = totalA + totalB * ((d.tiles_m + gM - 1) / gM);
      const double trafficN = totalB + totalA * ((d.tiles_n + gN - 1) / gN);
      d.raster_n = trafficN < trafficM ? 1 : 0;
      d.group = d.raster_n ? gN : gM;
    }
    tile_starts.push_back(tile_begin);
    tile_begin += d.tile_count;
    d.tau_max = q.tau_max;
    d.dyn_scalars = q.dyn_scalars;
    d.alpha = q.alpha; d.beta = q.beta; d.eps = q.eps; d.beta1 = q.beta1;
    d.symmetric = q.symmetric ? 1 : 0;
    d.clip = q.clip_mode ? q.clip : nullptr; d.clip_slots = q.clip_slots; d.clip_mode = q.clip_mode;
    d.fold_kb = fold ? (fold_override ? fold_override : q.fold_kb) : 0;
    if (d.clip && (q.clip_slots < 1 || (q.clip_mode == 1 && q.epilogue != EPI_ROTATED_ADAM) ||
                   (q.clip_mode == 2 && q.epilogue != EPI_AXPBY_F32)))
      return fail("tensor-core problem: clipping applies to the rotated-Adam and factor epilogues");
    if (q.symmetric && (q.Md != q.Nd || q.epilogue != EPI_AXPBY_F32))
      return fail("tensor-core problem: a symmetric product needs a square fp32 result");
    d.D = q.D; d.ldd = q.ldd; d.Dh = q.Dh; d.Dl = q.Dl; d.ldh = q.ldh; d.D2 = q.D2;
    const bool need_D = q.epilogue != EPI_SPLIT_BF16;
    const bool need_H = q.epilogue == EPI_SPLIT_BF16 || q.epilogue == EPI_ROTATED_ADAM;
    if (q.epilogue == EPI_ROTATED_ADAM && (!shared || !q.D2 || (reinterpret_cast<uintptr_t>(q.D2) & 15)))
      return fail("tensor-core problem: rotated Adam without operand pairs, or its second in/out pointer missing or misaligned");
    if ((need_D && (!q.D || (q.ldd % 4) || (reinterpret_cast<uintptr_t>(q.D) & 15))) ||
        (need_H && (!q.Dh || (q.ldh % 8) || (reinterpret_cast<uintptr_t>(q.Dh) & 15))) ||
        (q.Dl && (reinterpret_cast<uintptr_t>(q.Dl) & 15)))
      return fail("tensor-core problem: output pointer missing or misaligned");
    const double flops_before = flops;
    if (q.symmetric) {
      // executed work: the tiles that touch the upper triangle
      int64_t computed = 0;
      for (int64_t rb = 0; rb < d.tiles_m; ++rb)
        for (int64_t cb = 0; cb < d.tiles_n; ++cb)
          if (rb * TM < cb * BN + BN) ++computed;
      flops += 2.0 * (double)computed * TM * BN * (double)q.K * q.n_pairs;
    } else {
      flops += 2.0 * (double)q.Md * (double)q.Nd * (double)q.K * q.n_pairs;
    }
    prob_flops.push_back(flops - flops_before);
  }
  TcPlan* plan = new TcPlan();
  plan->fold = fold;
  plan->shared = shared;
  plan->pair = pair;
  plan->max_pairs = pairs;
  tile_starts.push_back(tile_begin);
  plan->tile_begin = tile_starts;
  plan->prob_flops = prob_flops;
  plan->n = n;
  plan->total_tiles = tile_begin;
  plan->flops = flops;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, device) == cudaSuccess) plan->sm_count = prop.multiProcessorCount;
  const int cap = pair ? pairs : plan->sm_count;
  plan->units = tile_begin < cap ? tile_begin : cap;
  const std::vector<int> schedule = make_schedule(host, tile_begin, plan->units, fold ? kFoldTileCost : kTileCost);
  cudaError_t ce = cudaMalloc(&plan->d_probs, sizeof(DevProblem) * n + sizeof(int) * schedule.size());
  if (ce == cudaSuccess) {
    plan->d_schedule = reinterpret_cast<int*>(plan->d_probs + n);
    ce = cudaMemcpyAsync(plan->d_probs, host.data(), sizeof(DevProblem) * n, cudaMemcpyHostToDevice, s);
  }
  if (ce == cudaSuccess)
    ce = cudaMemcpyAsync(plan->d_schedule, schedule.data(), sizeof(int) * schedule.size(), cudaMemcpyHostToDevice, s);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);   // `host` and `schedule` go out of scope
  if (ce != cudaSuccess) {
    if (plan->d_probs) cudaFree(plan->d_probs);
    delete plan;
    return fail(std::string("plan upload: ") + cudaGetErrorString(ce));
  }
  return plan;
}

void tc_plan_destroy(TcPlan* p) {
  if (!p) return;
  if (p->d_probs) cudaFree(p->d_probs);
  delete p;
}

double tc_plan_flops(const TcPlan* p) { return p ? p->flops : 0.0; }

cudaError_t tc_plan_launch_range(TcPlan* p, int first, int count, long long calls, int tau, float dyn_alpha,
                                 float dyn_beta, int* status_word, cudaStream_t s) {
  if (first < 0 || count < 1 || first + count > p->n) return cudaErrorInvalidValue;
  const int t0 = p->tile_begin[first], t1 = p->tile_begin[first + count];
  const int tiles = t1 - t0;
  TcKernel kernel = kernel_of(p->shared, p->pair, p->fold);
  // per-device attribute: set again when another device is current (cheap, idempotent)
  const int smem_bytes = p->fold ? SMEM_BYTES_FOLD : p->shared ? SMEM_BYTES : SMEM_BYTES_PLAIN;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const bool whole = first == 0 && count == p->n;
  if (p->pair) {
    const int units = whole ? p->units : tiles < p->max_pairs ? tiles : p->max_pairs;
    cfg.gridDim = dim3(2u * (unsigned)units);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
  } else {
    cfg.gridDim = dim3((unsigned)(whole ? p->units : tiles < p->sm_count ? tiles : p->sm_count));
  }
  cfg.blockDim = dim3(NUM_THREADS);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = s;
  return cudaLaunchKernelEx(&cfg, kernel, (const DevProblem*)p->d_probs, p->n, t0, t1,
                            (const int*)(whole ? p->d_schedule : nullptr), calls, tau, dyn_alpha,
                            dyn_beta, status_word);
}

cudaError_t tc_plan_launch(TcPlan* p, long long calls, int tau, float dyn_alpha, float dyn_beta,
                           int* status_word, cudaStream_t s) {
  return tc_plan_launch_range(p, 0, p->n, calls, tau, dyn_alpha, dyn_beta, status_word, s);
}

cudaError_t tc_wait_probe(uint64_t limit_ns, int* status_word, cudaStream_t s) {
  k_wait_probe<<<1, 32, 0, s>>>(limit_ns, status_word);
  return cudaGetLastError();
}

double tc_plan_flops_range(const TcPlan* p, int first, int count) {
  double f = 0.0;
  for (int i = first; i < first + count && i < p->n; ++i) f += p->prob_flops[i];
  return f;
}

}  // namespace br
