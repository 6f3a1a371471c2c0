// Prefill kernel (more than 128 rows, and smaller batches that neither the decode nor the batch kernel takes) of the pruned 4-bit
// linear layer, sm_100a: a dense contraction on
// the fifth-generation tensor cores (tcgen05.mma, accumulators in tensor memory).
//
// Orientation.  The packed weights are four times smaller than the activations, so the weight side
// takes the MMA's M dimension (128 retained weight rows per tile, de-quantised once per tile and
// k-block) and the tokens its N dimension (up to 256 per tile): D[row][token] += W[row][k] x[token][k].
//
// Roles inside a block (one persistent block per SM, tiles taken round-robin):
//   warp 0       TMA producer: boxes [64 k x BN tokens] of activations into a ring of four (128-byte swizzle);
//                one box per k-block, or two where a tile takes both accumulators (512 tokens)
//   warp 1       allocates tensor memory; one lane issues the MMAs of a k-block (4 x K=16 per box) and commits
//                them to the box's and the weight stage's "empty" barriers and, at the end of a tile, to
//                "accumulator full"
//   warps 4..7   epilogue: tcgen05.ld the fp32 accumulators (warp w owns TMEM lanes 32(w-4).., a lane
//                is a tile row and holds 32 tokens of it per pass), bias, rotary embedding on the
//                retained pair (Section 3.2; the pair's two rows are neighbouring lanes and swap
//                values by shuffle), one rounding, stores of 32 consecutive outputs of a token per
//                warp; two accumulator buffers of 256 columns let the epilogue of tile i overlap
//                the MMAs of tile i+1 (tiles of 512 tokens use both and hand them back one by one);
//                the epilogue of a block's last tile is shared with the de-quantiser warps, idle by then
//   warps 8..23  de-quantisers: the twelve of them whose scheduler does not host the MMA warp (warp % 4 != 1), two
//                teams of six warps on alternate stages; a thread converts 32 codes of a weight row per item --
//                nibbles to fp16 by magic number, (q-8) exact, then one fp16 FMA (q-8)*s + fp16(s*(8-z))
//                -- and writes them into the A-operand stage in the
//                canonical K-major 128-byte-swizzled layout; the packed codes of the next k-block
//                are already in registers.  All sixteen share the epilogue of the block's last segment.
// Work split (chosen by the launcher from a cost model): whole tiles round-robin; tiles left over after the whole
// rounds split along K over all blocks (stream-K: parts handed over through slots in the workspace, or added into
// one sum per tile) or, for tiles of two boxes, run as half tiles on twice the blocks; launches with few tiles as
// clusters of two blocks per tile, the second block's sums written into the first one's idle rings.
// Above 128 rows (PAIR instances): clusters of two blocks run tiles of 256 weight rows with cta_group::2 MMAs, one or two boxes
// of 256 tokens per tile; launches with few tiles as clusters of two to four such pairs per tile, a part of the contraction
// each.  Measured: Qwen2.5-7B gate at M = 2048 227 -> 193 us (1.44 PFLOP/s), 4096 x 4096 at M = 256 27 -> 19 us.
// Launched with programmatic stream serialization: what a block does before griddepcontrol.wait (barriers, tensor
// memory, the first weight stages) touches nothing a preceding kernel may still read or write.
// On-device pruning (Section 3.4) is index arithmetic: tile rows are compact output channels mapped to
// stored rows per thread; the input side is the leading k_in channels (the TMA tensor ends at k_in, so
// the tail of the last k-block is zero activations).
// bf16 activations: bf16 weights would carry 2^-9 relative rounding error each, which alone spends the
// 2e-3 error budget; instead the de-quantisers convert the activation tile to fp16 in place (exact in
// fp16's range, saturating beyond) and both operands are fp16.
//
// Every mbarrier wait is bounded; on expiry the block raises a flag, every role leaves its loop, the
// status word of the workspace is set, tensor memory is released and the block returns.
#include <cuda.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "tc.cuh"

namespace uniql {
namespace {

constexpr int MAXBN = 256;          // tokens per tile (MMA N), at most
constexpr int PSTAGES = 4;                   // ring of de-quantised weight stages (one k-block each)
constexpr int BSLOTS = 4;                    // ring of activation boxes (one k-block of MAXBN tokens each)
// block pairs: stages of weights and the k-block's half boxes (each block holds half of the tokens), one or two of them
constexpr int PSTAGES1 = 6, PSTAGES2 = 4;
constexpr int A_BYTES = BMW * BK * 2;        // 16 KB
constexpr int B_BYTES = MAXBN * BK * 2;      // 32 KB
constexpr int RING_BYTES = PSTAGES * A_BYTES + BSLOTS * B_BYTES;
constexpr int RING2_BYTES = PSTAGES2 * (A_BYTES + B_BYTES);
static_assert(PSTAGES1 * (A_BYTES + B_BYTES / 2) == RING2_BYTES, "the pair instances use the same shared memory");
constexpr int EPI_TOK = 32;                  // tokens per epilogue pass
constexpr int NWARPS = 24;
constexpr int PTH = NWARPS * 32;
constexpr int DQ_WARP0 = 8, DQ_WARPS = 8;      // warps 8 .. 8 + 2 * DQ_WARPS - 1: the de-quantisers and epilogue helpers
constexpr int DQ_TEAM_WARPS = 6;               // twelve of them convert: two teams of six warps on alternate stages
constexpr int EPI_WARP0 = 4;
constexpr int kMaxPJobs = kMaxJobs;

struct PrefillCfg {
  CUtensorMap xmap;          // activations: (k, token), box 64 x BN, 128-byte swizzle
  int bn;                    // tokens per MMA and activation box: 64, 128 or 256
  int nh;                    // boxes per tile: 2 when the tile takes both accumulators (512 tokens), else 1
  int n_ttiles;              // token tiles
  int wtile_begin[kMaxPJobs + 1];   // first weight tile of each job
  int n_tiles;               // weight tiles (all jobs) x token tiles
  int n_kb;                  // visited k-blocks of 64: kept blocks of every head, head after head
  int km_start, km_period;   // input map in k-blocks: first stored block of head 0, stored blocks per head
  int km_kbh, km_keep;       // kept k-blocks per head (the last may be partly kept), kept channels per head
  uint32_t idesc;
  int streamk;               // 1: contiguous ranges of (tile, k-block) units per block; 0: whole tiles round-robin
  int helpers;               // 1: the de-quantiser warps share the epilogue of the block's last tile
  int sk_atomic;             // stream-K hand-over: 1 = parts added into one sum per tile (reductions in L2), 0 = a slot per part
  int pair_split;            // clusters of two blocks on one tile, half of the contraction each; the second block's
                             // fp32 sums go into the first one's shared memory (the rings, idle by then)
  int csplit;                // block pairs, one box per tile: pairs (of one cluster) that share a tile's contraction
  int halves;                // tiles on both accumulators: the tiles left over after the whole rounds run as half tiles
                             // (one box of 256 tokens each, on twice as many blocks), every block's last segment
  int* status;
  int* counters;             // stream-K: arrivals per tile
  float* partials;           // stream-K: one slot [tokens / 32][128 rows][32 tokens] fp32 per (left-over tile, block) piece
};

// Work of a block as a sequence of segments (tile, k-blocks [kb0, kb1)): whole tiles t = b, b + grid, ...
// With stream-K only for as many rounds as fill every block; the k-blocks of the tiles left over are
// cut into equal contiguous ranges, one per block, so that every SM stays busy however few tiles remain.
// A block runs its range of the split tiles FIRST: handing over the partial tile and finishing the split
// tiles then overlap the main loop of the whole tiles that follow instead of standing at the kernel's end.  Blocks stay in step along k (few distinct k offsets are alive at a time, which keeps the
// activation slices in L2).  Every block adds its fp32 partial tile to the tile's accumulation buffer in the
// workspace (reductions done in L2); the last of the tile's blocks to arrive reads the sum
// and finishes the tile.  With more than two blocks on a tile the order of the additions, and so the last
// bit of the fp32 sum, depends on the order of arrival.
// Visited k-block v of the input map -> stored k-block, first compact activation column, kept channels in it.
// One family {start, period, keep, count}: head h keeps channels [0, keep) of its period; a leading block is
// the case count = 1.  The activation box of a partly kept block also covers the first columns of the next
// head: the de-quantisers write zeros for the pruned channels of the block, so those columns do not count.
// Walked without a division per k-block (a division by the kept blocks per head cost the per-head launches 8 us
// of 52): (head, kept block within the head) of a visited k-block, stepped.
struct KWalk {
  int h, r;
  __device__ inline void start(const PrefillCfg& c, int v) { h = v / c.km_kbh; r = v - h * c.km_kbh; }
  __device__ inline void step(const PrefillCfg& c, int n) { r += n; while (r >= c.km_kbh) { r -= c.km_kbh; ++h; } }
  __device__ inline int stored(const PrefillCfg& c) const { return c.km_start + h * c.km_period + r; }
  __device__ inline int xcol(const PrefillCfg& c) const { return h * c.km_keep + r * BK; }
  __device__ inline int valid(const PrefillCfg& c) const { return min(BK, c.km_keep - r * BK); }
};

// half: -1 the whole tile; 0 / 1: only the first / second box of a tile of two boxes (into accumulator 0 / 1)
struct Seg { int tile, kb0, kb1, half; };
struct SegIter {
  long u, ue;
  int t, t_end, n_kb, step, tail_tile0, half_tile, half, ps_tile, ps_kb0, ps_kb1;
  // part: which of the pairs that share a tile's contraction this one is (-1: tiles are not shared)
  __device__ inline void init(const PrefillCfg& c, int b, int grid, int part) {
    n_kb = c.n_kb; step = grid; t = b;
    half_tile = -1; half = 0;
    ps_tile = -1;
    if (c.pair_split) {
      // block 2t takes the first k-blocks of tile t and finishes it, block 2t + 1 the rest (the smaller half)
      t_end = 0; tail_tile0 = 0; u = ue = 0; t = 1;
      ps_tile = b >> 1;
      const int mid = n_kb - n_kb / 2;
      ps_kb0 = (b & 1) ? mid : 0;
      ps_kb1 = (b & 1) ? n_kb : mid;
      return;
    }
    if (part >= 0) {
      // one tile per cluster, a part of its k-blocks per pair
      t_end = 0; tail_tile0 = 0; u = ue = 0; t = 1;
      ps_tile = b;
      ps_kb0 = n_kb * part / c.csplit; ps_kb1 = n_kb * (part + 1) / c.csplit;
      return;
    }
    if (c.halves) {
      // whole rounds of whole tiles, then tile (rounds * grid + b / 2) as two halves on blocks b and b + 1
      const int full = (c.n_tiles / grid) * grid;
      t_end = full; tail_tile0 = full; u = ue = 0;
      if (full + b / 2 < c.n_tiles) { half_tile = full + b / 2; half = b & 1; }
      return;
    }
    const int base = c.streamk ? c.n_tiles / grid : (c.n_tiles + grid - 1) / grid;
    t_end = c.streamk ? base * grid : c.n_tiles;
    tail_tile0 = base * grid;
    u = ue = 0;
    if (c.streamk) {
      const long Ut = (long)(c.n_tiles - tail_tile0) * c.n_kb;
      const long Bt = grid < Ut ? grid : Ut;
      if (b < Bt) { u = Ut * b / Bt; ue = Ut * (b + 1) / Bt; }
    }
  }
  __device__ inline bool next(Seg& sg) {
    if (u < ue) {
      const int tt = (int)(u / n_kb);
      sg.tile = tail_tile0 + tt;
      sg.kb0 = (int)(u - (long)tt * n_kb);
      const long len = (n_kb - sg.kb0) < (ue - u) ? (n_kb - sg.kb0) : (ue - u);
      sg.kb1 = sg.kb0 + (int)len;
      sg.half = -1;
      u += len;
      return true;
    }
    if (t < t_end) {
      sg.tile = t; sg.kb0 = 0; sg.kb1 = n_kb; sg.half = -1;
      t += step;
      return true;
    }
    if (ps_tile >= 0) {
      sg.tile = ps_tile; sg.kb0 = ps_kb0; sg.kb1 = ps_kb1; sg.half = -1;
      ps_tile = -1;
      return true;
    }
    if (half_tile >= 0) {
      sg.tile = half_tile; sg.kb0 = 0; sg.kb1 = n_kb; sg.half = half;
      half_tile = -1;
      return true;
    }
    return false;
  }
};
// block whose range [U*b/B, U*(b+1)/B) of the left-over units holds unit u (exact in fp64 for these magnitudes)
__device__ inline int sk_owner(long u, long B, long U) {
  return (int)floor(((double)(u + 1) * (double)B - 1.0) / (double)U);
}

// bf16 activations -> fp16 copy in the workspace, once per call (every weight tile re-reads the tile of
// activations, so converting there would repeat the work once per 128 weight rows).
__global__ void x_to_f16_kernel(const __nv_bfloat16* __restrict__ x, int ldx, int M, int k_in, __half* __restrict__ o, int ldo) {
  // (programmatic dependent launch: the tensor-core kernel behind this one may set itself up meanwhile; this one
  //  waits for its own predecessor before it reads x or overwrites the copy that predecessor may still read)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int units = ldo / 8;                         // 16-byte units per output row (ldo is a multiple of 8)
  const long total = (long)M * units;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
    const int m = (int)(i / units), u = (int)(i - (long)m * units);
    const __nv_bfloat16* src = x + (size_t)m * ldx + u * 8;
    uint32_t w[4];
    if (u * 8 + 8 <= k_in && ((ldx & 7) == 0) && ((((uintptr_t)x) & 15) == 0)) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(src));
      w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int k0 = u * 8 + 2 * e;
        const uint32_t lo = k0 < k_in ? __bfloat16_as_ushort(src[2 * e]) : 0u;
        const uint32_t hi = k0 + 1 < k_in ? __bfloat16_as_ushort(src[2 * e + 1]) : 0u;
        w[e] = lo | (hi << 16);
      }
    }
    uint4 r;
    r.x = bf16x2_to_f16x2(w[0]); r.y = bf16x2_to_f16x2(w[1]); r.z = bf16x2_to_f16x2(w[2]); r.w = bf16x2_to_f16x2(w[3]);
    *reinterpret_cast<uint4*>(o + (size_t)m * ldo + u * 8) = r;
  }
}

// T: activation / output type.  CONV: the activation tiles arrive as bf16 and are converted to fp16 in
// shared memory by the de-quantisers (used when the workspace cannot hold a converted copy).
// HEADS: the input map is a family of per-head blocks (else a leading block).
// PAIR: clusters of two blocks work on tiles of 256 weight rows with cta_group::2 MMAs.  Each block de-quantises 128 rows
// into its own shared memory and fetches half of the tokens' boxes; the first block's MMA warp issues for both.  A block's
// shared memory then takes in 16 instead of 32 KB of activations per 256 tokens and k-block, which with one block per tile
// was what L2 could not deliver and the shared-memory port could not take beside the operand reads.  PAIR = 1 / 2: one or
// two boxes of 256 tokens per tile; 3: one box, and the pairs of a cluster share a tile (an instance of its own: inside 1 its
// registers cost every launch 3 - 10 %).
template <typename T, bool CONV, bool HEADS, int PAIR>
__global__ void __launch_bounds__(PTH, 1) prefill_kernel(const __grid_constant__ Params p,
                                                         const __grid_constant__ PrefillCfg c) {
  extern __shared__ unsigned char psmem_raw[];
  constexpr bool ONE = PAIR == 1 || PAIR == 3;              // block pairs, one box of tokens per tile
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (warp-uniform for the compiler)
  // Programmatic dependent launch: the next kernel of the stream may be set up while this one runs (its blocks
  // become resident as ours leave).  What a block does before its own `griddepcontrol.wait` touches nothing a
  // predecessor may still write or read: barriers, tensor memory, and the weights, which no kernel writes (the
  // de-quantisers fill the ring ahead); activations, positions, outputs and workspace come after the wait.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t raw = (uint32_t)__cvta_generic_to_shared(psmem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;           // swizzled tiles need 1024-byte alignment
  unsigned char* smem = psmem_raw + (sbase - raw);
  constexpr int NB = ONE ? PSTAGES1 : PAIR ? 2 * PSTAGES2 : BSLOTS;               // slots of the activation ring and their size
  constexpr int NB_BYTES = PAIR ? B_BYTES / 2 : B_BYTES;
  // PAIR: the pair's number and their count (3: the cluster's), and this pair's part of a shared tile
  const int n_share = PAIR == 3 ? c.csplit : 1, per = PAIR ? 2 * n_share : 1;
  const int bid = PAIR ? (int)blockIdx.x / per : (int)blockIdx.x, nblk = PAIR ? (int)gridDim.x / per : (int)gridDim.x;
  const uint32_t rank = (PAIR || c.pair_split) ? pcluster_rank() : 0u;
  const uint32_t crank = PAIR == 3 ? rank & 1u : rank, lrank = PAIR == 3 ? rank & ~1u : 0u;   // block of the pair, rank of the pair's first block
  const int part = PAIR == 3 ? (int)(rank >> 1) : -1;
  constexpr int NA = ONE ? PSTAGES1 : PAIR ? PSTAGES2 : PSTAGES;             // weight stages
  constexpr int RING = PAIR ? RING2_BYTES : RING_BYTES;
  constexpr int B_RING = NA * A_BYTES;                      // the activation boxes follow the weight stages
  constexpr int TEAM_WARPS = ONE ? DQ_WARPS : DQ_TEAM_WARPS;
  const uint32_t bars = sbase + RING;
  const uint32_t full_a = bars, empty_a = bars + 8 * NA;
  // (PAIR: a stage's weights and its half boxes share one pair of barriers -- the MMA warp's loop is one chain of
  //  dependent instructions, 890 cycles per k-block of one box with two waits and two commits where the MMAs take 512)
  const uint32_t full_b = PAIR ? full_a : bars + 16 * NA, empty_b = PAIR ? empty_a : full_b + 8 * NB;
  const uint32_t acc_full = bars + 16 * NA + 16 * NB, acc_empty = acc_full + 16, epi_bar = acc_full + 32;
  const uint32_t help_bar = acc_full + 40;         // the epilogue warps and the de-quantiser warps that help them
  const uint32_t last_full = acc_full + 48;        // the MMAs of the block's last segment are complete (one phase only)
  const uint32_t px_ready = acc_full + 56;         // pair split, second block: the first block's rings are idle
  const uint32_t px_done = acc_full + 64;          // pair split, first block: the second block's sums have arrived
  const uint32_t xq = acc_full + 72;               // pairs that share a tile: the others' sums have arrived, per quadrant
  unsigned char* misc = smem + RING + 16 * NA + 16 * NB + 104;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  if (tid == 0) {
    for (int s = 0; s < NA; ++s) {
      pmbar_init(full_a + 8 * s, PAIR ? 2 * TEAM_WARPS + 1 : TEAM_WARPS);
      pmbar_init(empty_a + 8 * s, 1);
    }
    for (int s = 0; s < NB && !PAIR; ++s) {
      pmbar_init(full_b + 8 * s, 1);
      pmbar_init(empty_b + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) { pmbar_init(acc_full + 8 * b, 1); pmbar_init(acc_empty + 8 * b, PAIR ? 8 : 4); }
    pmbar_init(epi_bar, 4);
    pmbar_init(help_bar, 4 + 2 * DQ_WARPS);
    pmbar_init(last_full, 1);
    pmbar_init(px_ready, 1);
    pmbar_init(px_done, c.helpers ? 4 + 2 * DQ_WARPS : 4);       // one arrival per warp that sends
    if (PAIR == 3)
      for (int b = 0; b < 4; ++b) pmbar_init(xq + 8 * b, max(1, (n_share - 1) * (c.helpers ? 5 : 1)));
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {                      // the whole tensor memory of the SM: two accumulators of 256 columns
    const uint32_t slot = (uint32_t)__cvta_generic_to_shared(const_cast<uint32_t*>(tmem_slot));
    if (PAIR) {
      tmem_alloc_pair(slot, 512);
    } else {
      tmem_alloc(slot, 512);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if (PAIR || c.pair_split) {                   // the other block's barriers exist before anything is sent to it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }

  // 128-row tile of its job that this block holds (PAIR: tiles are counted in pairs)
  auto local_tile = [&](int wt, int jn) { return PAIR ? 2 * (wt - c.wtile_begin[jn]) + (int)crank : wt - c.wtile_begin[jn]; };
  auto job_of_wt = [&](int wt) { int j = 0; while (j + 1 < p.n_jobs && wt >= c.wtile_begin[j + 1]) ++j; return j; };
  bool failed = false;

  // ---- the epilogue of one segment, for the warp that calls it: accumulator -> bias, rotary embedding or gated
  //      product, rounding, store.  A warp reaches the tensor-memory lanes 32 (warp % 4) .. + 31 (a lane is a tile
  //      row); it takes the chunks ch0, ch0 + chs, ... of 32 tokens.  chs == 1: the epilogue warp on its own (it
  //      also hands the accumulators back and runs the hand-over of a tile split along K).
  const int q = warp & 3;                          // TMEM lanes 32q .. 32q+31
  const int etid = 32 * q + lane;                  // tile row handled in the store phase
  uint32_t epar = 0;
  auto epi_sync = [&]() -> bool {
    __syncwarp();
    if (lane == 0) pmbar_arrive(epi_bar);
    const bool ok = pmbar_wait(epi_bar, epar, abort_flag);
    epar ^= 1;
    return ok;
  };
  volatile int* last_flag = reinterpret_cast<volatile int*>(misc + 8);
  uint32_t hpar = 0;
  auto help_sync = [&]() -> bool {
    __syncwarp();
    if (lane == 0) pmbar_arrive(help_bar);
    const bool ok = pmbar_wait(help_bar, hpar, abort_flag);
    hpar ^= 1;
    return ok;
  };
  auto epilogue_segment = [&](const Seg& sg, int tcount, int ch0, int chs, bool acc_known_full) {
      const int acc0 = c.nh == 2 ? 0 : (tcount & 1);     // as in the MMA warp
      const int au = c.nh == 2 ? tcount : (tcount >> 1);
      const int ntok = c.bn * c.nh;                      // tokens of the tile
      const int h_lo = sg.half < 0 ? 0 : sg.half, h_hi = sg.half < 0 ? c.nh : sg.half + 1;   // boxes of this segment
      const int t = sg.tile;
      const int wt = t / c.n_ttiles, tt = t - wt * c.n_ttiles;
      const int jn = job_of_wt(wt);
      const int tl = local_tile(wt, jn);
      // this thread owns tile row etid (= its TMEM lane); a rope pair sits in lanes 2i, 2i + 1
      const RowStore<T> rs(p, jn, tile_row(p.job[jn], tl, etid), (etid & 1) != 0);
      auto store_chunk = [&](int tok0, const auto& val) { rs.store(p, tt * ntok + tok0, val); };
      for (int h = h_lo; h < h_hi && !failed && !acc_known_full; ++h)
        if (!pmbar_wait(acc_full + 8 * (acc0 + h), au & 1, abort_flag)) failed = true;
      if (failed) return;
      tc_fence_after();
      // (the two accumulators are neighbours in tensor memory: a tile of two boxes is 512 consecutive columns)
      const uint32_t t_acc = tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc0 * MAXBN);
      const int row = 32 * q + lane;
      // this warp is done with the accumulator that holds token chunk `ch` once that chunk was its last
      auto release_after = [&](int ch) {
        if (((ch + 1) * EPI_TOK) % c.bn != 0) return;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          const uint32_t eb = acc_empty + 8 * (acc0 + (ch * EPI_TOK) / c.bn);
          if (PAIR) pmbar_signal_peer(ppeer_addr(eb, lrank)); else pmbar_arrive(eb);
        }
      };
      if (sg.kb0 == 0 && sg.kb1 == c.n_kb) {
        // ---- the whole contraction of this tile ran here (this warp takes every chs-th chunk of 32 tokens;
        //      of a half tile only the chunks of its box)
        const int cpb = c.bn / EPI_TOK;
        for (int ch = h_lo * cpb + ch0; ch < h_hi * cpb; ch += chs) {
          uint32_t v[32];
          tmem_ld32(t_acc + (uint32_t)(ch * EPI_TOK), v);
          tmem_ld_wait();
          if (chs == 1) release_after(ch);               // (the values are in registers)
          float val[32];
#pragma unroll
          for (int k = 0; k < 32; ++k) val[k] = __uint_as_float(v[k]);
          store_chunk(ch * EPI_TOK, val);
        }
      } else {
        // ---- a part of the contraction (stream-K): the fp32 partial tile goes to a slot of its own in the
        //      workspace, [token][row] (a warp writes and later reads 32 consecutive rows of a token: whole
        //      128-byte lines); the last of the tile's blocks to arrive adds the slots of all of them in block
        //      order (the same sum whatever the order of arrival) and finishes the tile.
        //      The pieces (tile, block) of the cut unit line are numbered lt + block: both grow along the line and
        //      one of them grows from each piece to the next, so no two pieces share a number.
        //      chs > 1: the block's last segment, shared with the de-quantiser warps (twenty warps write, meet at a
        //      barrier of their own, and -- in the last block to arrive -- read back and finish).
        //      Where a few split tiles in front of whole tiles have many parts each, reading all the slots back
        //      would take the four epilogue warps longer than the tiles behind can hide: such launches add the parts
        //      into ONE sum per tile instead (reductions done in L2, zero at launch; the last bit of a sum then
        //      depends on the order of arrival when more than two blocks share a tile).
        if (PAIR == 3) {
          // ---- the pairs of a cluster share this tile.  Eight tokens at a time: pair i % n_share finishes chunk i.  Each
          //      leaves its sums of the other pairs' chunks in a slot ([token][row], L2), tells them (remote arrivals,
          //      one per warp and pair), and adds up and finishes its own chunks in the order of the parts.
          float* slots = c.partials + row;
          const float* first = slots + (size_t)(blockIdx.x - rank + crank) * (MAXBN * BMW);   // part 0's block of the same rows
          float* mine = slots + (size_t)blockIdx.x * (MAXBN * BMW);
          constexpr int CH = 8, N_CH = MAXBN / CH;
          for (int ch = ch0; ch < N_CH; ch += chs) {
            if (ch % n_share == part) continue;
            uint32_t v[8];
            tmem_ld8(t_acc + (uint32_t)(ch * CH), v);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 8; ++k) __stcg(mine + (size_t)(ch * CH + k) * BMW, __uint_as_float(v[k]));
          }
          __syncwarp();
          if (lane < n_share && lane != part) {
            asm volatile("fence.acq_rel.cluster;" ::: "memory");
            pmbar_arrive_peer(ppeer_addr(xq + 8 * q, (uint32_t)(2 * lane) + crank));
          }
          if (!__all_sync(0xffffffffu, pmbar_wait_cluster(xq + 8 * q, 0, abort_flag))) { failed = true; return; }
          for (int own = ch0; part + own * n_share < N_CH; own += chs) {
            const int tk = (part + own * n_share) * CH;
            if (tt * ntok + tk >= p.M) break;
            uint32_t v[8];
            tmem_ld8(t_acc + (uint32_t)tk, v);
            tmem_ld_wait();
            float val[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) val[k] = 0.f;
            const float* src = first + (size_t)tk * BMW;
            for (int r0 = 0; r0 < n_share; r0 += 2) {          // two parts in flight, added in their order
              float a[8], b[8];
              const bool own_a = r0 == part, own_b = r0 + 1 == part, has_b = r0 + 1 < n_share;
#pragma unroll
              for (int k = 0; k < 8; ++k) a[k] = own_a ? __uint_as_float(v[k]) : __ldcg(src + (size_t)(2 * r0) * (MAXBN * BMW) + (size_t)k * BMW);
#pragma unroll
              for (int k = 0; k < 8; ++k) b[k] = own_b ? __uint_as_float(v[k]) : has_b ? __ldcg(src + (size_t)(2 * r0 + 2) * (MAXBN * BMW) + (size_t)k * BMW) : 0.f;
#pragma unroll
              for (int k = 0; k < 8; ++k) val[k] = (val[k] + a[k]) + b[k];
            }
            store_chunk(tk, val);
          }
          return;
        }
        const bool pair_send = c.pair_split && crank != 0;
        if (c.pair_split && !pair_send) {
          // ---- the two blocks of a cluster each ran half of the contraction.  The second block waits until the
          //      first one's MMAs are complete (its rings are idle then), writes its fp32 sums into them ([token][row]:
          //      a warp stores 32 consecutive rows of a token) and arrives, one arrival per warp, at the first block's
          //      barrier; the first block adds them to its own sums (always own + other: the same bits every run)
          //      and finishes the tile.  No traffic through L2, no counter, nothing to clear.
          {
            if (!pmbar_wait_cluster(px_done, 0, abort_flag)) { failed = true; return; }
            // (16 tokens at a time, as the read-back of the slots: what the registers of a thread hold)
            for (int tk = 16 * ch0; tk < ntok; tk += 16 * chs) {
              uint32_t v[16];
              tmem_ld16(t_acc + (uint32_t)tk, v);
              tmem_ld_wait();
              const uint32_t src = sbase + (uint32_t)((tk * BMW + row) * 4);
              float val[16];
              pld_add_f32x16<BMW * 4>(src, v, val);
              store_chunk(tk, val);
            }
          }
          return;
        }
        const bool main_lane = warp == EPI_WARP0 && lane == 0;
        const size_t slot_f = (size_t)ntok * BMW;
        const int T0 = (c.n_tiles / nblk) * nblk;              // first left-over tile
        // (PAIR: two slots side by side, a block's own 128 rows in each)
        auto slot_of = [&](int n) { return c.partials + (PAIR ? 2 * (size_t)n + crank : (size_t)n) * slot_f; };
        float* mine = slot_of((t - T0) + (c.sk_atomic ? 0 : bid));
        int* arrivals = &c.counters[PAIR ? 2 * t + (int)crank : t];
        if (pair_send) {
          // (the second block of a pair: its "slot" is the first block's rings, once they are idle)
          if (!pmbar_wait_cluster(px_ready, 0, abort_flag)) { failed = true; return; }
          mine = ppeer_generic(smem, 0u);
        }
        for (int ch = ch0; ch < ntok / EPI_TOK; ch += chs) {
          uint32_t v[32];
          tmem_ld32(t_acc + (uint32_t)(ch * EPI_TOK), v);
          tmem_ld_wait();
          if (chs == 1) release_after(ch);                     // the accumulator is free for the next segment
          float* dst = mine + (size_t)(ch * EPI_TOK) * BMW + row;
          if (pair_send) {
#pragma unroll
            for (int k = 0; k < 32; ++k) dst[(size_t)k * BMW] = __uint_as_float(v[k]);
          } else if (c.sk_atomic) {
#pragma unroll
            for (int k = 0; k < 32; ++k) atomicAdd(dst + (size_t)k * BMW, __uint_as_float(v[k]));
          } else {
#pragma unroll
            for (int k = 0; k < 32; ++k) __stcg(dst + (size_t)k * BMW, __uint_as_float(v[k]));
          }
        }
        if (pair_send) {
          __syncwarp();
          if (lane == 0) {
            asm volatile("fence.acq_rel.cluster;" ::: "memory");
            pmbar_arrive_peer(ppeer_addr(px_done, 0u));
          }
          return;
        }
        __threadfence();                                       // this thread's part is in place before ...
        if (!(chs == 1 ? epi_sync() : help_sync())) { failed = true; return; }
        const long U = (long)(c.n_tiles - T0) * c.n_kb, Bn = (long)nblk < U ? (long)nblk : U;
        const long tu = (long)(t - T0) * c.n_kb;                               // the tile's first left-over unit
        const int first = sk_owner(tu, Bn, U), last = sk_owner(tu + c.n_kb - 1, Bn, U);
        if (main_lane) {
          const int arrived = atomicAdd(arrivals, 1);          // ... the block's arrival shows
          *last_flag = arrived == last - first;
          __threadfence();
        }
        if (!(chs == 1 ? epi_sync() : help_sync())) { failed = true; return; }
        if (*last_flag) {
          const float* base = slot_of((t - T0) + (c.sk_atomic ? 0 : first));
          const size_t part_f = PAIR ? 2 * slot_f : slot_f;    // from one block's part to the next one's
          const int parts = c.sk_atomic ? 1 : last - first + 1;
          // 16 tokens at a time, the loads of two slots in flight together (what the registers of a thread hold)
          for (int tk = 16 * ch0; tk < ntok; tk += 16 * chs) {
            float val[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) val[k] = 0.f;
            const float* src = base + (size_t)tk * BMW + row;
            for (int s2 = 0; s2 < parts; s2 += 2) {
              const bool two = s2 + 1 < parts;
              float a[16], b[16];
#pragma unroll
              for (int k = 0; k < 16; ++k) a[k] = __ldcg(src + (size_t)s2 * part_f + (size_t)k * BMW);
#pragma unroll
              for (int k = 0; k < 16; ++k) b[k] = two ? __ldcg(src + (size_t)(s2 + 1) * part_f + (size_t)k * BMW) : 0.f;
#pragma unroll
              for (int k = 0; k < 16; ++k) val[k] = (val[k] + a[k]) + b[k];
            }
            store_chunk(tk, val);
          }
          if (main_lane) *arrivals = 0;                  // ready for the next call
        }
      }
  };

  if (warp == 0) {
    // ===================================================================== activations by TMA
    if (PAIR) {
      // (warp-uniform, as the MMA warp: one lane walking this loop took longer per k-block than the MMAs do)
      asm volatile("griddepcontrol.wait;" ::: "memory");
      constexpr int NH = ONE ? 1 : 2;
      const uint32_t rfull = ppeer_addr(full_a, lrank);       // both blocks' half boxes count on the first block's barriers
      int s = 0, it = 0; uint32_t par = 1;
      SegIter si; si.init(c, bid, nblk, part);
      Seg sg;
      while (!failed && si.next(sg)) {
        const int n_box = NH == 1 || sg.half >= 0 ? 1 : 2;
        const int y0 = ((sg.tile % c.n_ttiles) * NH + (NH == 2 && sg.half > 0 ? 1 : 0)) * MAXBN + (int)crank * (MAXBN / 2);
        KWalk kw;
        if (HEADS) kw.start(c, sg.kb0);
        for (int kb = sg.kb0; kb < sg.kb1; ++kb, ++it) {
          const int x = HEADS ? kw.xcol(c) : kb * BK;
          if (HEADS) kw.step(c, 1);
          if (it >= NA && !pmbar_wait_warp(empty_a + 8 * s, par, abort_flag)) { failed = true; break; }
          if (elect_one()) {
            if (crank == 0) pmbar_expect_tx(full_a + 8 * s, (uint32_t)(n_box * MAXBN * BK * 2));
            const uint32_t dst = sbase + B_RING + s * NH * NB_BYTES;
            tma_box2_pair(dst, &c.xmap, x, y0, rfull + 8 * s);
            if (n_box == 2) tma_box2_pair(dst + NB_BYTES, &c.xmap, x, y0 + MAXBN, rfull + 8 * s);
          }
          __syncwarp();
          if (++s == NA) { s = 0; par ^= 1; }
        }
      }
      if (failed)                           // copies may still be on their way into this block's shared memory: they land well
        for (int i = 0; i < 1000; ++i) __nanosleep(200);        // within this time
    } else if (lane == 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");   // the activations may come from the preceding kernel
      int s = 0; uint32_t par = 1; int jb = 0;             // box slot, parity of its previous use, boxes so far
      SegIter si; si.init(c, bid, nblk, part);
      Seg sg;
      while (!failed && si.next(sg)) {
        const int tt = sg.tile % c.n_ttiles;
        KWalk kw;
        if (HEADS) kw.start(c, sg.kb0);
        for (int kb = sg.kb0; kb < sg.kb1 && !failed; ++kb) {
          const int xcol = HEADS ? kw.xcol(c) : kb * BK;
          if (HEADS) kw.step(c, 1);
          const int h_lo = sg.half < 0 ? 0 : sg.half, h_hi = sg.half < 0 ? c.nh : sg.half + 1;
          for (int h = h_lo; h < h_hi; ++h, ++jb) {
            if (jb >= NB && !pmbar_wait(empty_b + 8 * s, par, abort_flag, true)) { failed = true; break; }
            const uint32_t fb = full_b + 8 * s;
            // (a box that starts at or beyond the last token is all zeros: the tensor map ends at M)
            pmbar_expect_tx(fb, (uint32_t)(c.bn * BK * 2));
            tma_box2(sbase + B_RING + s * NB_BYTES, &c.xmap, xcol, (tt * c.nh + h) * c.bn, fb);
            if (++s == NB) { s = 0; par ^= 1; }
          }
        }
      }
      if (failed)                           // copies may still be on their way into this block's shared memory: they land well
        for (int i = 0; i < 1000; ++i) __nanosleep(200);        // within this time
    }
  } else if (warp == 1) {
    // ===================================================================== MMA issue
    // (the whole warp walks the loop, so that stage indexes, parities and descriptors are warp-uniform; one elected
    //  lane issues)
    if (!PAIR || crank == 0) {
      const unsigned short pair_mask = (unsigned short)(3u << lrank);
      auto commit = [&](uint32_t bar) { if (PAIR) umma_commit_pair(bar, pair_mask); else umma_commit(bar); };
      int s = 0; uint32_t par = 0; int tcount = 0;         // weight stage and its parity
      int sb = 0; uint32_t parb = 0;                       // activation box slot and its parity
      SegIter si; si.init(c, bid, nblk, part);
      Seg sg;
      for (; !failed && si.next(sg); ++tcount) {
        // A tile of one box alternates between the two accumulators; a tile of two boxes holds both: the
        // de-quantised weight stage then serves 512 tokens, and the accumulator of the first 256 is drained by
        // the epilogue while the MMAs of the next tile already run on ... once it is free again (per-accumulator waits).
        const int acc0 = c.nh == 2 ? 0 : (tcount & 1);
        const int au = c.nh == 2 ? tcount : (tcount >> 1);   // earlier tiles that used this tile's accumulator(s)
        const int h_lo = sg.half < 0 ? 0 : sg.half, h_hi = sg.half < 0 ? c.nh : sg.half + 1;   // (a half tile is a block's last)
        for (int kb = sg.kb0; kb < sg.kb1 && !failed; ++kb) {
          if (!pmbar_wait_warp(full_a + 8 * s, par, abort_flag)) { failed = true; break; }
          const uint64_t adesc = smem_desc_sw128(sbase + s * A_BYTES);
          if (PAIR == 2) {
            // (one wait and one commit per k-block; the same shape for one box measured 20 % slower than the loop below)
            constexpr int NH = 2;
            const uint64_t bdesc = smem_desc_sw128(sbase + B_RING + s * NH * NB_BYTES);
            const uint32_t more = kb > sg.kb0 ? 1u : 0u;
            const int n_box = h_hi - h_lo;
            if (kb == sg.kb0 && au >= 1) {                // (the accumulators are still being drained: one after the other)
              for (int h = 0; h < n_box; ++h) {
                if (!pmbar_wait_warp(acc_empty + 8 * (acc0 + h_lo + h), (au - 1) & 1, abort_flag)) { failed = true; break; }
                tc_fence_after();
                if (elect_one()) umma_kblock<true>(tmem_base + (uint32_t)((acc0 + h_lo + h) * MAXBN), adesc, bdesc + h * (NB_BYTES >> 4), c.idesc, 0u);
                __syncwarp();
              }
              if (failed) break;
              if (elect_one()) umma_commit_pair(empty_a + 8 * s, pair_mask);
            } else {
              tc_fence_after();
              if (elect_one()) {
                umma_kblock<true>(tmem_base + (uint32_t)((acc0 + h_lo) * MAXBN), adesc, bdesc, c.idesc, more);
                if (n_box == 2) umma_kblock<true>(tmem_base + (uint32_t)((acc0 + 1) * MAXBN), adesc, bdesc + (NB_BYTES >> 4), c.idesc, more);
                umma_commit_pair(empty_a + 8 * s, pair_mask);        // the stage is free once these MMAs have read it
              }
            }
            __syncwarp();
            if (++s == NA) { s = 0; par ^= 1; }
            continue;
          }
          for (int h = h_lo; h < h_hi; ++h) {
            if (kb == sg.kb0 && au >= 1 && !pmbar_wait_warp(acc_empty + 8 * (acc0 + h), (au - 1) & 1, abort_flag)) { failed = true; break; }
            // (bf16: the de-quantisers waited for the activation box themselves and converted it)
            if (!CONV && !ONE && !pmbar_wait_warp(full_b + 8 * sb, parb, abort_flag)) { failed = true; break; }
            tc_fence_after();
            const uint32_t d_tmem = tmem_base + (uint32_t)((acc0 + h) * MAXBN);
            const uint64_t bdesc = smem_desc_sw128(sbase + B_RING + sb * NB_BYTES);
            if (elect_one()) {
              umma_kblock<PAIR != 0>(d_tmem, adesc, bdesc, c.idesc, kb > sg.kb0 ? 1u : 0u);
              if (!ONE) commit(empty_b + 8 * sb);    // the box is free once these MMAs have read it
              if (ONE || h == h_hi - 1) commit(empty_a + 8 * s);   // ... and the weight stage after the last of them
            }
            __syncwarp();
            if (++sb == NB) { sb = 0; parb ^= 1; }
          }
          if (failed) break;
          if (++s == NA) { s = 0; par ^= 1; }
        }
        if (failed) break;
        // (the de-quantiser warps that help with the last segment's epilogue cannot follow the phases of the
        //  accumulator barriers -- a parity wait cannot tell "not yet" from "two phases ago" -- so the last
        //  segment completes a barrier of its own, which has this one phase)
        SegIter peek = si;
        Seg nxt;
        const bool last = !peek.next(nxt);
        if (elect_one()) {
          for (int h = h_lo; h < h_hi; ++h) commit(acc_full + 8 * (acc0 + h));
          if (last) commit(last_full);
        }
        __syncwarp();
      }
      if (c.pair_split && crank == 0 && !failed) {
        // the first block of a pair: once its own MMAs are complete nothing reads its rings any more
        if (pmbar_wait_warp(last_full, 0, abort_flag)) {
          if (lane == 0) {
            asm volatile("fence.acq_rel.cluster;" ::: "memory");
            pmbar_arrive_peer(ppeer_addr(px_ready, 1u));
          }
        } else {
          failed = true;
        }
      }
    }
  } else if (warp >= DQ_WARP0) {
    // ===================================================================== de-quantisers
    // Two teams of six warps take alternate stages (a team always meets the same ring slots again, so its parity
    // waits are never more than one phase away from their barriers); a thread converts 32 codes of a weight row,
    // the first 64 threads of a team a second such item (256 items on 192 threads).  The teams are the twelve
    // warps on the three schedulers that do NOT host the MMA warp (warp % 4 != 1): the lane that issues the MMAs
    // runs one dependent instruction after the other, and with four busy warps on its scheduler every one of them
    // waited longer for its issue slot (measured with those four warps idle, results wrong by construction: Qwen
    // gate at M = 2048 296 -> 266 us with tiles of 256 tokens, 251 -> 232 us with 512).  The four warps 9, 13, 17,
    // 21 only help with the block's last epilogue (below).
    const int sc = warp & 3;
    // Pairs with one box per tile: all sixteen warps, two teams of eight with one item per thread.  (The MMA lane of a pair
    // has half as much to issue per k-block, and a k-block half the time: with twelve warps a team's two rounds of items,
    // 1130 cycles, set the pace.  With two boxes per tile the twelve are 4 % faster there too.)
    if (TEAM_WARPS == DQ_WARPS || sc != 1) {
    const int pos = TEAM_WARPS == DQ_WARPS ? warp - DQ_WARP0 : ((warp - DQ_WARP0) >> 2) * 3 + (sc == 0 ? 0 : sc - 1);   // among the sixteen or twelve
    const int team = pos >= TEAM_WARPS ? 1 : 0;
    const int dt = (pos - team * TEAM_WARPS) * 32 + lane;                       // 0..191 or 0..255
    constexpr int TEAM_TH = TEAM_WARPS * 32;
    const int n_items = ONE ? 1 : dt + TEAM_TH < 2 * BMW ? 2 : 1;                         // items dt and dt + 192 of 256
    const int G = p.K / kGroup;
    int done = 0;                      // stage iterations before this segment
    constexpr bool heads = HEADS;
    SegIter si; si.init(c, bid, nblk, part);
    Seg sg;
    for (; !failed && si.next(sg); done += sg.kb1 - sg.kb0) {
      const int it0 = done - sg.kb0;   // stage iteration of k-block kb of this segment = it0 + kb
      const int wt = sg.tile / c.n_ttiles;
      const int jn = job_of_wt(wt);
      const JobDev& jb = p.job[jn];
      bool live[2];
      const uint8_t* wrow[2];
      const __half* srow[2];
      const __half* zrow[2];
      uint32_t st_off[2];              // row and half of the item inside a stage (the swizzle is applied per word)
      int hf_of[2], r7[2];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        if (ONE && m > 0) { live[m] = false; wrow[m] = nullptr; srow[m] = zrow[m] = nullptr; st_off[m] = 0; hf_of[m] = r7[m] = 0; break; }
        const int item = dt + m * TEAM_TH;
        const int r = (item >> 1) & (BMW - 1), hf = item & 1;
        const RowInfo ri = tile_row(jb, local_tile(wt, jn), r);
        live[m] = m < n_items && ri.stored >= 0;
        const JobDev& src = (jb.pair == 1 && (r & 1)) ? p.job[jn + 1] : jb;    // odd rows of a SwiGLU pair: the up matrix
        wrow[m] = src.w + (size_t)(live[m] ? ri.stored : 0) * (p.K / 2) + hf * 16;
        srow[m] = src.scales + (size_t)(live[m] ? ri.stored : 0) * G;
        zrow[m] = src.zeros + (size_t)(live[m] ? ri.stored : 0) * G;
        st_off[m] = (uint32_t)(r * 128);
        hf_of[m] = hf; r7[m] = r & 7;
      }
      const int kb0 = ((done & 1) == team) ? sg.kb0 : sg.kb0 + 1;
      // codes and scale / zero-point of this team's next k-block are kept in registers
      uint4 q0[2];
      __half s0[2], z0[2];
#pragma unroll
      for (int m = 0; m < 2; ++m) { q0[m] = make_uint4(0, 0, 0, 0); s0[m] = __ushort_as_half(0); z0[m] = s0[m]; }
      // codes, scale and zero-point of visited k-block v of an item's row; `valid` channels of it are kept
      // (a leading block needs no mask: the activation tensor map ends at k_in, so the tail of its last k-block
      //  meets zeros)
      // (the stored k-block of a visited one costs a division with per-head maps: worked out once for both items)
      auto fetch = [&](int m, int stored, uint4& q, __half& sc2, __half& zr) {
        q = __ldg(reinterpret_cast<const uint4*>(wrow[m] + (size_t)stored * 32));
        sc2 = __ldg(srow[m] + (stored >> 1)); zr = __ldg(zrow[m] + (stored >> 1));
      };
      KWalk kw;                                            // this team's current k-block
      if (heads && kb0 < sg.kb1) kw.start(c, kb0);
      if (kb0 < sg.kb1) {
        const int st0 = heads ? kw.stored(c) : kb0;
#pragma unroll
        for (int m = 0; m < 2; ++m)
          if (live[m]) fetch(m, st0, q0[m], s0[m], z0[m]);
      }
      for (int kb = kb0; kb < sg.kb1; kb += 2) {
        const int it = it0 + kb;
        const int s = it % NA;
        const uint32_t use = (uint32_t)(it / NA);
        uint4 q1[2];
        __half s1[2], z1[2];
        const bool more = kb + 2 < sg.kb1;
        const int v0 = heads ? kw.valid(c) : BK;           // kept channels of this k-block
        if (heads) kw.step(c, 2);
        const int st1 = (heads && more) ? kw.stored(c) : kb + 2;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          q1[m] = make_uint4(0, 0, 0, 0); s1[m] = s0[m]; z1[m] = z0[m];
          if (live[m] && more) fetch(m, st1, q1[m], s1[m], z1[m]);
        }
        if (it >= NA && !pmbar_wait(empty_a + 8 * s, (use - 1) & 1, abort_flag)) { failed = true; break; }
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          if (m >= n_items) break;
          const uint32_t a_st = sbase + s * A_BYTES + st_off[m];
          const __half2 sh2 = __half2half2(s0[m]);
          const __half2 cz2 = __float2half2_rn((8.f - __half2float(z0[m])) * __half2float(s0[m]));
          const uint32_t qw[4] = {q0[m].x, q0[m].y, q0[m].z, q0[m].w};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // (eight channels per word; keep counts are multiples of eight, so a word is kept or pruned whole)
            const uint4 o = (live[m] && (!HEADS || hf_of[m] * 32 + j * 8 < v0)) ? dequant_word(qw[j], sh2, cz2) : make_uint4(0, 0, 0, 0);
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a_st + (uint32_t)(((hf_of[m] * 4 + j) ^ r7[m]) * 16)), "r"(o.x), "r"(o.y), "r"(o.z), "r"(o.w) : "memory");
          }
        }
        if constexpr (CONV) {
          // bf16 activations: the tensor cores run on fp16 (8 more mantissa bits for the weights than bf16
          // would leave them); the activation tile that TMA delivered is converted in place
          for (int h = 0; h < c.nh && !failed; ++h) {
            const int jb2 = it * c.nh + h;                 // the k-block's boxes in the order the producer issued them
            const int sb = jb2 % BSLOTS;
            if (!pmbar_wait(full_b + 8 * sb, (uint32_t)(jb2 / BSLOTS) & 1, abort_flag)) { failed = true; break; }
            const uint32_t b_st = sbase + B_RING + sb * B_BYTES;
            for (int ci = dt; ci < c.bn * 8; ci += TEAM_TH) {
              uint32_t v0, v1, v2, v3;
              asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v0), "=r"(v1), "=r"(v2), "=r"(v3) : "r"(b_st + ci * 16));
              v0 = bf16x2_to_f16x2(v0); v1 = bf16x2_to_f16x2(v1); v2 = bf16x2_to_f16x2(v2); v3 = bf16x2_to_f16x2(v3);
              asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(b_st + ci * 16), "r"(v0), "r"(v1), "r"(v2), "r"(v3) : "memory");
            }
          }
          if (failed) break;
        }
        fence_async_smem();            // generic-proxy writes must be visible to the tensor core (async proxy)
        __syncwarp();
        if (lane == 0) {
          if (PAIR && crank != 0) pmbar_signal_peer(ppeer_addr(full_a + 8 * s, lrank)); else pmbar_arrive(full_a + 8 * s);
        }
#pragma unroll
        for (int m = 0; m < 2; ++m) { q0[m] = q1[m]; s0[m] = s1[m]; z0[m] = z1[m]; }
      }
    }
    }
    // the block's segments, counted by every warp of this group (the idle four included)
    Seg last_sg = {0, 0, 0, -1};
    int n_seg = 0;
    {
      SegIter sj; sj.init(c, bid, nblk, part);
      Seg sgj;
      while (sj.next(sgj)) { last_sg = sgj; ++n_seg; }
    }
    // the block's last segment: this warp takes a fifth of its chunks beside the epilogue warp of its tensor-memory
    // quadrant (warps 8 + q, 12 + q, 16 + q, 20 + q: chunks 1, 2, 3, 4 of every five)
    if (c.helpers && !failed && n_seg > 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");   // outputs and workspace: after the preceding kernel
      if (!pmbar_wait(last_full, 0, abort_flag, true)) failed = true;
      if (!failed) epilogue_segment(last_sg, n_seg - 1, 1 + (warp - DQ_WARP0) / 4, 5, true);
    }
  } else if (warp >= EPI_WARP0) {
    // ===================================================================== epilogue
    asm volatile("griddepcontrol.wait;" ::: "memory");     // positions, outputs and workspace: after the preceding kernel
    int tcount = 0;
    SegIter si; si.init(c, bid, nblk, part);
    Seg sg;
    for (; !failed && si.next(sg); ++tcount) {
      // The block's last segment: nothing is left to overlap its epilogue with, and the sixteen de-quantiser warps
      // are idle by then, so the four of each tensor-memory quadrant take four fifths of its chunks.
      SegIter peek = si;
      Seg nxt;
      const bool helped = c.helpers && !peek.next(nxt);
      epilogue_segment(sg, tcount, 0, helped ? 5 : 1, false);
    }
  }

  if (failed && lane == 0) atomicExch(c.status, UNIQL_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (PAIR) {                           // (tensor memory of both blocks is given back together, after the last MMA)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
  } else if (warp == 1) {
    tmem_dealloc(tmem_base, 512);
  }
  if (PAIR || c.pair_split) {                   // neither block of a pair leaves while the other may still send to it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// -------------------------------------------------------------------------------- host side
typedef CUresult (*PEncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

PEncodeFn p_encoder() {
  static PEncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qr) == cudaSuccess &&
        qr == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PEncodeFn>(ptr);
    else
      cudaGetLastError();
  });
  return fn;
}

int host_job_tiles(const JobDev& j) {
  if (j.pair == 2) return 0;                                       // its rows ride in the tiles of the job before
  if (j.pair == 1) return (j.k_out + BMW / 2 - 1) / (BMW / 2);
  if (j.rope.enabled) return (j.rope.n_heads * (j.rope.head_keep / 2) + BMW / 2 - 1) / (BMW / 2);
  return (j.k_out + BMW - 1) / BMW;
}

template <typename T, bool CONV, bool HEADS, int PAIR>
int launch_pth(const Params& p, const PrefillCfg& c, int grid, cudaStream_t stream) {
  const size_t smem = 1024 + (size_t)(PAIR ? RING2_BYTES : RING_BYTES) + 512;
  auto kern = prefill_kernel<T, CONV, HEADS, PAIR>;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return UNIQL_ERR_CUDA;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(PTH);
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = opt(kOptPdl) ? 1 : 0;
  if (PAIR || c.pair_split) {
    // clusters of two, only when every pair can be resident at once; else the caller plans without them
    attr[lc.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[lc.numAttrs].val.clusterDim.x = PAIR == 3 ? 2 * c.csplit : 2;
    attr[lc.numAttrs].val.clusterDim.y = 1;
    attr[lc.numAttrs].val.clusterDim.z = 1;
    ++lc.numAttrs;
    // (asked once per kernel instance: the answer depends on the block's resources, which do not change)
    static std::atomic<int> max_clusters{-1};
    int n_clusters = PAIR ? device_sms() / 2 : max_clusters.load();          // (PAIR: the caller has asked pair_capacity())
    if (n_clusters < 0) {
      if (cudaOccupancyMaxActiveClusters(&n_clusters, kern, &lc) != cudaSuccess) { cudaGetLastError(); n_clusters = 0; }
      max_clusters.store(n_clusters);
    }
    if (n_clusters * 2 < grid) return UNIQL_ERR_UNSUPPORTED;
  }
  if (cudaLaunchKernelEx(&lc, kern, p, c) != cudaSuccess) { cudaGetLastError(); return PAIR || c.pair_split ? UNIQL_ERR_UNSUPPORTED : UNIQL_ERR_CUDA; }
  return UNIQL_OK;
}
template <typename T, bool CONV, int PAIR>
int launch_pt(const Params& p, const PrefillCfg& c, int grid, cudaStream_t stream) {
  return c.km_period != 0 ? launch_pth<T, CONV, true, PAIR>(p, c, grid, stream) : launch_pth<T, CONV, false, PAIR>(p, c, grid, stream);
}

// Clusters of `share` block pairs that the device holds at once (asked once per device; the instances need the same
// resources).
constexpr int kMaxShare = 4;
int pair_capacity(int share) {
  static std::atomic<int> n[64][kMaxShare + 1] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = n[dev][share].load(std::memory_order_relaxed);
  if (v != 0) return v - 1;
  auto kern = prefill_kernel<__half, false, false, 3>;
  const size_t smem = 1024 + (size_t)RING2_BYTES + 512;
  const int most = device_sms() / (2 * share);
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3((unsigned)(most * 2 * share));
  lc.blockDim = dim3(PTH);
  lc.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2 * share;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&v, kern, &lc) != cudaSuccess) {
    cudaGetLastError();
    v = 0;
  }
  if (v > most) v = most;
  n[dev][share].store(v + 1);
  return v;
}

}  // namespace

int device_sms() {
  static std::atomic<int> n[64] = {};
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if ((v = n[dev].load(std::memory_order_relaxed)) > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) return 148;
  n[dev].store(v);
  return v;
}

int launch_x_to_f16(const void* x, int ldx, int M, int k_in, void* out, int ldo, cudaStream_t stream) {
  const long units = (long)M * (ldo / 8), most = (long)device_sms() * 8;
  const long blocks = (units + 255) / 256;
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3((unsigned)(blocks < most ? blocks : most));
  lc.blockDim = dim3(256);
  lc.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = opt(kOptPdl) ? 1 : 0;
  if (cudaLaunchKernelEx(&lc, x_to_f16_kernel, reinterpret_cast<const __nv_bfloat16*>(x), ldx, M, k_in, reinterpret_cast<__half*>(out), ldo) !=
      cudaSuccess) {
    cudaGetLastError();
    return UNIQL_ERR_CUDA;
  }
  return UNIQL_OK;
}

int encode_x_map(void* map, const void* x, int k_in, int M, int ldx, int rows, bool bf16) {
  PEncodeFn enc = p_encoder();
  if (!enc) return UNIQL_ERR_CUDA;
  const cuuint64_t dims[2] = {(cuuint64_t)k_in, (cuuint64_t)M};
  const cuuint64_t strides[1] = {(cuuint64_t)ldx * 2};
  const cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)rows};
  const cuuint32_t es[2] = {1, 1};
  const CUresult r = enc(reinterpret_cast<CUtensorMap*>(map), bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                         const_cast<void*>(x), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? UNIQL_OK : UNIQL_ERR_CUDA;
}

// The tensor-core path takes: the leading k_in input channels (the hidden dimension D_h is never pruned,
// D_int is pruned as a leading block: Section 3.4) or one family of per-head kept blocks (the input side of
// o_proj / out_proj: heads on 64-channel boundaries, keep a multiple of 8), any output map, both activation types.
int prefill_supported(const Params& p) {
  if (p.M < 1) return 0;
  if (p.dt != UNIQL_F16 && p.dt != UNIQL_BF16) return 0;
  if (p.imap.n_fam != 1) return 0;
  {
    const Fam& a = p.imap.fam[0];
    if (a.count == 1) {
      if (a.start != 0) return 0;
    } else if ((a.start % BK) != 0 || (a.period % BK) != 0 || (a.keep % 8) != 0) {
      return 0;                    // per-head input maps: heads on k-block boundaries, 16-byte activation boxes
    }
  }
  if ((p.ldx % 8) != 0 || (((uintptr_t)p.x) & 15) != 0) return 0;       // TMA: 16-byte base and row pitch
  if ((p.K % kGroup) != 0) return 0;
  return 1;
}

int launch_prefill(const Params& p, const LaunchCfg& cfg) {
  if (!cfg.workspace || cfg.ws_bytes < decode_workspace_header_bytes()) return UNIQL_ERR_WORKSPACE;   // status word
  // up to 128 rows: the batch kernel (bf16: where the workspace has room for the fp16 copy)
  if (batch_supported(p) &&
      (p.dt != UNIQL_BF16 || (opt(kOptPrefillConvert) != 1 && cfg.ws_bytes >= ((decode_workspace_header_bytes() + 255) & ~(size_t)255) +
                                                                               (size_t)p.M * ((p.k_in + 63) / 64 * 64) * 2 + 256)))
    return launch_batch(p, cfg);
  const int env_grid = opt(kOptPrefillGrid), env_streamk = opt(kOptPrefillStreamk);
  PrefillCfg c;
  memset(&c, 0, sizeof(c));
  c.bn = p.M <= 64 ? 64 : (p.M <= 128 ? 128 : 256);
  int wt = 0;
  for (int j = 0; j < p.n_jobs; ++j) { c.wtile_begin[j] = wt; wt += host_job_tiles(p.job[j]); }
  for (int j = p.n_jobs; j <= kMaxPJobs; ++j) c.wtile_begin[j] = wt;
  if (wt < 1) return UNIQL_ERR_SHAPE;
  {
    const Fam& a = p.imap.fam[0];
    c.km_start = a.start / BK;
    c.km_period = a.count > 1 ? a.period / BK : 0;
    c.km_keep = a.keep;
    c.km_kbh = (a.keep + BK - 1) / BK;
    c.n_kb = c.km_kbh * a.count;
  }
  const uint32_t fmt = 0u;      // both operands fp16 (bf16 activations are converted in shared memory)
  // instruction descriptor: fp32 accumulate, A and B of the activation type, both K-major, N = bn, M = 128
  c.idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(c.bn >> 3) << 17) | ((uint32_t)(BMW >> 4) << 24);
  c.status = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(cfg.workspace) + decode_status_offset());
  const int sms = device_sms();
  // workspace: [header: counters, status][fp16 copy of bf16 activations][stream-K partial tiles]
  size_t ws_used = (decode_workspace_header_bytes() + 255) & ~(size_t)255;
  c.counters = reinterpret_cast<int*>(cfg.workspace);
  // bf16 activations: fp16 copy in the workspace when it fits (else converted tile by tile in the kernel)
  const void* xsrc = p.x;
  int ldxs = p.ldx;
  bool conv_in_kernel = false;
  __half* x16 = nullptr;              // fp16 copy to be written by the pre-pass
  int x16_ld = 0;
  if (p.dt == UNIQL_BF16) {
    // (a row pitch of whole 128-byte lines: a box row that straddles two lines costs a second L2 request, measured
    //  as 1.09 instead of 0.85 us per k-block on the Qwen2.5-7B down projection at 12312 of 18944 input channels)
    int ldo = (p.k_in + 63) / 64 * 64;
    const size_t off = ws_used;
    if (cfg.ws_bytes < off + (size_t)p.M * ldo * 2) ldo = (p.k_in + 7) / 8 * 8;
    const size_t need = off + (size_t)p.M * ldo * 2;
    if (cfg.ws_bytes >= need && opt(kOptPrefillConvert) != 1) {
      x16 = reinterpret_cast<__half*>(reinterpret_cast<unsigned char*>(cfg.workspace) + off);
      x16_ld = ldo;
      xsrc = x16;
      ldxs = ldo;
      ws_used = (need + 255) & ~(size_t)255;
    } else {
      conv_in_kernel = true;
    }
  }
  // The shape of the work: tokens per tile (one accumulator, or both = 512 tokens, so that a de-quantised weight
  // stage serves twice the tokens) and whether the tiles left over after the whole rounds are split along K.
  // Stream-K serves the tiles left over when whole tiles would leave SMs idle in their last round and the slots
  // of the parts fit in the workspace.  It pays when the k-blocks a block no longer waits for outweigh the
  // hand-over.  Measured on B200: a k-block takes about 0.65 us (1.07 us on both accumulators: 1.65 times the time
  // for twice the work); a hand-over at the end of a block (every tile split) 20 - 40 us, growing with the number
  // of blocks on a tile and the tile's width; a hand-over in front of whole tiles is hidden behind them unless a
  // tile has so many parts that reading them back (11 us per part of 256 tokens) outlasts the whole tiles.
  // Both tile widths are costed with these figures and the cheaper one runs: wide tiles win where they still fill
  // the SMs (Qwen2.5-7B gate at M = 512..4096: 17-22 % faster), narrow ones where wide tiles would leave most SMs
  // without a tile (q / o projections at M = 512) or push a few left-over tiles into a round of their own.
  int g1 = sms;
  if (env_grid >= 1 && env_grid <= sms) g1 = env_grid;            // tests: odd splits on small problems
  bool any_rope = false;
  for (int j = 0; j < p.n_jobs; ++j) any_rope = any_rope || p.job[j].rope.enabled != 0;
  // Block pairs (cta_group::2): tiles of 256 rows, a cluster of two blocks where the other plans have one block.
  const int opt_pair = opt(kOptPrefillPair);
  int wt2 = 0, gp = 0;
  // (options that steer the one-block plans, forced by tests, keep the pairs out unless they are forced too)
  const bool pair_auto = opt_pair < 0 && env_grid == 0 && (env_streamk <= 0 || env_streamk > 10) && opt(kOptPrefillDual) <= 0;
  if (c.bn == MAXBN && !conv_in_kernel && (pair_auto || opt_pair >= 1)) {
    for (int j = 0; j < p.n_jobs; ++j) wt2 += (host_job_tiles(p.job[j]) + 1) / 2;
    gp = pair_capacity(1);
    if (env_grid >= 1 && env_grid < gp) gp = env_grid;
  }
  struct Plan { int nh, ttiles, tiles, left, g; int share; bool streamk, atomic, halves, pair, cg2; size_t sums; double us; };
  static std::atomic<bool> pair_refused{false};       // a cluster launch was refused once: planned without from then on
  auto plan_for = [&](int nh, bool cg2) {
    Plan q;
    q.nh = nh;
    q.cg2 = cg2;
    q.share = 1;
    const int g2 = cg2 ? gp : g1;
    q.g = g2;
    const int ntok = c.bn * nh;
    q.ttiles = (p.M + ntok - 1) / ntok;
    const long tiles = (long)(cg2 ? wt2 : wt) * q.ttiles;
    q.tiles = tiles <= (1 << 24) ? (int)tiles : (1 << 24);
    q.left = q.tiles % g2;
    // (pairs: fitted over 7 layer shapes at M = 160 .. 2048, every form forced in turn; worst choice 6 % off the best)
    const double kcost = cg2 ? (nh == 2 ? 0.60 : 0.365) : (nh == 2 ? 1.07 : 0.65);
    const double wide = ntok / 256.0;
    // blocks on the split tile with the most of them: its finishing block reads that many slots back
    const long units = (long)q.left * c.n_kb;
    const long bt = units < g2 ? units : g2;
    const double pmax = q.left ? (double)((bt + q.left - 1) / q.left + 1) : 0.0;
    double hand_over;
    q.atomic = false;
    // a k-block of a one-box tile by the number of busy SMs (0.45 us with 28 of them, 0.61 us with all)
    auto kb1 = [&](int busy) { return cg2 ? 0.365 : 0.42 + 0.19 * (busy < g2 ? busy : g2) / g2; };
    if (q.tiles < g2) {
      // every tile is split and every block ends on a split tile: the hand-over is shared with the de-quantiser warps
      // (one-box tiles, measured at M = 64 .. 512 on seven layer shapes: 5 us per 64 tokens of the tile)
      // (64-token tiles, measured on four shapes with 3 to 52 tiles: 0.9 us for every part that the finishing block adds; a
      //  contraction of 4744 channels and three tiles took 47 us split over all SMs and 24 us over pairs of blocks)
      hand_over = nh == 2 ? 24.0 + 2.0 * pmax * wide : c.bn == 64 ? 5.0 + 0.9 * pmax : (14.0 + pmax) * wide;
    } else {
      // The split tiles come first and whole tiles follow.  Reading a tile's slots back takes the four epilogue
      // warps 11 us per slot of 256 tokens, and a split tile in front of whole tiles has three or more parts: that
      // outlasts the first whole tile, whose epilogue then waits (measured 37 us lost on the Qwen2.5-7B gate at keep
      // 0.65, M = 2048, three parts).  Here the parts are added into one sum per tile instead (reductions done in
      // L2): 14 us per 256 tokens, measured, most of it hidden behind the whole tiles.
      q.atomic = true;
      hand_over = 14.0 * wide;
    }
    // (a tile with the rotary epilogue costs its finishing block about twice as long: measured on the Qwen2.5-7B
    //  q|k launch at M = 2048, head dim 84, where the split forms lost 8 us against this estimate without it)
    if (any_rope) hand_over += 12.0 * wide;
    if (env_streamk == 1) q.atomic = false;                            // tests: the form of the hand-over forced
    if (env_streamk == 2) q.atomic = true;
    // (a split is taken where it is estimated 5 % ahead: its hand-over varies more than a whole tile's time)
    double us_split = 1.05 * ((double)q.tiles / g2 * c.n_kb * ((nh == 1 && q.tiles < g2) ? kb1(g2) : kcost) + hand_over);
    // Whole tiles.  On both accumulators a k-block takes 0.84 us when every SM runs one and less when some have no
    // tile (0.79 us with 28 busy SMs: they share the activation traffic out of L2), and between two tiles of a block
    // the MMAs wait 7 - 10 us for the epilogue to drain the accumulators (in-kernel time stamps, Qwen2.5-7B gate at
    // M = 2048); fitted over 48 launches (16 shapes at M = 512, 1024, 2048, every width and hand-over forced in turn).
    const int rounds = (q.tiles + g2 - 1) / g2;
    double us_whole = (double)rounds * c.n_kb * kcost;
    if (nh == 1 && q.tiles <= g2) us_whole = c.n_kb * kb1(q.tiles);
    if (nh == 2 && cg2)
      us_whole = (double)rounds * (c.n_kb * 0.60 + 9.0);
    else if (nh == 2)
      us_whole = (double)(q.tiles / g2) * c.n_kb * 0.96 + (q.left ? c.n_kb * (0.90 + 0.06 * q.left / g2) : 0.0) + 10.0 * (rounds - 1);
    if (cg2 && nh == 1) { us_whole += 5.5; us_split += 5.5; }                  // start and last epilogue
    // one fp32 slot per (left-over tile, block) piece, or one sum per left-over tile
    q.sums = (size_t)(q.atomic ? q.left : q.left + g2) * ntok * BMW * 4 * (cg2 ? 2 : 1);
    // (pairs: only where forced -- with a k-block at 0.36 us no split of the left-over tiles measured ahead of whole tiles)
    const bool want = env_streamk >= 0 ? (env_streamk >= 1 && env_streamk < 10) : (!cg2 && q.left != 0 && us_split < us_whole);
    q.streamk = want && q.left != 0 && cfg.ws_bytes >= ws_used + q.sums && q.tiles <= (1 << 15);
    q.us = q.streamk ? us_split : us_whole;
    // Tiles of two boxes left over after the whole rounds, when they are few: each runs as two half tiles (one box,
    // 256 tokens) on two blocks, a block's last segment -- no hand-over, and the round takes a one-box tile's time
    // (0.45 - 0.6 us per k-block by the number of busy SMs) instead of a two-box tile's on a few SMs.
    q.halves = false;
    if (nh == 2 && q.left != 0 && 2 * q.left <= g2 && q.tiles > g2 && !conv_in_kernel && env_streamk < 1 && opt(kOptPrefillDual) != 2) {
      const double us_halves = cg2 ? (double)(q.tiles / g2) * (c.n_kb * 0.60 + 9.0) + c.n_kb * 0.365 + 5.5
                                   : (double)(q.tiles / g2) * (c.n_kb * 0.96 + 10.0) + c.n_kb * (0.45 + 0.15 * 2 * q.left / g2);
      if (us_halves < q.us || opt(kOptPrefillDual) == 3) { q.halves = true; q.streamk = false; q.us = us_halves; }
    }
    // Few tiles of one box (at most one for every two SMs): a cluster of two blocks per tile, half of the
    // contraction each, the second block's sums handed over through the first one's shared memory (about 5 us
    // against the 11 - 28 us of a hand-over through the workspace; a k-block takes the same 0.5 - 0.65 us).
    q.pair = false;
    if (nh == 1 && !cg2 && 2 * q.tiles <= sms && c.n_kb >= 4 && env_grid == 0 && !pair_refused.load() && (env_streamk < 0 || env_streamk == 3)) {
      const double us_pair = (double)(c.n_kb - c.n_kb / 2) * kb1(2 * q.tiles) + 1.0 + 4.5 * wide + (any_rope ? 3.0 : 0.0);
      // (against a split over all SMs it has to be 10 % ahead: with long contractions the two come out level and
      //  the split measured ahead, Qwen2.5-7B down projection at M = 512)
      if (us_pair * (q.streamk ? 1.10 : 1.0) < q.us || env_streamk == 3) { q.pair = true; q.streamk = false; q.us = us_pair; }
    }
    // Few tiles of a pair: a cluster of two to four pairs per tile, a part of the contraction each (0.34 us per k-block, 7 us
    // for the exchange beside what a whole tile's start and end take; 4096 x 4096 at M = 256: 25.7 -> 19.0 us).
    if (cg2 && nh == 1 && env_streamk != 0 && c.n_kb >= 8) {
      for (int k = 2; k <= kMaxShare; ++k) {
        const int cap = env_grid >= 1 ? env_grid / k : pair_capacity(k);
        const bool fits = q.tiles <= cap && cfg.ws_bytes >= ws_used + (size_t)q.tiles * k * 2 * MAXBN * BMW * 4;
        const double us = (c.n_kb + k - 1) / k * 0.34 + 12.5;
        if (fits && (env_streamk == 10 + k || (env_streamk < 0 && us < q.us))) { q.share = k; q.streamk = false; q.us = us; }
      }
    }
    return q;
  };
  Plan pl = plan_for(1, false);
  {
    // -1: by cost, 0: never, 1: wherever M > 256; tests: 2 the same without half tiles, 3 with them wherever they fit
    const int dual = opt(kOptPrefillDual);
    if (p.M > MAXBN && dual != 0) {
      const Plan p2 = plan_for(2, false);
      if (dual >= 1 || p2.us < pl.us) pl = p2;
    }
    if (gp >= 1 && env_streamk != 3) {
      // (above 128 rows pairs measured ahead of every one-block plan on all 20 layer shapes tried, 10 - 40 %)
      if (opt_pair < 0) pl.us = 1e30;
      // (tests: 1 / 2 force pairs with one or two boxes per tile)
      for (int nh = 1; nh <= 2; ++nh) {
        if ((nh == 2 && (p.M <= MAXBN || dual == 0)) || (nh == 1 && p.M > MAXBN && dual >= 1)) continue;
        const Plan q = plan_for(nh, true);
        if (opt_pair == nh || (opt_pair < 0 && (q.us < pl.us))) pl = q;
      }
    }
  }
  c.helpers = opt(kOptPrefillHelpers) != 0;
  c.nh = pl.nh;
  c.halves = pl.halves ? 1 : 0;
  c.pair_split = pl.pair ? 1 : 0;
  c.csplit = pl.share;
  c.n_ttiles = pl.ttiles;
  c.n_tiles = pl.tiles;
  if (pl.cg2) {
    int w = 0;
    for (int j = 0; j < p.n_jobs; ++j) { c.wtile_begin[j] = w; w += (host_job_tiles(p.job[j]) + 1) / 2; }
    for (int j = p.n_jobs; j <= kMaxPJobs; ++j) c.wtile_begin[j] = w;
    c.idesc = (c.idesc & ~(0x1fu << 24)) | ((uint32_t)((2 * BMW) >> 4) << 24);       // 256 rows
  }
  if ((long)wt * pl.ttiles > (1 << 24)) return UNIQL_ERR_SHAPE;
  int grid = c.n_tiles < pl.g ? c.n_tiles : pl.g;
  if (pl.pair) grid = 2 * c.n_tiles;
  {
    if (pl.streamk) {
      c.streamk = 1;
      c.sk_atomic = pl.atomic ? 1 : 0;
      c.partials = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(cfg.workspace) + ws_used);
      grid = pl.g;
      // (slots are written before they are read; sums start at zero)
      if (pl.atomic && cudaMemsetAsync(c.partials, 0, pl.sums, cfg.stream) != cudaSuccess) return UNIQL_ERR_CUDA;
    }
    if (x16) {
      const int rc = launch_x_to_f16(p.x, p.ldx, p.M, p.k_in, x16, x16_ld, cfg.stream);
      if (rc != UNIQL_OK) return rc;
    }
  }
  if (pl.cg2) grid *= 2 * pl.share;
  if (pl.share > 1) c.partials = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(cfg.workspace) + ws_used);
  int rc = encode_x_map(&c.xmap, xsrc, p.k_in, p.M, ldxs, pl.cg2 ? c.bn / 2 : c.bn, conv_in_kernel);
  if (rc != UNIQL_OK) return rc;
  if (p.dt == UNIQL_BF16)
    rc = conv_in_kernel ? launch_pt<__nv_bfloat16, true, 0>(p, c, grid, cfg.stream)
         : !pl.cg2      ? launch_pt<__nv_bfloat16, false, 0>(p, c, grid, cfg.stream)
         : c.csplit > 1 ? launch_pt<__nv_bfloat16, false, 3>(p, c, grid, cfg.stream)
         : c.nh == 1    ? launch_pt<__nv_bfloat16, false, 1>(p, c, grid, cfg.stream)
                        : launch_pt<__nv_bfloat16, false, 2>(p, c, grid, cfg.stream);
  else
    rc = !pl.cg2        ? launch_pt<__half, false, 0>(p, c, grid, cfg.stream)
         : c.csplit > 1 ? launch_pt<__half, false, 3>(p, c, grid, cfg.stream)
         : c.nh == 1    ? launch_pt<__half, false, 1>(p, c, grid, cfg.stream)
                        : launch_pt<__half, false, 2>(p, c, grid, cfg.stream);
  if (rc == UNIQL_ERR_UNSUPPORTED && c.pair_split) {
    // the pairs cannot all be resident (or clusters cannot be launched here): planned again without them
    pair_refused.store(true);
    return launch_prefill(p, cfg);
  }
  return rc;
}

size_t prefill_workspace_bytes(int M, int K) {
  // status word and counters (shared header) + room for the fp16 copy of bf16 activations + the slots of tiles
  // split along K: fewer than two per SM, of 256 tokens, or of 512 where tiles take both accumulators
  return ((decode_workspace_header_bytes() + 255) & ~(size_t)255) + (size_t)M * ((K + 63) / 64 * 64) * 2 + 256 +
         (size_t)2 * device_sms() * (M > MAXBN ? 2 * MAXBN : MAXBN) * BMW * 4;
}

}  // namespace uniql
