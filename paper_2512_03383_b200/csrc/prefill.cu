// Block pairs (clusters of two blocks on tiles of 256 weight rows with cta_group::2 MMAs) and the planner of the tensor-core
// kernels described in prefill.cuh.
//
// Work split of the pairs (chosen by the launcher from a cost model): one or two boxes of 256 tokens per tile, whole tiles
// round-robin; left-over tiles of two boxes as half tiles on twice the pairs; launches with few tiles as clusters of two to
// four pairs per tile, a part of the contraction each.  Measured against one block per tile: Qwen2.5-7B gate at M = 2048
// 227 -> 193 us (1.44 PFLOP/s), 4096 x 4096 at M = 256 27 -> 19 us.
#include <string.h>

#include <atomic>
#include <mutex>

#include "prefill.cuh"

namespace uniql {
namespace {

// stages of weights and the k-block's half boxes (each block holds half of the tokens), one or two of them
constexpr int PSTAGES1 = 6, PSTAGES2 = 4;
constexpr int RING_BYTES = PSTAGES2 * (A_BYTES + B_BYTES);
static_assert(PSTAGES1 * (A_BYTES + B_BYTES / 2) == RING_BYTES, "both widths use the same shared memory");

// Work of a pair as a sequence of segments: whole tiles t = b, b + grid, ..., the ones left over after the whole rounds as
// halves, or a part of one tile's k-blocks (part >= 0: which of the pairs that share the tile this one is).
struct SegIter {
  int t, t_end, n_kb, step, half_tile, half, part_tile, part_kb0, part_kb1;
  __device__ inline void init(const PrefillCfg& c, int b, int grid, int part) {
    n_kb = c.n_kb; step = grid; t = b; t_end = c.n_tiles;
    half_tile = part_tile = -1;
    half = 0;
    if (part >= 0) {
      t_end = 0;
      part_tile = b;
      part_kb0 = n_kb * part / c.csplit; part_kb1 = n_kb * (part + 1) / c.csplit;
    } else if (c.halves) {
      // whole rounds of whole tiles, then tile (rounds * grid + b / 2) as two halves on pairs b and b + 1
      t_end = (c.n_tiles / grid) * grid;
      if (t_end + b / 2 < c.n_tiles) { half_tile = t_end + b / 2; half = b & 1; }
    }
  }
  __device__ inline bool next(Seg& sg) {
    if (t < t_end) {
      sg.tile = t; sg.kb0 = 0; sg.kb1 = n_kb; sg.half = -1;
      t += step;
      return true;
    }
    if (part_tile >= 0) {
      sg.tile = part_tile; sg.kb0 = part_kb0; sg.kb1 = part_kb1; sg.half = -1;
      part_tile = -1;
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

// bf16 activations -> fp16 copy in the workspace, once per call (every weight tile re-reads the tile of
// activations, so converting there would repeat the work once per 128 weight rows).
// Few blocks of 256 threads: the next launch's blocks come in beside these, and with a few rows cut into four times as many blocks
// they came in unevenly (Mamba2-2.7B mixer at 16 rows 22.4 -> 28.3 us, Bamba-v2-9B 43.9 -> 44.8; at 1024 rows 78.0 -> 82.0, Qwen2.5-7B layer at
// 256 rows, keep 0.65, 117.8 -> 124.1 us; ahead only for Llama-3-8B at 112 to 128 rows, keep 0.65, 100.5 -> 96.2 us).
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

// T: activation / output type.  HEADS: the input map is a family of per-head blocks (else a leading block).
// Clusters of two blocks work on tiles of 256 weight rows with cta_group::2 MMAs.  Each block de-quantises 128 rows into its own
// shared memory and fetches half of the tokens' boxes; the first block's MMA warp issues for both.  A block's shared memory then
// takes in 16 instead of 32 KB of activations per 256 tokens and k-block, which with one block per tile was what L2 could not
// deliver and the shared-memory port could not take beside the operand reads.  PAIR = 1 / 2: one or two boxes of 256 tokens per
// tile; 3: one box, and the pairs of a cluster share a tile (an instance of its own: inside 1 its registers cost every launch
// 3 - 10 %).
template <typename T, bool HEADS, int PAIR>
__global__ void __launch_bounds__(PTH, 1) pair_kernel(const __grid_constant__ Params p,
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
  constexpr int NA = ONE ? PSTAGES1 : PSTAGES2;             // weight stages, each with the k-block's half boxes
  constexpr int NB_BYTES = B_BYTES / 2;
  // this pair's number and their count (3: the cluster's), and this pair's part of a shared tile
  const int n_share = PAIR == 3 ? c.csplit : 1, per = 2 * n_share;
  const int bid = (int)blockIdx.x / per, nblk = (int)gridDim.x / per;
  const uint32_t rank = pcluster_rank();
  const uint32_t crank = PAIR == 3 ? rank & 1u : rank, lrank = PAIR == 3 ? rank & ~1u : 0u;   // block of the pair, rank of the pair's first block
  const int part = PAIR == 3 ? (int)(rank >> 1) : -1;
  constexpr int B_RING = NA * A_BYTES;                      // the activation boxes follow the weight stages
  constexpr int TEAM_WARPS = ONE ? DQ_WARPS : DQ_TEAM_WARPS;
  const uint32_t bars = sbase + RING_BYTES;
  // (a stage's weights and its half boxes share one pair of barriers -- the MMA warp's loop is one chain of dependent
  //  instructions, 890 cycles per k-block of one box with two waits and two commits where the MMAs take 512)
  const uint32_t full_a = bars, empty_a = bars + 8 * NA;
  const uint32_t acc_full = bars + 16 * NA, acc_empty = acc_full + 16;
  const uint32_t last_full = acc_full + 32;        // the MMAs of the block's last segment are complete (one phase only)
  const uint32_t xq = acc_full + 40;               // pairs that share a tile: the others' sums have arrived, per quadrant
  unsigned char* misc = smem + RING_BYTES + 16 * NA + 72;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  if (tid == 0) {
    for (int s = 0; s < NA; ++s) {
      pmbar_init(full_a + 8 * s, 2 * TEAM_WARPS + 1);
      pmbar_init(empty_a + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) { pmbar_init(acc_full + 8 * b, 1); pmbar_init(acc_empty + 8 * b, 8); }
    pmbar_init(last_full, 1);
    if (PAIR == 3)
      for (int b = 0; b < 4; ++b) pmbar_init(xq + 8 * b, max(1, (n_share - 1) * (c.helpers ? 5 : 1)));
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the whole tensor memory of the SM: two accumulators of 256 columns
  if (warp == 1) tmem_alloc_pair((uint32_t)__cvta_generic_to_shared(const_cast<uint32_t*>(tmem_slot)), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the other blocks' barriers exist before anything is sent to them
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  // 128-row tile of its job that this block holds (tiles are counted in pairs)
  auto local_tile = [&](int wt, int jn) { return 2 * (wt - c.wtile_begin[jn]) + (int)crank; };
  auto job_of_wt = [&](int wt) { int j = 0; while (j + 1 < p.n_jobs && wt >= c.wtile_begin[j + 1]) ++j; return j; };
  bool failed = false;

  // ---- the epilogue of one segment, for the warp that calls it: accumulator -> bias, rotary embedding or gated
  //      product, rounding, store.  A warp reaches the tensor-memory lanes 32 (warp % 4) .. + 31 (a lane is a tile
  //      row); it takes the chunks ch0, ch0 + chs, ... of 32 tokens.  chs == 1: the epilogue warp on its own (it
  //      also hands the accumulators back).
  const int q = warp & 3;                          // TMEM lanes 32q .. 32q+31
  const int etid = 32 * q + lane;                  // tile row handled in the store phase
  auto epilogue_segment = [&](const Seg& sg, int tcount, int ch0, int chs, bool helper) {
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
      // helper: a de-quantiser warp on the block's last segment, which follows the barrier of that segment alone.  It waits here and not in
      // front of the call: the row's index arithmetic above, and what loads a bias and a rotation need, run beside the last MMAs
      // (passes back to back, in turn with the wait in front: Llama-3-8B layer at 512 rows, keep 0.75, 194.1 -> 192.8 us, Mamba2-2.7B
      // mixer at 1024 rows, keep 0.75, 76.7 -> 76.1, Qwen2.5-7B layer at 677 rows, keep 0.65, 254.6 -> 253.6, where the runs of one
      // side differ by 0.1 - 0.6 %).  Left at once where a wait expires: with one test of `failed` behind both waits whole tiles spill.
      if (helper) {
        if (!pmbar_poll_warp(last_full, 0, abort_flag, true)) { failed = true; return; }
      } else {
        for (int h = h_lo; h < h_hi; ++h)
          if (!pmbar_poll_warp(acc_full + 8 * (acc0 + h), au & 1, abort_flag)) { failed = true; return; }
      }
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
          pmbar_signal_peer(ppeer_addr(eb, lrank));
        }
      };
      if constexpr (PAIR == 3) {
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
        if (!pmbar_wait_cluster_warp(xq + 8 * q, 0, abort_flag)) { failed = true; return; }
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
      } else {
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
      }
  };

  if (warp == 0) {
    // ===================================================================== activations by TMA
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
  } else if (warp == 1) {
    // ===================================================================== MMA issue
    // (the whole warp walks the loop, so that stage indexes, parities and descriptors are warp-uniform; one elected
    //  lane issues)
    if (crank == 0) {
      const unsigned short pair_mask = (unsigned short)(3u << lrank);
      int s = 0; uint32_t par = 0; int tcount = 0;         // weight stage and its parity
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
          if (kb == sg.kb0 && au >= 1 && !pmbar_wait_warp(acc_empty + 8 * acc0, (au - 1) & 1, abort_flag)) { failed = true; break; }
          tc_fence_after();
          if (elect_one()) {
            umma_kblock<true>(tmem_base + (uint32_t)(acc0 * MAXBN), adesc, smem_desc_sw128(sbase + B_RING + s * NB_BYTES), c.idesc, kb > sg.kb0 ? 1u : 0u);
            umma_commit_pair(empty_a + 8 * s, pair_mask);        // the stage is free once these MMAs have read it
          }
          __syncwarp();
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
          for (int h = h_lo; h < h_hi; ++h) umma_commit_pair(acc_full + 8 * (acc0 + h), pair_mask);
          if (last) umma_commit_pair(last_full, pair_mask);
        }
        __syncwarp();
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
        if (it >= NA && !pmbar_wait_warp(empty_a + 8 * s, (use - 1) & 1, abort_flag)) { failed = true; break; }
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
        fence_async_smem();            // generic-proxy writes must be visible to the tensor core (async proxy)
        __syncwarp();
        if (lane == 0) {
          if (crank != 0) pmbar_signal_peer(ppeer_addr(full_a + 8 * s, lrank)); else pmbar_arrive(full_a + 8 * s);
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
      epilogue_segment(last_sg, n_seg - 1, 1 + (warp - DQ_WARP0) / 4, 5, true);
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
  // (tensor memory of both blocks is given back together, after the last MMA; no block leaves while another may still send to it)
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
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

// UNIQL_ERR_UNSUPPORTED: the clusters were refused, and nothing was launched.
template <typename T, bool HEADS, int PAIR>
int launch_as(const Params& p, const PrefillCfg& c, int grid, cudaStream_t stream) {
  const size_t smem = 1024 + (size_t)RING_BYTES + 512;
  auto kern = pair_kernel<T, HEADS, PAIR>;
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
  attr[lc.numAttrs].id = cudaLaunchAttributeClusterDimension;
  attr[lc.numAttrs].val.clusterDim.x = PAIR == 3 ? 2 * c.csplit : 2;
  attr[lc.numAttrs].val.clusterDim.y = 1;
  attr[lc.numAttrs].val.clusterDim.z = 1;
  ++lc.numAttrs;
  if (opt(kOptPrefillPair) == 3) return UNIQL_ERR_UNSUPPORTED;             // tests
  if (cudaLaunchKernelEx(&lc, kern, p, c) != cudaSuccess) { cudaGetLastError(); return UNIQL_ERR_UNSUPPORTED; }
  return UNIQL_OK;
}
template <typename T, int PAIR>
int launch_pair(const Params& p, const PrefillCfg& c, int grid, cudaStream_t stream) {
  return c.km_period != 0 ? launch_as<T, true, PAIR>(p, c, grid, stream) : launch_as<T, false, PAIR>(p, c, grid, stream);
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
  auto kern = pair_kernel<__half, false, 3>;
  const size_t smem = 1024 + (size_t)RING_BYTES + 512;
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

namespace {

// clusters: false after a launch as clusters was refused
int launch_planned(const Params& p, const LaunchCfg& cfg, bool clusters) {
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
  if (p.dt == UNIQL_BF16 && !p.x_f16) {
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
  const int opt_pair = opt(kOptPrefillPair) == 3 ? -1 : opt(kOptPrefillPair);
  int wt2 = 0, gp = 0;
  // (options that steer the one-block plans, forced by tests, keep the pairs out unless they are forced too)
  const bool pair_auto = opt_pair < 0 && env_grid == 0 && (env_streamk <= 0 || env_streamk > 10) && opt(kOptPrefillDual) <= 0;
  if (clusters && c.bn == MAXBN && !conv_in_kernel && (pair_auto || opt_pair >= 1)) {
    for (int j = 0; j < p.n_jobs; ++j) wt2 += (host_job_tiles(p.job[j]) + 1) / 2;
    gp = pair_capacity(1);
    if (env_grid >= 1 && env_grid < gp) gp = env_grid;
  }
  struct Plan { int nh, ttiles, tiles, left, g; int share; bool streamk, atomic, halves, pair, cg2; size_t sums; double us; };
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
    // a k-block of a one-box tile by the number of busy SMs (256 tokens: 0.45 us with 28 of them, 0.61 us with all)
    auto busy_part = [&](int busy) { return (double)(busy < g2 ? busy : g2) / g2; };
    auto kb1 = [&](int busy) { return c.bn < MAXBN ? 0.435 + 0.06 * busy_part(busy) : 0.42 + 0.19 * busy_part(busy); };
    // Up to 128 rows, fewer tiles than SMs: the lines for whole tiles, pairs of blocks and tiles split over all SMs are fitted to
    // 60 shapes with an odd number of groups (2 to 112 tiles, 18 to 222 k-blocks, half of them above 64 rows), every form forced in
    // turn.  On these and on 60 others the plans they choose are within 3 % of the best of the three, but for three within 8 %.
    const bool small = c.bn < MAXBN && q.tiles < g2;
    if (q.tiles < g2) {
      // every tile is split and every block ends on a split tile: the hand-over is shared with the de-quantiser warps
      // (one-box tiles, measured at M = 64 .. 512 on seven layer shapes: 5 us per 64 tokens of the tile)
      // (64-token tiles: 0.3 us for every part that the finishing block adds; 568 x 7296 at 26 rows, five tiles in 30 parts,
      //  takes 22 us split over all SMs and 32 us over pairs of blocks.  128-token tiles: 0.7 us; where a block's range crosses
      //  from one tile into the next its first part is handed over by the epilogue warps alone, and with a few k-blocks per
      //  block they can be the last to arrive, and read the tile back alone: 640 x 7296 at 93 rows, 3.9 k-blocks per block, takes
      //  75 us, 568 x 12416 at 125 rows, 6.6 of them, 36 us)
      const double per_block = bt ? (double)units / (double)bt : 0.0;
      const bool crosses = q.left != 0 && bt % q.left != 0 && per_block > 1.5;
      const double hand128 = !crosses ? 8.0 + 0.75 * pmax : per_block < 6.0 ? 10.0 + 2.0 * pmax : per_block < 20.0 ? 8.0 + pmax : 8.0 + 0.9 * pmax;
      hand_over = nh == 2 ? 24.0 + 2.0 * pmax * wide : c.bn == 64 ? 10.3 + 0.3 * pmax : c.bn == 128 ? hand128 : (14.0 + pmax) * wide;
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
    const double us_split = 1.05 * ((double)q.tiles / g2 * c.n_kb * ((nh == 1 && q.tiles < g2) ? kb1(g2) : kcost) + hand_over);
    // Whole tiles.  On both accumulators a k-block takes 0.84 us when every SM runs one and less when some have no
    // tile (0.79 us with 28 busy SMs: they share the activation traffic out of L2), and between two tiles of a block
    // the MMAs wait 7 - 10 us for the epilogue to drain the accumulators (in-kernel time stamps, Qwen2.5-7B gate at
    // M = 2048); fitted over 48 launches (16 shapes at M = 512, 1024, 2048, every width and hand-over forced in turn).
    const int rounds = (q.tiles + g2 - 1) / g2;
    double us_whole = (double)rounds * c.n_kb * kcost;
    if (nh == 1 && !cg2 && q.tiles <= g2) us_whole = c.n_kb * kb1(q.tiles) + (small ? 3.0 : 0.0);
    if (nh == 2 && cg2)
      us_whole = (double)rounds * (c.n_kb * 0.60 + 9.0);
    else if (nh == 2)
      us_whole = (double)(q.tiles / g2) * c.n_kb * 0.96 + (q.left ? c.n_kb * (0.90 + 0.06 * q.left / g2) : 0.0) + 10.0 * (rounds - 1);
    if (cg2 && nh == 1) us_whole += 5.5;                                       // start and last epilogue
    // one fp32 slot per (left-over tile, block) piece, or one sum per left-over tile
    q.sums = (size_t)(q.atomic ? q.left : q.left + g2) * ntok * BMW * 4;
    // (pairs: never -- with a k-block at 0.36 us no split of the left-over tiles measured ahead of whole tiles)
    const bool want = env_streamk >= 0 ? (env_streamk >= 1 && env_streamk < 10) : us_split < us_whole;
    q.streamk = want && !cg2 && q.left != 0 && cfg.ws_bytes >= ws_used + q.sums && q.tiles <= (1 << 15);
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
    if (nh == 1 && !cg2 && 2 * q.tiles <= sms && c.n_kb >= 4 && env_grid == 0 && clusters && (env_streamk < 0 || env_streamk == 3)) {
      const double ends = small ? 3.3 + 6.5 * wide + 2.6 * busy_part(2 * q.tiles) * busy_part(2 * q.tiles) : 1.0 + 4.5 * wide;
      const double us_pair = (double)(c.n_kb - c.n_kb / 2) * kb1(2 * q.tiles) + ends + (any_rope ? 3.0 : 0.0);
      // (256 tokens: against a split over all SMs it has to be 10 % ahead: with long contractions the two come out level and
      //  the split measured ahead, Qwen2.5-7B down projection at M = 512)
      if (us_pair * (q.streamk && !small ? 1.10 : 1.0) < q.us || env_streamk == 3) { q.pair = true; q.streamk = false; q.us = us_pair; }
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
  if (!pl.cg2)
    rc = launch_one_block(p, c, grid, conv_in_kernel, cfg.stream);
  else if (p.dt == UNIQL_BF16)
    rc = c.csplit > 1 ? launch_pair<__nv_bfloat16, 3>(p, c, grid, cfg.stream)
         : c.nh == 1  ? launch_pair<__nv_bfloat16, 1>(p, c, grid, cfg.stream)
                      : launch_pair<__nv_bfloat16, 2>(p, c, grid, cfg.stream);
  else
    rc = c.csplit > 1 ? launch_pair<__half, 3>(p, c, grid, cfg.stream)
         : c.nh == 1  ? launch_pair<__half, 1>(p, c, grid, cfg.stream)
                      : launch_pair<__half, 2>(p, c, grid, cfg.stream);
  // (the clusters cannot all be resident, or cannot be launched here: planned again without them)
  return rc == UNIQL_ERR_UNSUPPORTED && clusters ? launch_planned(p, cfg, false) : rc;
}

}  // namespace

int launch_prefill(const Params& p, const LaunchCfg& cfg) {
  if (!cfg.workspace || cfg.ws_bytes < decode_workspace_header_bytes()) return UNIQL_ERR_WORKSPACE;   // status word
  // up to 128 rows: the batch kernel (bf16: where the workspace has room for the fp16 copy)
  if (batch_supported(p) &&
      (p.dt != UNIQL_BF16 || p.x_f16 || (opt(kOptPrefillConvert) != 1 && cfg.ws_bytes >= batch_workspace_min(true, p.M, p.k_in))))
    return launch_batch(p, cfg);
  return launch_planned(p, cfg, true);
}

size_t prefill_workspace_bytes(int M, int K) {
  // status word and counters (shared header) + room for the fp16 copy of bf16 activations + the slots of tiles
  // split along K: fewer than two per SM, of 256 tokens, or of 512 where tiles take both accumulators
  return ((decode_workspace_header_bytes() + 255) & ~(size_t)255) + (size_t)M * ((K + 63) / 64 * 64) * 2 + 256 +
         (size_t)2 * device_sms() * (M > MAXBN ? 2 * MAXBN : MAXBN) * BMW * 4;
}

}  // namespace uniql
