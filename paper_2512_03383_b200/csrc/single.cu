// One-block kernel of the pruned 4-bit linear layer, sm_100a: tiles of 128 weight rows on one block each, for what neither the
// decode nor the batch kernel nor the block pairs of prefill.cu take: up to 128 rows with an odd number of 128-channel groups
// or other maps than the batch kernel's, bf16 activations that have no room for an fp16 copy, and devices that refuse clusters.
// Roles, layouts and arithmetic as prefill.cuh describes them.
// What bounds it at those sizes: a k-block takes 0.44 - 0.49 us whatever its number of tokens (de-quantise, hand-shake, MMAs:
// 4 KB of codes per SM and k-block, 1.3 TB/s over the device), and a launch 3 us before and behind them.  4096 x 4224 at 17 rows
// 18.5 us, 10192 x 10624 at two rows 52 us where its bytes take 9.
//
// Work split (chosen by the launcher from a cost model): whole tiles round-robin; tiles left over after the whole
// rounds split along K over all blocks (stream-K: parts handed over through slots in the workspace, or added into
// one sum per tile) or, for tiles of two boxes, run as half tiles on twice the blocks; launches with few tiles as
// clusters of two blocks per tile, the second block's sums written into the first one's idle rings.
#include <string.h>

#include <atomic>

#include "prefill.cuh"

namespace uniql {
namespace {

constexpr int PSTAGES = 4;                   // ring of de-quantised weight stages (one k-block each)
constexpr int BSLOTS = 4;                    // ring of activation boxes (one k-block of MAXBN tokens each)
constexpr int B_RING = PSTAGES * A_BYTES;    // the boxes follow the weight stages
constexpr int RING_BYTES = PSTAGES * A_BYTES + BSLOTS * B_BYTES;

// Work of a block as a sequence of segments (tile, k-blocks [kb0, kb1)): whole tiles t = b, b + grid, ...
// With stream-K only for as many rounds as fill every block; the k-blocks of the tiles left over are
// cut into equal contiguous ranges, one per block, so that every SM stays busy however few tiles remain.
// A block runs its range of the split tiles FIRST: handing over the partial tile and finishing the split
// tiles then overlap the main loop of the whole tiles that follow instead of standing at the kernel's end.  Blocks stay in step along k (few distinct k offsets are alive at a time, which keeps the
// activation slices in L2).  Every block adds its fp32 partial tile to the tile's accumulation buffer in the
// workspace (reductions done in L2); the last of the tile's blocks to arrive reads the sum
// and finishes the tile.  With more than two blocks on a tile the order of the additions, and so the last
// bit of the fp32 sum, depends on the order of arrival.
struct SegIter {
  long u, ue;
  int t, t_end, n_kb, step, tail_tile0, half_tile, half, ps_tile, ps_kb0, ps_kb1;
  __device__ inline void init(const PrefillCfg& c, int b, int grid) {
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

// T: activation / output type.  CONV: the activation tiles arrive as bf16 and are converted to fp16 in
// shared memory by the de-quantisers (used when the workspace cannot hold a converted copy).
// HEADS: the input map is a family of per-head blocks (else a leading block).
template <typename T, bool CONV, bool HEADS>
__global__ void __launch_bounds__(PTH, 1) one_block_kernel(const __grid_constant__ Params p,
                                                         const __grid_constant__ PrefillCfg c) {
  extern __shared__ unsigned char psmem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // (warp-uniform for the compiler)
  // Programmatic dependent launch: the next kernel of the stream may be set up while this one runs (its blocks
  // become resident as ours leave).  What a block does before its own `griddepcontrol.wait` touches nothing a
  // predecessor may still write or read: barriers, tensor memory, and the weights, which no kernel writes (the
  // de-quantisers fill the ring ahead); activations, positions, outputs and workspace come after the wait.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t raw = (uint32_t)__cvta_generic_to_shared(psmem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;           // swizzled tiles need 1024-byte alignment
  unsigned char* smem = psmem_raw + (sbase - raw);
  const uint32_t bars = sbase + RING_BYTES;
  const uint32_t full_a = bars, empty_a = bars + 8 * PSTAGES;
  const uint32_t full_b = bars + 16 * PSTAGES, empty_b = full_b + 8 * BSLOTS;
  const uint32_t acc_full = full_b + 16 * BSLOTS, acc_empty = acc_full + 16, epi_bar = acc_full + 32;
  const uint32_t help_bar = acc_full + 40;         // the epilogue warps and the de-quantiser warps that help them
  const uint32_t last_full = acc_full + 48;        // the MMAs of the block's last segment are complete (one phase only)
  const uint32_t px_ready = acc_full + 56;         // pair split, second block: the first block's rings are idle
  const uint32_t px_done = acc_full + 64;          // pair split, first block: the second block's sums have arrived
  unsigned char* misc = smem + RING_BYTES + 16 * PSTAGES + 16 * BSLOTS + 72;
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  if (tid == 0) {
    for (int s = 0; s < PSTAGES; ++s) {
      pmbar_init(full_a + 8 * s, DQ_TEAM_WARPS);
      pmbar_init(empty_a + 8 * s, 1);
    }
    for (int s = 0; s < BSLOTS; ++s) {
      pmbar_init(full_b + 8 * s, 1);
      pmbar_init(empty_b + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) { pmbar_init(acc_full + 8 * b, 1); pmbar_init(acc_empty + 8 * b, 4); }
    pmbar_init(epi_bar, 4);
    pmbar_init(help_bar, 4 + 2 * DQ_WARPS);
    pmbar_init(last_full, 1);
    pmbar_init(px_ready, 1);
    pmbar_init(px_done, c.helpers ? 4 + 2 * DQ_WARPS : 4);       // one arrival per warp that sends
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {                      // the whole tensor memory of the SM: two accumulators of 256 columns
    tmem_alloc((uint32_t)__cvta_generic_to_shared(const_cast<uint32_t*>(tmem_slot)), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t crank = c.pair_split ? pcluster_rank() : 0u;
  if (c.pair_split) {                   // the other block's barriers exist before anything is sent to it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }

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
    const bool ok = pmbar_poll_warp(epi_bar, epar, abort_flag);
    epar ^= 1;
    return ok;
  };
  volatile int* last_flag = reinterpret_cast<volatile int*>(misc + 8);
  uint32_t hpar = 0;
  auto help_sync = [&]() -> bool {
    __syncwarp();
    if (lane == 0) pmbar_arrive(help_bar);
    const bool ok = pmbar_poll_warp(help_bar, hpar, abort_flag);
    hpar ^= 1;
    return ok;
  };
  auto epilogue_segment = [&](const Seg& sg, int tcount, int ch0, int chs, bool helper) {
      const int acc0 = c.nh == 2 ? 0 : (tcount & 1);     // as in the MMA warp
      const int au = c.nh == 2 ? tcount : (tcount >> 1);
      const int ntok = c.bn * c.nh;                      // tokens of the tile
      const int h_lo = sg.half < 0 ? 0 : sg.half, h_hi = sg.half < 0 ? c.nh : sg.half + 1;   // boxes of this segment
      const int t = sg.tile;
      const int wt = t / c.n_ttiles, tt = t - wt * c.n_ttiles;
      const int jn = job_of_wt(wt);
      const JobDev& jb = p.job[jn];
      const int tl = wt - c.wtile_begin[jn];
      T* y = reinterpret_cast<T*>(jb.y);
      const T* bias = reinterpret_cast<const T*>(jb.bias);
      const bool rope = jb.rope.enabled != 0;
      // this thread owns tile row etid (= its TMEM lane); a rope pair sits in lanes 2i, 2i + 1
      const RowInfo ri = tile_row(jb, tl, etid);
      float b_own = 0.f;
      unsigned long long turn = 0;
      const bool swiglu = jb.pair == 1;
      if (ri.stored >= 0) {
        const T* bias_own = (swiglu && (etid & 1)) ? reinterpret_cast<const T*>(p.job[jn + 1].bias) : bias;
        if (bias_own) b_own = DT<T>::to_f(bias_own[ri.stored]);
        if (rope) {
          const int half = jb.rope.head_keep >> 1;
          int pidx = p.idx[(ri.head / jb.rope.rep) * half + ri.pair_c];
          pidx = min(max(pidx, 0), (jb.rope.head_dim >> 1) - 1);
          turn = p.rope_turn[pidx];
        }
      }
      // bias, rotary embedding, rounding and store of 32 tokens of this row (all lanes of the warp call it)
      auto store_chunk = [&](int tok0, const auto& val) {
        constexpr int NV = (int)(sizeof(val) / sizeof(float));
        const int m0 = tt * ntok + tok0;
        if (rope) {
          // the even lane of a pair rotates the even tokens, the odd lane the odd ones: one exchange hands
          // each the other member's value of its token, and it stores both rotated members
          const bool second = (lane & 1) != 0;
          const int half = jb.rope.head_keep >> 1;
          const float b_other = __shfl_xor_sync(0xffffffffu, b_own, 1);
          const float b_lo = second ? b_other : b_own, b_hi = second ? b_own : b_other;
          const bool live = ri.stored >= 0;
          const int left = p.M - m0, odd = second ? 1 : 0;
          T* yp = y + (live ? ri.out_col - (second ? half : 0) : 0) + (size_t)(m0 + odd) * jb.ldy;   // this lane's first token
          const size_t step = 2 * (size_t)jb.ldy;
          const int32_t* pp = p.pos + m0 + odd;
          if (left >= NV) {                       // a whole chunk of tokens: no test per token
#pragma unroll
            for (int k = 0; k < NV; k += 2) {
              const float got = __shfl_xor_sync(0xffffffffu, second ? val[k] : val[k + 1], 1);
              const float lo = (second ? got : val[k]) + b_lo, hi = (second ? val[k + 1] : got) + b_hi;
              float cs, sn;
              rope_cos_sin(__ldg(pp + k), turn, cs, sn);
              if (live) {
                yp[0] = DT<T>::from_f(fmaf(-hi, sn, lo * cs));
                yp[half] = DT<T>::from_f(fmaf(lo, sn, hi * cs));
              }
              yp += step;
            }
          } else {
#pragma unroll
            for (int k = 0; k < NV; k += 2) {
              if (k >= left) break;
              const float got = __shfl_xor_sync(0xffffffffu, second ? val[k] : val[k + 1], 1);
              const float lo = (second ? got : val[k]) + b_lo, hi = (second ? val[k + 1] : got) + b_hi;
              if (live && k + odd < left) {
                float cs, sn;
                rope_cos_sin(__ldg(pp + k), turn, cs, sn);
                yp[0] = DT<T>::from_f(fmaf(-hi, sn, lo * cs));
                yp[half] = DT<T>::from_f(fmaf(lo, sn, hi * cs));
              }
              yp += step;
            }
          }
        } else if (swiglu) {
          // as for a rotation pair: the even lane (gate row) takes the even tokens, the odd lane (up row) the odd
          // ones, one exchange gives each the other matrix's sum of its token; h = silu(g) * u, one rounding
          // (the approximate division: two instructions instead of ten in warps that share the issue slots
          //  with the de-quantisers; exp(-g) beyond fp32 gives a quotient of zero, the limit of silu)
          const bool second = (lane & 1) != 0;
          const float b_other = __shfl_xor_sync(0xffffffffu, b_own, 1);
          const float b_g = second ? b_other : b_own, b_u = second ? b_own : b_other;
          const bool live = ri.stored >= 0;
          const int left = p.M - m0, odd = second ? 1 : 0;
          T* yp = y + (live ? ri.out_col : 0) + (size_t)(m0 + odd) * jb.ldy;          // this lane's first token
          const size_t step = 2 * (size_t)jb.ldy;
          if (left >= NV) {                       // a whole chunk of tokens: no test per token
#pragma unroll
            for (int k = 0; k < NV; k += 2) {
              const float got = __shfl_xor_sync(0xffffffffu, second ? val[k] : val[k + 1], 1);
              const float g = (second ? got : val[k]) + b_g, u = (second ? val[k + 1] : got) + b_u;
              if (live) *yp = DT<T>::from_f(__fdividef(g, 1.f + __expf(-g)) * u);
              yp += step;
            }
          } else {
#pragma unroll
            for (int k = 0; k < NV; k += 2) {
              if (k >= left) break;
              const float got = __shfl_xor_sync(0xffffffffu, second ? val[k] : val[k + 1], 1);
              const float g = (second ? got : val[k]) + b_g, u = (second ? val[k + 1] : got) + b_u;
              if (live && k + odd < left) *yp = DT<T>::from_f(__fdividef(g, 1.f + __expf(-g)) * u);
              yp += step;
            }
          }
        } else {
          if (ri.stored < 0) return;
          T* yr = y + ri.out_col + (size_t)m0 * jb.ldy;
          const int left = p.M - m0;
          if (left >= NV) {                       // a whole chunk of tokens: no test per token
#pragma unroll
            for (int k = 0; k < NV; ++k) { *yr = DT<T>::from_f(val[k] + b_own); yr += jb.ldy; }
          } else {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
              if (k >= left) break;
              *yr = DT<T>::from_f(val[k] + b_own);
              yr += jb.ldy;
            }
          }
        }
      };
      for (int h = h_lo; h < h_hi && !failed && !helper; ++h)
        if (!pmbar_poll_warp(acc_full + 8 * (acc0 + h), au & 1, abort_flag)) failed = true;
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
        if (lane == 0) pmbar_arrive(acc_empty + 8 * (acc0 + (ch * EPI_TOK) / c.bn));
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
        const bool pair_send = c.pair_split && crank != 0;
        if (c.pair_split && !pair_send) {
          // ---- the two blocks of a cluster each ran half of the contraction.  The second block waits until the
          //      first one's MMAs are complete (its rings are idle then), writes its fp32 sums into them ([token][row]:
          //      a warp stores 32 consecutive rows of a token) and arrives, one arrival per warp, at the first block's
          //      barrier; the first block adds them to its own sums (always own + other: the same bits every run)
          //      and finishes the tile.  No traffic through L2, no counter, nothing to clear.
          {
            if (!pmbar_wait_cluster_warp(px_done, 0, abort_flag)) { failed = true; return; }
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
        const int T0 = (c.n_tiles / (int)gridDim.x) * (int)gridDim.x;          // first left-over tile
        float* mine = c.partials + ((size_t)(t - T0) + (c.sk_atomic ? 0 : blockIdx.x)) * slot_f;
        if (pair_send) {
          // (the second block of a pair: its "slot" is the first block's rings, once they are idle)
          if (!pmbar_wait_cluster_warp(px_ready, 0, abort_flag)) { failed = true; return; }
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
        const long U = (long)(c.n_tiles - T0) * c.n_kb, Bn = (long)gridDim.x < U ? (long)gridDim.x : U;
        const long tu = (long)(t - T0) * c.n_kb;                               // the tile's first left-over unit
        const int first = sk_owner(tu, Bn, U), last = sk_owner(tu + c.n_kb - 1, Bn, U);
        if (main_lane) {
          const int arrived = atomicAdd(&c.counters[t], 1);    // ... the block's arrival shows
          *last_flag = arrived == last - first;
          __threadfence();
        }
        if (!(chs == 1 ? epi_sync() : help_sync())) { failed = true; return; }
        if (*last_flag) {
          const float* base = c.partials + ((size_t)(t - T0) + (c.sk_atomic ? 0 : first)) * slot_f;
          const int parts = c.sk_atomic ? 1 : last - first + 1;
          // 16 tokens at a time, the loads of two slots in flight together (what the registers of a thread hold)
          for (int tk = 16 * ch0; tk < ntok && tt * ntok + tk < p.M; tk += 16 * chs) {
            float val[16];
#pragma unroll
            for (int k = 0; k < 16; ++k) val[k] = 0.f;
            const float* src = base + (size_t)tk * BMW + row;
            for (int s2 = 0; s2 < parts; s2 += 2) {
              const bool two = s2 + 1 < parts;
              float a[16], b[16];
#pragma unroll
              for (int k = 0; k < 16; ++k) a[k] = __ldcg(src + (size_t)s2 * slot_f + (size_t)k * BMW);
#pragma unroll
              for (int k = 0; k < 16; ++k) b[k] = two ? __ldcg(src + (size_t)(s2 + 1) * slot_f + (size_t)k * BMW) : 0.f;
#pragma unroll
              for (int k = 0; k < 16; ++k) val[k] = (val[k] + a[k]) + b[k];
            }
            store_chunk(tk, val);
          }
          if (main_lane) c.counters[t] = 0;              // ready for the next call
        }
      }
  };

  if (warp == 0) {
    // ===================================================================== activations by TMA
    if (lane == 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");   // the activations may come from the preceding kernel
      int s = 0; uint32_t par = 1; int jb = 0;             // box slot, parity of its previous use, boxes so far
      SegIter si; si.init(c, blockIdx.x, gridDim.x);
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
            if (jb >= BSLOTS && !pmbar_wait_lane(empty_b + 8 * s, par, abort_flag, true)) { failed = true; break; }
            const uint32_t fb = full_b + 8 * s;
            pmbar_expect_tx(fb, (uint32_t)(c.bn * BK * 2));
            // (a box that starts at or beyond the last token is all zeros: the tensor map ends at M)
            tma_box2(sbase + B_RING + s * B_BYTES, &c.xmap, xcol, (tt * c.nh + h) * c.bn, fb);
            if (++s == BSLOTS) { s = 0; par ^= 1; }
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
    int s = 0; uint32_t par = 0; int tcount = 0;         // weight stage and its parity
    int sb = 0; uint32_t parb = 0;                       // activation box slot and its parity
    SegIter si; si.init(c, blockIdx.x, gridDim.x);
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
        for (int h = h_lo; h < h_hi; ++h) {
          if (kb == sg.kb0 && au >= 1 && !pmbar_wait_warp(acc_empty + 8 * (acc0 + h), (au - 1) & 1, abort_flag)) { failed = true; break; }
          // (bf16: the de-quantisers waited for the activation box themselves and converted it)
          if (!CONV && !pmbar_wait_warp(full_b + 8 * sb, parb, abort_flag)) { failed = true; break; }
          tc_fence_after();
          const uint64_t bdesc = smem_desc_sw128(sbase + B_RING + sb * B_BYTES);
          if (elect_one()) {
            umma_kblock<false>(tmem_base + (uint32_t)((acc0 + h) * MAXBN), adesc, bdesc, c.idesc, kb > sg.kb0 ? 1u : 0u);
            umma_commit(empty_b + 8 * sb);              // the box is free once these MMAs have read it
            if (h == h_hi - 1) umma_commit(empty_a + 8 * s);   // ... and the weight stage after the last of them
          }
          __syncwarp();
          if (++sb == BSLOTS) { sb = 0; parb ^= 1; }
        }
        if (failed) break;
        if (++s == PSTAGES) { s = 0; par ^= 1; }
      }
      if (failed) break;
      // (the de-quantiser warps that help with the last segment's epilogue cannot follow the phases of the
      //  accumulator barriers -- a parity wait cannot tell "not yet" from "two phases ago" -- so the last
      //  segment completes a barrier of its own, which has this one phase)
      SegIter peek = si;
      Seg nxt;
      const bool last = !peek.next(nxt);
      if (elect_one()) {
        for (int h = h_lo; h < h_hi; ++h) umma_commit(acc_full + 8 * (acc0 + h));
        if (last) umma_commit(last_full);
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
    if (sc != 1) {
    const int pos = ((warp - DQ_WARP0) >> 2) * 3 + (sc == 0 ? 0 : sc - 1);      // 0..11 among the twelve
    const int team = pos / DQ_TEAM_WARPS;
    const int dt = (pos - team * DQ_TEAM_WARPS) * 32 + lane;                    // 0..191
    constexpr int TEAM_TH = DQ_TEAM_WARPS * 32;
    const int n_items = dt + TEAM_TH < 2 * BMW ? 2 : 1;                         // items dt and dt + 192 of 256
    const int G = p.K / kGroup;
    int done = 0;                      // stage iterations before this segment
    constexpr bool heads = HEADS;
    SegIter si; si.init(c, blockIdx.x, gridDim.x);
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
        const int item = dt + m * TEAM_TH;
        const int r = (item >> 1) & (BMW - 1), hf = item & 1;
        const RowInfo ri = tile_row(jb, wt - c.wtile_begin[jn], r);
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
        const int s = it & (PSTAGES - 1);
        const uint32_t use = (uint32_t)(it / PSTAGES);
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
        if (it >= PSTAGES && !pmbar_wait_warp(empty_a + 8 * s, (use - 1) & 1, abort_flag)) { failed = true; break; }
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
            if (!pmbar_wait_warp(full_b + 8 * sb, (uint32_t)(jb2 / BSLOTS) & 1, abort_flag)) { failed = true; break; }
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
        if (lane == 0) pmbar_arrive(full_a + 8 * s);
#pragma unroll
        for (int m = 0; m < 2; ++m) { q0[m] = q1[m]; s0[m] = s1[m]; z0[m] = z1[m]; }
      }
    }
    }
    // the block's segments, counted by every warp of this group (the idle four included)
    Seg last_sg = {0, 0, 0, -1};
    int n_seg = 0;
    {
      SegIter sj; sj.init(c, blockIdx.x, gridDim.x);
      Seg sgj;
      while (sj.next(sgj)) { last_sg = sgj; ++n_seg; }
    }
    // the block's last segment: this warp takes a fifth of its chunks beside the epilogue warp of its tensor-memory
    // quadrant (warps 8 + q, 12 + q, 16 + q, 20 + q: chunks 1, 2, 3, 4 of every five)
    if (c.helpers && !failed && n_seg > 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");   // outputs and workspace: after the preceding kernel
      // (the wait behind the row's set-up, as the block pairs have it, changed nothing here: Llama-3-8B layer at 512 rows, keep 0.75, on
      //  this kernel 241.8 us with either, Qwen2.5-7B at 677 rows, keep 0.65, 320.7 and 322.4, 14336 x 4224 at 96 rows 35.9 and 35.7)
      if (!pmbar_poll_warp(last_full, 0, abort_flag, true)) failed = true;
      if (!failed) epilogue_segment(last_sg, n_seg - 1, 1 + (warp - DQ_WARP0) / 4, 5, true);
    }
  } else if (warp >= EPI_WARP0) {
    // ===================================================================== epilogue
    asm volatile("griddepcontrol.wait;" ::: "memory");     // positions, outputs and workspace: after the preceding kernel
    int tcount = 0;
    SegIter si; si.init(c, blockIdx.x, gridDim.x);
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
  if (warp == 1) tmem_dealloc(tmem_base, 512);
  if (c.pair_split) {                   // neither block of a pair leaves while the other may still send to it
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}


template <typename T, bool CONV, bool HEADS>
int launch_as(const Params& p, const PrefillCfg& c, int grid, cudaStream_t stream) {
  const size_t smem = 1024 + (size_t)RING_BYTES + 512;
  auto kern = one_block_kernel<T, CONV, HEADS>;
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
  if (c.pair_split) {
    // clusters of two, only when every pair can be resident at once; else the caller plans without them
    attr[lc.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[lc.numAttrs].val.clusterDim.x = 2;
    attr[lc.numAttrs].val.clusterDim.y = 1;
    attr[lc.numAttrs].val.clusterDim.z = 1;
    ++lc.numAttrs;
    // (asked once per kernel instance: the answer depends on the block's resources, which do not change)
    static std::atomic<int> max_clusters{-1};
    int n_clusters = max_clusters.load();
    if (n_clusters < 0) {
      if (cudaOccupancyMaxActiveClusters(&n_clusters, kern, &lc) != cudaSuccess) { cudaGetLastError(); n_clusters = 0; }
      max_clusters.store(n_clusters);
    }
    if (n_clusters * 2 < grid || opt(kOptPrefillPair) == 3) return UNIQL_ERR_UNSUPPORTED;
  }
  if (cudaLaunchKernelEx(&lc, kern, p, c) != cudaSuccess) { cudaGetLastError(); return c.pair_split ? UNIQL_ERR_UNSUPPORTED : UNIQL_ERR_CUDA; }
  return UNIQL_OK;
}

}  // namespace

int launch_one_block(const Params& p, const PrefillCfg& c, int grid, bool conv, cudaStream_t stream) {
  const bool heads = c.km_period != 0;
  if (p.dt == UNIQL_BF16 && conv)
    return heads ? launch_as<__nv_bfloat16, true, true>(p, c, grid, stream) : launch_as<__nv_bfloat16, true, false>(p, c, grid, stream);
  if (p.dt == UNIQL_BF16)
    return heads ? launch_as<__nv_bfloat16, false, true>(p, c, grid, stream) : launch_as<__nv_bfloat16, false, false>(p, c, grid, stream);
  return heads ? launch_as<__half, false, true>(p, c, grid, stream) : launch_as<__half, false, false>(p, c, grid, stream);
}

}  // namespace uniql
