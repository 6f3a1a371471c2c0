// Batch kernel (17 to 128 rows, the serving batches between decode and prefill) of the pruned 4-bit linear layer,
// sm_100a: tcgen05 MMAs whose weight operand lies in tensor memory.
//
// What bounds it.  At these sizes the weights stream once and each is used for 17 - 128 tokens: 16 MB of codes are 2.5 us
// of HBM and at most 1 us of tensor time, but every code has to become an fp16 value on the way.  The prefill kernel
// writes those values to shared memory, one 64-channel k-block (4 KB of codes) per hand-shake, and took 0.45 us per
// k-block and SM whatever the batch: 1.3 TB/s.  Here
//  - a stage is 256 channels of 128 weight rows (16 KB of codes), fetched by cp.async up to seven stages ahead, so that
//    100 KB per SM are in flight and the hand-shakes are a quarter as many per byte;
//  - a de-quantiser thread owns a weight row (= a lane of tensor memory) and 64 channels of the stage: two 16-byte
//    shared loads, 64 values in 32 registers, ONE tcgen05.st: nothing goes back through shared memory, where 16 KB
//    written and 16 KB read per 8192 weights alone would take 256 cycles against the 195 that HBM needs for their codes;
//  - the MMAs take A from tensor memory (measured: 24 / 42 / 67 cycles per 128 x N x 16 at N = 16 / 64 / 128, against
//    90 - 96 with A in shared memory), N is the batch rounded up to 16.
// Measured figures stand at launch_batch().
//
// Roles (one persistent block per SM, 24 warps):
//   warp 0       activations by TMA: four boxes [64 k x N tokens] per stage, 128-byte swizzle
//   warp 1       tensor-memory allocation, MMA issue (16 per stage)
//   warps 2, 3   loaders: codes and scales of a stage by cp.async, 64 rows each
//   warps 4..7   epilogue (bias, rotation or gated product, store; RowStore)
//   warps 8..23  de-quantisers: warp w rows 32 (w % 4) .. + 31, channels 64 ((w - 8) / 4) .. + 63 of every stage; they
//                share the epilogue of the block's last segment
// Tensor memory: two accumulators of N columns, then two or three A stages of 128 columns.
//
// Work split: every block runs the same number of whole tiles; the stages of the tiles left over are cut into equal
// ranges (stream-K), run FIRST, so that their hand-over overlaps the whole tiles.  A part goes to a slot in the workspace
// ([token][row] fp32); the last block of a tile to arrive adds the slots in block order (deterministic).
// Pruning (Section 3.4): the rows of a tile are compact output channels mapped to stored rows per lane; the input side is
// the leading k_in channels (the tensor map of x ends there) or the kept channels of heads whose k-blocks are all
// visited (pruned words of a partly kept k-block become zero weights).
// Every wait is bounded; on expiry the block raises a flag, all roles leave, the status word is set.
#include <cuda.h>
#include <string.h>

#include <atomic>
#include <mutex>

#include "tc.cuh"

namespace uniql {
namespace {

constexpr int KS = 4;                          // k-blocks per stage
constexpr int NW = 24, NTHB = NW * 32;
constexpr int WST_BYTES = BMW * 128;           // codes of a stage: 128 bytes per row, 16-byte pieces XOR-swizzled by row
constexpr int SZ_BYTES = BMW * 8;              // two scales and two zero-points per row: [row] half2 s, [row] half2 z
constexpr int WSTAGE = WST_BYTES + SZ_BYTES;
constexpr int MAX_WST = 8, MAX_BST = 4, MAX_AST = 3;
constexpr int LOADERS = 2, LD_WARP0 = 2, EPI0 = 4, DQ0 = 8, DQN = 16;
constexpr int kSmemBatch = 227 * 1024;
constexpr int kTokChunk = 16;                  // tokens per epilogue pass

struct BatchCfg {
  CUtensorMap xmap;          // activations: (k, token), box 64 x n
  int n;                     // tokens of an MMA: M rounded up to 16
  int n_ast, acc_stride, a_base;               // tensor memory: A stages, columns between the accumulators, first A column
  int wst, bst, off_w, off_bar;                // ring depths and shared-memory offsets (the activation ring is first)
  int wtile_begin[kMaxJobs + 1];
  int n_tiles, n_kb, spt;    // weight tiles of 128 rows, k-blocks, stages per tile
  int kb_first;              // first stored k-block
  int head_kb, head_keep;    // per-head maps: k-blocks and kept channels per head (0: leading block)
  uint32_t idesc;
  int base, left, sharers;   // whole tiles per block; tiles left over; blocks that share the stages of those
  int* status;
  int* counters;
  float* partials;           // one slot [n tokens][128 rows] per (left-over tile, block) piece
};

__device__ inline void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// 32 columns of this thread's lane
__device__ inline void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
        "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
        "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31]) : "memory");
}
__device__ inline void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ inline void bcp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// (through L1: eight consecutive stages use the same 32-byte sector of a row's scales)
__device__ inline void bcp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ inline void bcp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// A block's work as segments (tile, stages [s0, s1)): its range of the left-over tiles first, then its whole tiles.
struct BSeg { int tile, s0, s1; };
struct BSegIter {
  int u, ue, t, t_end, spt, tail0;
  __device__ inline void init(const BatchCfg& c, int b, int grid) {
    spt = c.spt;
    tail0 = c.base * grid;
    t = b * c.base; t_end = t + c.base;
    u = ue = 0;
    if (b < c.sharers) {
      const unsigned long long U = (unsigned long long)c.left * c.spt;
      u = (int)(U * b / c.sharers); ue = (int)(U * (b + 1) / c.sharers);
    }
  }
  __device__ inline bool next(BSeg& g) {
    if (u < ue) {
      const int tt = u / spt;
      g.tile = tail0 + tt; g.s0 = u - tt * spt;
      const int len = min(spt - g.s0, ue - u);
      g.s1 = g.s0 + len;
      u += len;
      return true;
    }
    if (t < t_end) { g.tile = t++; g.s0 = 0; g.s1 = spt; return true; }
    return false;
  }
};
// the block whose range of the left-over stages holds stage u
__device__ inline int bowner(int u, int B, int U) { return (int)((((unsigned long long)u + 1) * B - 1) / U); }

template <typename T, bool HEADS>
__global__ void __launch_bounds__(NTHB, 1) batch_kernel(const __grid_constant__ Params p, const __grid_constant__ BatchCfg c) {
  extern __shared__ unsigned char bsm_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t raw = (uint32_t)__cvta_generic_to_shared(bsm_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  unsigned char* smem = bsm_raw + (sbase - raw);
  const uint32_t bars = sbase + (uint32_t)c.off_bar;
  const uint32_t w_full = bars, w_empty = w_full + 8 * MAX_WST, b_full = w_empty + 8 * MAX_WST, b_empty = b_full + 8 * MAX_BST;
  const uint32_t a_full = b_empty + 8 * MAX_BST, a_empty = a_full + 8 * MAX_AST;
  const uint32_t acc_full = a_empty + 8 * MAX_AST, acc_empty = acc_full + 16, epi_bar = acc_empty + 16, help_bar = epi_bar + 8;
  const uint32_t last_full = help_bar + 8;
  unsigned char* misc = smem + c.off_bar + 8 * (2 * MAX_WST + 2 * MAX_BST + 2 * MAX_AST + 4 + 3);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);
  volatile int* last_flag = reinterpret_cast<volatile int*>(misc + 8);

  if (tid == 0) {
    for (int s = 0; s < MAX_WST; ++s) { pmbar_init(w_full + 8 * s, LOADERS * 32); pmbar_init(w_empty + 8 * s, DQN); }
    for (int s = 0; s < MAX_BST; ++s) { pmbar_init(b_full + 8 * s, 1); pmbar_init(b_empty + 8 * s, 1); }
    for (int s = 0; s < MAX_AST; ++s) { pmbar_init(a_full + 8 * s, DQN); pmbar_init(a_empty + 8 * s, 1); }
    for (int s = 0; s < 2; ++s) { pmbar_init(acc_full + 8 * s, 1); pmbar_init(acc_empty + 8 * s, 4); }
    pmbar_init(epi_bar, 4);
    pmbar_init(help_bar, 4 + DQN);
    pmbar_init(last_full, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc((uint32_t)__cvta_generic_to_shared(const_cast<uint32_t*>(tmem_slot)), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int grid = (int)gridDim.x;
  bool failed = false;
  auto job_of_tile = [&](int t) { int j = 0; while (j + 1 < p.n_jobs && t >= c.wtile_begin[j + 1]) ++j; return j; };

  // ---- epilogue of one segment for the warp that calls it: token chunks ch0, ch0 + chs, ... (chs == 1: the epilogue warp
  //      on its own, which also hands the accumulator back)
  uint32_t epar = 0;
  auto group_sync = [&](uint32_t bar) -> bool {
    __syncwarp();
    if (lane == 0) pmbar_arrive(bar);
    const bool ok = pmbar_wait_warp(bar, epar, abort_flag);
    epar ^= 1;
    return ok;
  };
  auto epilogue_segment = [&](const BSeg& sg, int count, int ch0, int chs) {
    const int q = warp & 3, acc = count & 1;
    const int jn = job_of_tile(sg.tile);
    const RowStore<T> rs(p, jn, sg.tile - c.wtile_begin[jn], 32 * q + lane);
    const uint32_t t_acc = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * c.acc_stride);
    const uint32_t bar = chs == 1 ? epi_bar : help_bar;
    tc_fence_after();
    auto release = [&]() {                                     // (chs == 1) the accumulator's values are in registers
      tc_fence_before();
      __syncwarp();
      if (lane == 0) pmbar_arrive(acc_empty + 8 * acc);
    };
    const bool whole = sg.s0 == 0 && sg.s1 == c.spt;
    const int tail0 = c.base * grid, lt = sg.tile - tail0;
    const size_t slot_f = (size_t)c.n * BMW;
    float* mine = whole ? nullptr : c.partials + ((size_t)lt + blockIdx.x) * slot_f + 32 * q + lane;
    for (int tk = kTokChunk * ch0; tk < c.n; tk += kTokChunk * chs) {
      uint32_t v[16];
      tmem_ld16(t_acc + (uint32_t)tk, v);
      tmem_ld_wait();
      if (chs == 1 && tk + kTokChunk >= c.n) release();
      if (whole) {
        float val[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) val[k] = __uint_as_float(v[k]);
        rs.store(p, tk, val);
      } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) __stcg(mine + (size_t)(tk + k) * BMW, __uint_as_float(v[k]));
      }
    }
    if (whole) return;
    __threadfence();                                           // this thread's part is in place before ...
    if (!group_sync(bar)) { failed = true; return; }
    const int U = c.left * c.spt;
    const int first = bowner(lt * c.spt, c.sharers, U), last = bowner(lt * c.spt + c.spt - 1, c.sharers, U);
    const bool main_lane = warp == EPI0 && lane == 0;
    if (main_lane) {
      *last_flag = atomicAdd(&c.counters[sg.tile], 1) == last - first;      // ... the block's arrival shows
      __threadfence();
    }
    if (!group_sync(bar)) { failed = true; return; }
    if (*last_flag) {
      const float* src0 = c.partials + ((size_t)lt + first) * slot_f + 32 * q + lane;
      const int parts = last - first + 1;
      for (int tk = kTokChunk * ch0; tk < c.n; tk += kTokChunk * chs) {
        const float* src = src0 + (size_t)tk * BMW;
        float val[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) val[k] = __ldcg(src + (size_t)k * BMW);
        for (int s = 1; s < parts; s += 2) {                   // the loads of two slots in flight
          const bool two = s + 1 < parts;
          const float* sp = src + (size_t)s * slot_f;
          float a[16], b[16];
#pragma unroll
          for (int k = 0; k < 16; ++k) a[k] = __ldcg(sp + (size_t)k * BMW);
#pragma unroll
          for (int k = 0; k < 16; ++k) b[k] = two ? __ldcg(sp + slot_f + (size_t)k * BMW) : 0.f;
#pragma unroll
          for (int k = 0; k < 16; ++k) val[k] = (val[k] + a[k]) + b[k];
        }
        rs.store(p, tk, val);
      }
      if (main_lane) c.counters[sg.tile] = 0;                  // ready for the next call
    }
  };

  BSegIter si;
  si.init(c, (int)blockIdx.x, grid);
  BSeg sg;
  if (warp == 0) {
    // ===================================================================== activations
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int s = 0, it = 0; uint32_t par = 1;
    const uint32_t box = (uint32_t)c.n * 128u;
    while (!failed && si.next(sg)) {
      for (int st = sg.s0; st < sg.s1; ++st, ++it) {
        if (it >= c.bst && !pmbar_wait_warp(b_empty + 8 * s, par, abort_flag, true)) { failed = true; break; }
        const int v0 = st * KS, nv = min(KS, c.n_kb - v0);
        const uint32_t fb = b_full + 8 * s;
        if (elect_one()) {
          pmbar_expect_tx(fb, (uint32_t)nv * box);
          for (int i = 0; i < nv; ++i) {
            const int v = v0 + i;
            const int x = HEADS ? (v / c.head_kb) * c.head_keep + (v % c.head_kb) * BK : v * BK;
            tma_box2(sbase + (uint32_t)(s * KS + i) * box, &c.xmap, x, 0, fb);
          }
        }
        __syncwarp();
        if (++s == c.bst) { s = 0; par ^= 1; }
      }
    }
    if (failed) {                           // let the copies still armed land before the block goes away
      for (int j = it > c.bst ? it - c.bst : 0; j < it; ++j)
        for (int i = 0; i < kPWait && !pmbar_try(b_full + 8 * (j % c.bst), (j / c.bst) & 1); ++i) {}
    }
  } else if (warp == 1) {
    // ===================================================================== MMA issue
    int as = 0, bs = 0, count = 0; uint32_t apar = 0, bpar = 0;
    for (; !failed && si.next(sg); ++count) {
      const int acc = count & 1, use = count >> 1;
      const uint32_t d = tmem + (uint32_t)(acc * c.acc_stride);
      if (use >= 1 && !pmbar_wait_warp(acc_empty + 8 * acc, (use - 1) & 1, abort_flag)) { failed = true; break; }
      for (int st = sg.s0; st < sg.s1; ++st) {
        if (!pmbar_wait_warp(b_full + 8 * bs, bpar, abort_flag) || !pmbar_wait_warp(a_full + 8 * as, apar, abort_flag)) { failed = true; break; }
        tc_fence_after();
        const int nv = min(KS, c.n_kb - st * KS);
        const uint32_t a0 = tmem + (uint32_t)(c.a_base + 128 * as);
        const uint32_t b0 = sbase + (uint32_t)(bs * KS * c.n) * 128u;
        if (elect_one()) {
          for (int i = 0; i < nv; ++i) {
            const uint64_t bd = smem_desc_sw128(b0 + (uint32_t)(i * c.n) * 128u);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_ts(d, a0 + 32 * i + 8 * k, bd + 2 * k, c.idesc, (st > sg.s0 || i > 0 || k > 0) ? 1u : 0u);
          }
          umma_commit(a_empty + 8 * as);
          umma_commit(b_empty + 8 * bs);
        }
        __syncwarp();
        if (++as == c.n_ast) { as = 0; apar ^= 1; }
        if (++bs == c.bst) { bs = 0; bpar ^= 1; }
      }
      if (failed) break;
      BSegIter peek = si;
      BSeg nxt;
      const bool last = !peek.next(nxt);
      if (elect_one()) {
        umma_commit(acc_full + 8 * acc);
        if (last) umma_commit(last_full);      // (the helpers' own barrier: one phase, no parity to lose)
      }
      __syncwarp();
    }
  } else if (warp < EPI0) {
    // ===================================================================== loaders: 64 rows each
    // A piece is 16 bytes: eight lanes fetch the 128 bytes of a row (four rows, four cache lines per instruction).
    const int r0 = (warp - LD_WARP0) * 64;
    const int G = p.K / kGroup;
    int s = 0, it = 0; uint32_t par = 1;
    while (!failed && si.next(sg)) {
      const int jn = job_of_tile(sg.tile);
      const JobDev& jb = p.job[jn];
      const int tl = sg.tile - c.wtile_begin[jn];
      const bool pair = jb.pair == 1;
      // stored rows r0 + lane and r0 + 32 + lane (-1: empty, its sums are never stored)
      const int row0 = tile_row(jb, tl, r0 + lane).stored, row1 = tile_row(jb, tl, r0 + 32 + lane).stored;
      // odd rows of a SwiGLU pair come from the up matrix
      const JobDev& jw = (pair && ((lane >> 3) & 1)) ? p.job[jn + 1] : jb;      // of the rows this lane fetches codes for
      const JobDev& js = (pair && (lane & 1)) ? p.job[jn + 1] : jb;             // of the rows it fetches scales for
      const uint8_t* wbase = jw.w + (size_t)c.kb_first * 32 + (lane & 7) * 16;
      const __half* sb = js.scales + c.kb_first / 2;
      const __half* zb = js.zeros + c.kb_first / 2;
      const size_t kbytes = (size_t)p.K / 2;
      for (int st = sg.s0; st < sg.s1; ++st, ++it) {
        if (it >= c.wst && !pmbar_wait_warp(w_empty + 8 * s, par, abort_flag)) { failed = true; break; }
        const int nv = min(KS, c.n_kb - st * KS);
        const uint32_t dst = sbase + (uint32_t)(c.off_w + s * WSTAGE);
        const bool piece = ((lane & 7) >> 1) < nv;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int rl = i * 4 + (lane >> 3);                                   // row within the 64
          const int row = __shfl_sync(0xffffffffu, i < 8 ? row0 : row1, rl & 31);
          if (row >= 0 && piece)
            bcp_async16(dst + (uint32_t)((r0 + rl) * 128 + (((lane & 7) ^ (rl & 7)) * 16)), wbase + (size_t)row * kbytes + (size_t)st * (KS * 32));
        }
        const uint32_t sd = dst + WST_BYTES + (uint32_t)((r0 + lane) * 4);
        if (row0 >= 0) {
          bcp_async4(sd, sb + (size_t)row0 * G + st * 2);
          bcp_async4(sd + BMW * 4, zb + (size_t)row0 * G + st * 2);
        }
        if (row1 >= 0) {
          bcp_async4(sd + 128, sb + (size_t)row1 * G + st * 2);
          bcp_async4(sd + BMW * 4 + 128, zb + (size_t)row1 * G + st * 2);
        }
        bcp_async_arrive(w_full + 8 * s);
        if (++s == c.wst) { s = 0; par ^= 1; }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else if (warp >= DQ0) {
    // ===================================================================== de-quantisers
    const int q = warp & 3, kq = (warp - DQ0) >> 2;
    const int r = 32 * q + lane;
    const uint32_t w_off = (uint32_t)(r * 128), x0 = (uint32_t)(((2 * kq) ^ (r & 7)) * 16), x1 = (uint32_t)(((2 * kq + 1) ^ (r & 7)) * 16);
    const uint32_t s_off = (uint32_t)(WST_BYTES + r * 4 + (kq >> 1) * 2);
    const uint32_t a_lane = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(c.a_base + 32 * kq);
    int ws = 0, as = 0, it = 0; uint32_t wpar = 0, apar = 1;
    int n_seg = 0;
    BSeg last_sg = {0, 0, 0};
    while (!failed && si.next(sg)) {
      last_sg = sg;
      ++n_seg;
      for (int st = sg.s0; st < sg.s1; ++st, ++it) {
        if (!pmbar_wait_warp(w_full + 8 * ws, wpar, abort_flag)) { failed = true; break; }
        const uint32_t src = sbase + (uint32_t)(c.off_w + ws * WSTAGE);
        uint32_t w[8];
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(src + w_off + x0));
        asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "r"(src + w_off + x1));
        unsigned short sh, zh;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(sh) : "r"(src + s_off));
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(zh) : "r"(src + s_off + BMW * 4));
        const __half sc = __ushort_as_half(sh);
        const __half2 s2 = __half2half2(sc);
        const __half2 cz2 = __float2half2_rn((8.f - __half2float(__ushort_as_half(zh))) * __half2float(sc));
        uint32_t o[32];
        int valid = BK;
        if (HEADS) valid = min(BK, c.head_keep - ((st * KS + kq) % c.head_kb) * BK);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint4 d = (!HEADS || j * 8 < valid) ? dequant_word(w[j], s2, cz2) : make_uint4(0, 0, 0, 0);
          o[4 * j] = d.x; o[4 * j + 1] = d.y; o[4 * j + 2] = d.z; o[4 * j + 3] = d.w;
        }
        __syncwarp();
        if (lane == 0) pmbar_arrive(w_empty + 8 * ws);
        if (it >= c.n_ast && !pmbar_wait_warp(a_empty + 8 * as, apar, abort_flag)) { failed = true; break; }
        tc_fence_after();
        tmem_st32(a_lane + (uint32_t)(128 * as), o);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) pmbar_arrive(a_full + 8 * as);
        if (++ws == c.wst) { ws = 0; wpar ^= 1; }
        if (++as == c.n_ast) { as = 0; apar ^= 1; }
      }
    }
    if (!failed && n_seg > 0) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (!pmbar_wait_warp(last_full, 0, abort_flag)) failed = true;
      if (!failed) epilogue_segment(last_sg, n_seg - 1, 1 + kq, 5);
    }
  } else {
    // ===================================================================== epilogue
    asm volatile("griddepcontrol.wait;" ::: "memory");
    int count = 0;
    for (; !failed && si.next(sg); ++count) {
      BSegIter peek = si;
      BSeg nxt;
      const bool last = !peek.next(nxt);
      if (!pmbar_wait_warp(acc_full + 8 * (count & 1), (count >> 1) & 1, abort_flag)) { failed = true; break; }
      // (the phase of help_bar starts at zero with the last segment; epi_bar's own is not used after it)
      if (last) epar = 0;
      epilogue_segment(sg, count, 0, last ? 5 : 1);
    }
  }
  if (failed && lane == 0) atomicExch(c.status, UNIQL_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// -------------------------------------------------------------------------------- host side
int batch_tiles(const JobDev& j) {
  if (j.pair == 2) return 0;                                       // its rows ride in the tiles of the job before
  if (j.pair == 1) return (j.k_out + BMW / 2 - 1) / (BMW / 2);
  if (j.rope.enabled) return (j.rope.n_heads * (j.rope.head_keep / 2) + BMW / 2 - 1) / (BMW / 2);
  return (j.k_out + BMW - 1) / BMW;
}

template <typename T, bool HEADS>
int launch_b(const Params& p, const BatchCfg& c, int grid, size_t smem, cudaStream_t stream) {
  auto kern = batch_kernel<T, HEADS>;
  {
    static std::mutex mu;                    // (the shared-memory limit is raised once per device)
    static bool done[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return UNIQL_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (dev < 0 || dev >= 64 || !done[dev]) {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBatch) != cudaSuccess) return UNIQL_ERR_CUDA;
      if (dev >= 0 && dev < 64) done[dev] = true;
    }
  }
  cudaLaunchConfig_t lc;
  memset(&lc, 0, sizeof(lc));
  lc.gridDim = dim3(grid);
  lc.blockDim = dim3(NTHB);
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = attr;
  lc.numAttrs = opt(kOptPdl) ? 1 : 0;
  if (cudaLaunchKernelEx(&lc, kern, p, c) != cudaSuccess) { cudaGetLastError(); return UNIQL_ERR_CUDA; }
  return UNIQL_OK;
}

}  // namespace

// Up to 128 rows; an input map whose k-blocks are all visited from a 256-channel boundary on (a leading block, or heads
// that keep a part of every k-block); scale rows that can be copied two groups at a time.
int batch_supported(const Params& p) {
  if (p.M < 1 || p.M > 128 || p.K % (2 * kGroup) != 0 || p.imap.n_fam != 1) return 0;
  const Fam& a = p.imap.fam[0];
  if (a.count == 1) {
    if (a.start != 0) return 0;
  } else if (a.start % (KS * BK) != 0 || a.period % BK != 0 || a.keep % 8 != 0 || a.keep <= a.period - BK) {
    return 0;
  }
  if ((p.ldx % 8) != 0 || (((uintptr_t)p.x) & 15) != 0) return 0;
  for (int j = 0; j < p.n_jobs; ++j)
    if ((((uintptr_t)p.job[j].scales) | ((uintptr_t)p.job[j].zeros)) & 3) return 0;
  return 1;
}

int launch_batch(const Params& p, const LaunchCfg& cfg) {
  BatchCfg c;
  memset(&c, 0, sizeof(c));
  for (int j = 0; j < p.n_jobs; ++j) { c.wtile_begin[j] = c.n_tiles; c.n_tiles += batch_tiles(p.job[j]); }
  for (int j = p.n_jobs; j <= kMaxJobs; ++j) c.wtile_begin[j] = c.n_tiles;
  if (c.n_tiles < 1) return UNIQL_ERR_SHAPE;
  c.n = (p.M + 15) / 16 * 16;
  const Fam& a = p.imap.fam[0];
  const int kbh = (a.keep + BK - 1) / BK;
  c.n_kb = kbh * a.count;
  c.spt = (c.n_kb + KS - 1) / KS;
  c.kb_first = a.start / BK;
  c.head_kb = a.count > 1 ? kbh : 0;
  c.head_keep = a.keep;
  // fp32 accumulate, A and B fp16, both K-major, N tokens, 128 rows
  c.idesc = (1u << 4) | ((uint32_t)(c.n >> 3) << 17) | ((uint32_t)(BMW >> 4) << 24);
  c.acc_stride = c.n <= 64 ? 64 : 128;
  c.n_ast = c.n <= 64 ? 3 : 2;
  c.a_base = 2 * c.acc_stride;
  // shared memory: two to four stages of activations, the rest for the codes (deep: HBM's latency is theirs to cover)
  c.bst = c.n > 80 ? 2 : (c.n > 32 ? 3 : 4);
  c.off_w = c.bst * KS * c.n * 128;
  const int room = kSmemBatch - 1024 - 512 - c.off_w;
  c.wst = room / WSTAGE < MAX_WST ? room / WSTAGE : MAX_WST;
  c.off_bar = c.off_w + c.wst * WSTAGE;
  const size_t smem = 1024 + (size_t)c.off_bar + 512;
  c.status = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(cfg.workspace) + decode_status_offset());
  c.counters = reinterpret_cast<int*>(cfg.workspace);
  size_t used = (decode_workspace_header_bytes() + 255) & ~(size_t)255;
  const void* x = p.x;
  int ldx = p.ldx;
  if (p.dt == UNIQL_BF16) {                     // (room for the copy was checked by the caller)
    ldx = (p.k_in + 63) / 64 * 64;
    x = reinterpret_cast<unsigned char*>(cfg.workspace) + used;
    used = (used + (size_t)p.M * ldx * 2 + 255) & ~(size_t)255;
  }
  const int sms = device_sms();
  int g = sms;
  const int env_grid = opt(kOptPrefillGrid), env_split = opt(kOptPrefillStreamk);
  if (env_grid >= 1 && env_grid <= sms) g = env_grid;
  // The split: a stage takes about half a microsecond, a hand-over at a block's end (no whole tiles behind it) about
  // seven stages more, in front of whole tiles about one.
  c.base = c.n_tiles / g;
  c.left = c.n_tiles - c.base * g;
  c.sharers = 0;
  int grid = g;
  if (c.left > 0) {
    const long U = (long)c.left * c.spt;
    const long B = U < g ? U : g;
    const double split = (double)U / B + (c.base == 0 ? 7.0 : 1.0);
    const size_t slots = (size_t)(c.left + g) * c.n * BMW * 4;
    const bool want = env_split >= 0 ? env_split >= 1 : split < c.spt;
    if (want && c.n_tiles <= (1 << 16) && cfg.ws_bytes >= used + slots) c.sharers = (int)B;
    else c.sharers = c.left;                    // one left-over tile each, whole
    c.partials = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(cfg.workspace) + used);
    if (c.base == 0) grid = c.sharers;
  }
  if (p.dt == UNIQL_BF16) {
    const int rc = launch_x_to_f16(p.x, p.ldx, p.M, p.k_in, const_cast<void*>(x), ldx, cfg.stream);
    if (rc != UNIQL_OK) return rc;
  }
  const int rc = encode_x_map(&c.xmap, x, p.k_in, p.M, ldx, c.n, false);
  if (rc != UNIQL_OK) return rc;
  const bool heads = c.head_kb != 0;
  if (p.dt == UNIQL_BF16)
    return heads ? launch_b<__nv_bfloat16, true>(p, c, grid, smem, cfg.stream) : launch_b<__nv_bfloat16, false>(p, c, grid, smem, cfg.stream);
  return heads ? launch_b<__half, true>(p, c, grid, smem, cfg.stream) : launch_b<__half, false>(p, c, grid, smem, cfg.stream);
}

}  // namespace uniql
