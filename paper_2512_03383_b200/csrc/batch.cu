// Batch kernel (17 to 128 rows, the serving batches between decode and prefill) of the pruned 4-bit linear layer,
// sm_100a: tcgen05 MMAs whose weight operand lies in tensor memory.
//
// What bounds it.  At these sizes the weights stream once and each is used for 17 - 128 tokens: 16 MB of codes are 2.5 us
// of HBM and at most 1 us of tensor time, but every code has to become an fp16 value on the way.  The prefill kernel
// writes those values to shared memory, one 64-channel k-block (4 KB of codes) per hand-shake, and took 0.45 us per
// k-block and SM whatever the batch: 1.3 TB/s.  Here
//  - a stage is 256 channels of 128 weight rows (16 KB of codes), one TMA box or a few, fetched up to eight stages ahead,
//    so that 100 KB per SM are in flight and the hand-shakes are a quarter as many per byte;
//  - a de-quantiser thread owns a weight row (= a lane of tensor memory) and 128 channels of the stage: four 16-byte
//    shared loads, two times 64 values in 32 registers and a tcgen05.st: nothing goes back through shared memory, where
//    16 KB written and 16 KB read per 8192 weights alone would take 256 cycles against the 195 that HBM needs for their
//    codes;
//  - the MMAs take A from tensor memory (measured: 24 / 42 / 67 cycles per 128 x N x 16 at N = 16 / 64 / 128, against
//    90 - 96 with A in shared memory), N is the batch rounded up to 16;
//  - two blocks share an SM (half of its shared memory, tensor memory and registers each).  A launch is 5 - 20 us of
//    which a block spends 4 on its way to the first stage and 3 on the exchange at its end; with one block per SM
//    nothing covered those, and blocks that entered late (their SM's predecessor had left late) left late again.
// Measured figures stand at launch_batch().
//
// Roles (12 warps, two blocks per SM):
//   warp 0       activations by TMA: two boxes [64 k x N tokens] per half stage, 128-byte swizzle
//   warp 1       tensor-memory allocation, MMA issue (8 per half stage of 128 channels)
//   warps 2, 3   loaders: codes by TMA (warp 2), scales and zero-points by cp.async (64 rows each)
//   warps 4..11  de-quantisers: warp w rows 32 (w % 4) .. + 31, channels 128 ((w - 4) / 4) .. + 127 of every stage, and
//                then the tile's epilogue (bias, rotation or gated product, store; RowStore)
// Tensor memory (256 columns): an accumulator of N columns, two or three half-stage A operands of 64 columns.
//
// EXACT instance (fp16, up to 16 rows).  The decode kernel, which takes these sizes otherwise, multiplies the codes
// themselves; rounding code x scale to fp16 would lose precision against it.  So here A holds codes - 8 (exact in fp16), a
// half stage is one group of 128 channels with accumulators of its own (P = sum (q - 8) x of 16 tokens and, from an operand
// of ones, X = sum x in every lane), and the de-quantiser thread that made the operand adds s P + s (8 - z) X to fp32
// registers: activations and codes enter unrounded, all sums are fp32.  The group's accumulators are read where the
// thread waits for its A slot anyway.  Two FMAs per token and group replace one per pair of codes.
//
// Work split: clusters of p blocks share a tile, every block a p-th of its stages; the cluster takes tiles round-robin.
// Each block then owns every p-th chunk of 16 tokens: it leaves its fp32 sums of the other chunks in a slot of its own
// ([token][row], L2), tells the peers (remote arrivals on a barrier in their shared memory), and adds up and finishes its
// own chunks, always in rank order (deterministic).  No block is the last one that reads everybody's parts: with
// tiles cut into ranges for single blocks, the last block to arrive finished 6 - 9 us after its last MMA, and the next
// launch's activations waited for it.
// Pruning (Section 3.4): a family of kept row blocks is a 3-D tensor (byte in row, row in block, block) as in the decode
// kernel; a tile is up to 128 rows of one block, or several whole blocks of a box each; the input side is
// the leading k_in channels (the tensor map of x ends there) or the kept channels of heads whose k-blocks are all
// visited (pruned words of a partly kept k-block become zero weights).
// Every wait is bounded; on expiry the block raises a flag, all roles leave, the status word is set.
#include <cuda.h>
#include <string.h>

#include <atomic>
#include <mutex>
#include <type_traits>

#include "tc.cuh"

namespace uniql {
namespace {

constexpr int KS = 4;                          // k-blocks per stage
constexpr int NTHB = 384;
constexpr int WST_BYTES = BMW * 128;           // codes of a stage: 128 bytes per row, 16-byte pieces XOR-swizzled by row
constexpr int SZ_BYTES = BMW * 8;              // two scales and two zero-points per row: [row] half2 s, [row] half2 z
constexpr int WSTAGE = WST_BYTES + SZ_BYTES;
constexpr int kMaxBF = 8;                      // row families of a launch
constexpr int MAX_WST = 6, MAX_BST = 4, MAX_AST = 3;
constexpr int LOADERS = 2, LD_WARP0 = 2, DQ0 = 4, DQN = 8;
constexpr int kSmemBatch = 113 * 1024;         // two blocks per SM
constexpr int kSmemAlone = 118 * 1024;         // one (never beside another block of this kernel)
constexpr int kTmemCols = 256;
constexpr int kTokChunk = 8;                   // tokens per epilogue pass; chunk i is finished by block i % p of the cluster

// One family of kept row blocks {start, period, keep, count} of a job.  Plain: a block of up to 128 rows is one box and
// `per_tile` blocks share a tile; a longer block takes `tpb` tiles of its own.  Rotation pairs and SwiGLU pairs: rows are
// pairs, a tile holds half as many, and each block has two boxes (first and second half of a head; gate and up).
struct BFam {
  int tile_begin, job, mode;
  int keep, count, start, period, out_base;
  int box_rows, per_tile, tpb;
};
enum { kBPlain = 0, kBRope = 1, kBSwiglu = 2 };

struct BatchCfg {
  CUtensorMap wmap[kMaxBF];  // packed weights of each family
  CUtensorMap wmap_up;       // SwiGLU: the up matrix (wmap[] holds the gate matrix)
  CUtensorMap xmap;          // activations: (k, token), box 64 x n
  int n;                     // tokens of an MMA: M rounded up to 16
  int n_ast, a_base;         // tensor memory: half-stage A operands, their first column
  int exact;                 // codes as operands, scales applied to the groups' sums
  uint32_t never;            // 0, unknown to the compiler: makes an instruction wait for values that do not change its result
  int wst, bst, off_w, off_bar;                // ring depths and shared-memory offsets (the activation ring is first)
  BFam fam[kMaxBF];
  int n_fam;
  int n_tiles, n_kb, spt;    // weight tiles of 128 rows, k-blocks, stages per tile
  int kb_first;              // first stored k-block
  int head_kb, head_keep;    // per-head maps: k-blocks and kept channels per head (0: leading block)
  int heads;                 // the instance: see batch_kernel()
  uint32_t idesc;
  int p;                     // blocks per tile (cluster size)
  int* status;
  float* partials;           // two slots [n tokens][128 rows] fp32 per block (p > 1)
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
__device__ inline void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]) : "memory");
}
__device__ inline void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// (through L1: eight consecutive stages use the same 32-byte sector of a row's scales)
__device__ inline void bcp_async4(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
__device__ inline void bcp_async_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

// Row r (a lane of tensor memory) of a tile: what it is, and where its codes lie in a stage.
struct BRow { RowInfo info; int smem_row; };
__device__ inline BRow batch_row(const BatchCfg& c, const Params& p, const BFam& f, int tile, int r) {
  BRow o;
  o.info.stored = -1; o.info.out_col = -1; o.info.pair_c = 0; o.info.head = 0;
  const int tl = tile - f.tile_begin, m = r & 1;
  const bool pairs = f.mode != kBPlain;
  const int i = pairs ? r >> 1 : r;                   // row or pair within the tile
  int h, row, b = 0;
  if (f.per_tile == 0) {                              // a long block: this is one of its tiles
    h = tl / f.tpb;
    row = (tl - h * f.tpb) * (pairs ? BMW / 2 : BMW) + i;
    o.smem_row = pairs ? m * (BMW / 2) + i : i;
  } else {
    b = i / f.box_rows;
    row = i - b * f.box_rows;
    h = tl * f.per_tile + b;
    o.smem_row = (pairs ? (2 * b + m) * f.box_rows + row : i) & (BMW - 1);
    if (b >= f.per_tile) row = f.keep;                // (rows behind the tile's last box)
  }
  if (row >= f.keep || h >= f.count) return o;
  const JobDev& jb = p.job[f.job];
  if (f.mode == kBRope) {
    o.info.stored = h * jb.rope.head_dim + m * (jb.rope.head_dim >> 1) + row;
    o.info.out_col = h * jb.rope.head_keep + m * f.keep + row;
    o.info.pair_c = row; o.info.head = h;
  } else {
    o.info.stored = f.start + h * f.period + row;
    o.info.out_col = f.out_base + h * f.keep + row;
    o.info.pair_c = m;
  }
  return o;
}
__device__ inline const BFam& fam_of_tile(const BatchCfg& c, int t) {
  int k = 0;
  while (k + 1 < c.n_fam && t >= c.fam[k + 1].tile_begin) ++k;
  return c.fam[k];
}

// A block's work: of every tile of its cluster the stages [s0, s1).  Which rank gets the longer shares rotates from tile
// to tile.
struct BSeg { int tile, s0, s1; };
struct BSegIter {
  int t, step, n, spt, p, r;
  __device__ inline void init(const BatchCfg& c, int rank) {
    p = c.p; spt = c.spt; n = c.n_tiles; r = rank;
    t = (int)blockIdx.x / p; step = (int)gridDim.x / p;
  }
  __device__ inline bool next(BSeg& g) {
    if (t >= n) return false;
    g.tile = t;
    g.s0 = spt * r / p; g.s1 = spt * (r + 1) / p;
    t += step;
    if (++r == p) r = 0;
    return true;
  }
};

// Heads that keep 4 (mod 8) channels.  A box of activations starts on a 16-byte boundary, and every second head's first column
// lies 4 channels behind one: its boxes begin those 4 columns early, and the de-quantisers move the codes of the head up by as
// many, with zero weights under what the boxes hold of the neighbours.  A copy of the activations re-laid by a kernel in front
// took 2.8 us of the 69 us of a Llama-3-8B layer at 64 rows (head dim 108).  Channels of k-block r of head h in its box:
// [lead, end).
struct HeadSpan { int shift, lead, end; };
template <bool FOURS>
__device__ inline HeadSpan head_span(const BatchCfg& c, int v) {
  HeadSpan s = {0, 0, BK};
  const int h = v / c.head_kb, r = v - h * c.head_kb;
  if (FOURS) {
    s.shift = (h & 1) ? 4 : 0;
    s.lead = r == 0 ? s.shift : 0;
  }
  s.end = min(BK, c.head_keep + s.shift - r * BK);
  return s;
}

// Tensor memory of the EXACT instance: [0, 32) the tile's sums of the two halves, then per half P and X of a group, then
// the operand of ones (eight columns; four columns of zeros behind it, so that four columns on it covers 8 channels).
constexpr uint32_t kExP = 32, kExOnes = 96, kExA = 112;

// HEADS: 0 a leading block of input channels, 1 heads that keep a multiple of 8 channels, 2 heads that keep 4 (mod 8) (an
// instance of its own: inside 1 the shifts and selects per word cost a Bamba-v2-9B mixer at 30 rows 32.2 -> 32.7 us).
template <typename T, int HEADS, bool EXACT>
__global__ void __launch_bounds__(NTHB, 2) batch_kernel(const __grid_constant__ Params p, const __grid_constant__ BatchCfg c) {
  extern __shared__ unsigned char bsm_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t raw = (uint32_t)__cvta_generic_to_shared(bsm_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  unsigned char* smem = bsm_raw + (sbase - raw);
  const uint32_t bars = sbase + (uint32_t)c.off_bar;
  const uint32_t w_full = bars, w_empty = w_full + 8 * MAX_WST, b_full = w_empty + 8 * MAX_WST, b_empty = b_full + 8 * MAX_BST;
  const uint32_t a_full = b_empty + 8 * MAX_BST, a_empty = a_full + 8 * MAX_AST;
  const uint32_t acc_full = a_empty + 8 * MAX_AST, acc_empty = acc_full + 8;
  const uint32_t xbar = acc_empty + 8;             // exchange between the blocks of a cluster: two per quadrant
  unsigned char* misc = smem + c.off_bar + 8 * (2 * MAX_WST + 2 * MAX_BST + 2 * MAX_AST + 2 + 8);
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(misc);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 4);

  if (tid == 0) {
    for (int s = 0; s < MAX_WST; ++s) { pmbar_init(w_full + 8 * s, LOADERS * 32 + 1); pmbar_init(w_empty + 8 * s, DQN); }
    for (int s = 0; s < MAX_BST; ++s) { pmbar_init(b_full + 8 * s, 1); pmbar_init(b_empty + 8 * s, 1); }
    for (int s = 0; s < MAX_AST; ++s) { pmbar_init(a_full + 8 * s, DQN / 2); pmbar_init(a_empty + 8 * s, 1); }
    pmbar_init(acc_full, EXACT ? DQN : 1);
    pmbar_init(acc_empty, DQN);
    for (int q = 0; q < 8; ++q) pmbar_init(xbar + 8 * q, max(1, 2 * (c.p - 1)));
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc((uint32_t)__cvta_generic_to_shared(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int rank = c.p > 1 ? (int)pcluster_rank() : 0;
  if (c.p > 1) {                        // the peers' barriers exist before anything arrives at them
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  bool failed = false;

  // the sums of 8 or 16 tokens from column `col` of the accumulator
  auto load8 = [&](uint32_t col, uint32_t (&v)[8]) {
    tmem_ld8(col, v);
    if (EXACT) {
      uint32_t u[8];
      tmem_ld8(col + 16, u);
      tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __float_as_uint(__uint_as_float(v[k]) + __uint_as_float(u[k]));
    }
  };
  // ---- epilogue of the block's tile number `count` for the de-quantiser warp that calls it; the two warps of a quadrant
  //      (`half`) share the chunks
  using Store = RowStore<T, !std::is_same<T, __half>::value>;
  auto epilogue_tile = [&](const Store& rs, int count, int half) {
    const int q = warp & 3;
    const uint32_t t_acc = tmem + ((uint32_t)(32 * q) << 16);
    const int n_ch = c.n / kTokChunk;
    tc_fence_after();
    if (c.p == 1) {                                            // nothing to exchange: sixteen tokens at a time
      for (int tk = 16 * half; tk < c.n; tk += 32) {
        uint32_t v[16];
        tmem_ld16(t_acc + (uint32_t)tk, v);
        tmem_ld_wait();
        float val[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) val[k] = __uint_as_float(v[k]);
        if (EXACT) {
          tmem_ld16(t_acc + 16, v);
          tmem_ld_wait();
#pragma unroll
          for (int k = 0; k < 16; ++k) val[k] += __uint_as_float(v[k]);
        }
        rs.store(p, tk, val);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) pmbar_arrive(acc_empty);
      return;
    }
    const size_t slot_f = (size_t)c.n * BMW;
    float* slots = c.partials + (size_t)(count & 1) * slot_f + 32 * q + lane;      // + block * 2 slots + token * BMW
    const float* block0 = slots + (size_t)((int)blockIdx.x - rank) * 2 * slot_f;
    // the sums of the chunks that other blocks finish
    float* mine = slots + (size_t)blockIdx.x * 2 * slot_f;
    for (int ch = half; ch < n_ch; ch += 2) {
      if (ch % c.p == rank) continue;
      uint32_t v[8];
      load8(t_acc + (uint32_t)(ch * kTokChunk), v);
      tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 8; ++k) __stcg(mine + (size_t)(ch * kTokChunk + k) * BMW, __uint_as_float(v[k]));
    }
    __syncwarp();
    // (barriers alternate from tile to tile: a peer may be a tile ahead before another peer's arrival has come in)
    const uint32_t xb = xbar + 32 * (count & 1) + 8 * q;
    if (lane < c.p && lane != rank) {
      asm volatile("fence.acq_rel.cluster;" ::: "memory");
      pmbar_arrive_peer(ppeer_addr(xb, (uint32_t)lane));
    }
    if (!pmbar_wait_cluster_warp(xb, (count >> 1) & 1, abort_flag)) { failed = true; return; }
    for (int own = half; rank + own * c.p < n_ch; own += 2) {
      const int ch = rank + own * c.p;
      uint32_t v[8];
      load8(t_acc + (uint32_t)(ch * kTokChunk), v);
      float val[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) val[k] = 0.f;
      const float* src = block0 + (size_t)(ch * kTokChunk) * BMW;
      for (int r0 = 0; r0 < c.p; r0 += 4) {                    // four blocks' sums in flight, added in rank order
        float a[4][8];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int k = 0; k < 8; ++k)
            a[r][k] = (r0 + r < c.p && r0 + r != rank) ? __ldcg(src + (size_t)(r0 + r) * 2 * slot_f + (size_t)k * BMW) : 0.f;
        tmem_ld_wait();
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int k = 0; k < 8; ++k) val[k] += r0 + r == rank ? __uint_as_float(v[k]) : a[r][k];
      }
      rs.store(p, ch * kTokChunk, val);
    }
    tc_fence_before();                                         // the accumulator is free for the next tile
    __syncwarp();
    if (lane == 0) pmbar_arrive(acc_empty);
  };
  auto row_store = [&](int tile) {
    const BFam& f = fam_of_tile(c, tile);
    const int r = 32 * (warp & 3) + lane;
    return Store(p, f.job, batch_row(c, p, f, tile, r).info, (r & 1) != 0);
  };

  BSegIter si;
  si.init(c, rank);
  BSeg sg;
  if (warp == 0) {
    // ===================================================================== activations
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // Only now may the next launch's blocks come in: as two launches fit an SM, triggering at entry let the launch after
    // the next one in as well, whose blocks then sat in slots that this launch's blocks needed.
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int s = 0, it = 0; uint32_t par = 1;
    const uint32_t box = (uint32_t)c.n * 128u;
    while (!failed && si.next(sg)) {
      for (int v0 = sg.s0 * KS; v0 < min(sg.s1 * KS, c.n_kb); v0 += KS / 2, ++it) {
        if (it >= c.bst && !pmbar_wait_warp(b_empty + 8 * s, par, abort_flag)) { failed = true; break; }
        const int nv = min(KS / 2, c.n_kb - v0);
        const uint32_t fb = b_full + 8 * s;
        if (elect_one()) {
          pmbar_expect_tx(fb, (uint32_t)nv * box);
          for (int i = 0; i < nv; ++i) {
            const int v = v0 + i;
            const int x = HEADS ? (((v / c.head_kb) * c.head_keep) & ~7) + (v % c.head_kb) * BK : v * BK;
            tma_box2(sbase + (uint32_t)(s * (KS / 2) + i) * box, &c.xmap, x, 0, fb);
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
    const uint64_t box_step = (uint64_t)(c.n * 8);             // a box of n * 128 bytes, in the descriptor's 16-byte units
    for (; !failed && si.next(sg); ++count) {
      if (!EXACT && count >= 1 && !pmbar_wait_warp(acc_empty, (count - 1) & 1, abort_flag)) { failed = true; break; }
      for (int v0 = sg.s0 * KS; v0 < sg.s1 * KS; v0 += KS / 2) {
        const int nv = c.n_kb - v0;                            // k-blocks of this half stage (none behind the last: only handed back)
        if ((nv > 0 && !pmbar_wait_warp(b_full + 8 * bs, bpar, abort_flag)) || !pmbar_wait_warp(a_full + 8 * as, apar, abort_flag)) {
          failed = true;
          break;
        }
        tc_fence_after();
        const uint32_t a0 = tmem + (uint32_t)(c.a_base + 64 * as);
        const uint64_t bd = smem_desc_sw128(sbase + (uint32_t)(bs * (KS / 2) * c.n) * 128u);
        if (elect_one()) {
#pragma unroll
          for (int i = 0; i < KS / 2; ++i) {
            if (i >= nv) break;
            if (EXACT) {                                       // (slot = half = accumulator)
              const uint32_t d = tmem + kExP + 32u * (uint32_t)as;
              const int kept = HEADS ? c.head_keep - ((v0 + i) % c.head_kb) * BK : BK;
#pragma unroll
              for (int k = 0; k < BK / 16; ++k) {
                const uint32_t more = (i > 0 || k > 0) ? 1u : 0u;
                umma_ts(d, a0 + 32 * i + 8 * k, bd + i * box_step + 2 * k, c.idesc, more);
                if (!HEADS || 16 * k < kept)                   // (kept channels are a multiple of 8)
                  umma_ts(d + 16, tmem + kExOnes + (HEADS && 16 * k + 8 == kept ? 4u : 0u), bd + i * box_step + 2 * k, c.idesc, more);
              }
              continue;
            }
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              umma_ts(tmem, a0 + 32 * i + 8 * k, bd + i * box_step + 2 * k, c.idesc, (v0 > sg.s0 * KS || i > 0 || k > 0) ? 1u : 0u);
          }
          umma_commit(a_empty + 8 * as);
          if (nv > 0) umma_commit(b_empty + 8 * bs);
        }
        __syncwarp();
        if (++as == c.n_ast) { as = 0; apar ^= 1; }
        if (nv > 0 && ++bs == c.bst) { bs = 0; bpar ^= 1; }
      }
      if (failed) break;
      if (!EXACT && elect_one()) umma_commit(acc_full);
      __syncwarp();
    }
  } else if (warp < DQ0) {
    // ===================================================================== loaders
    // Codes by TMA, issued by warp 2 (a box per lane).  (The first version copied them with cp.async, sixteen 16-byte
    // pieces per lane and stage: 1100 cycles of issue per stage and loader warp, which set the pace.)  Scales and
    // zero-points are two fp16 per row and stage at any row pitch: cp.async of 4 bytes, 64 rows per warp.
    const int r0 = (warp - LD_WARP0) * 64;
    const int G = p.sz_pitch ? p.sz_pitch : p.K / kGroup;
    bool sz_waited = p.sz_pitch == 0;              // (else the kernel in front makes the copy that these rows are)
    int s = 0, it = 0; uint32_t par = 1;
    while (!failed && si.next(sg)) {
      const BFam& f = fam_of_tile(c, sg.tile);
      const JobDev& js = p.job[f.job + ((f.mode == kBSwiglu && (lane & 1)) ? 1 : 0)];   // odd rows of a SwiGLU pair: the up matrix
      const int row0 = batch_row(c, p, f, sg.tile, r0 + lane).info.stored, row1 = batch_row(c, p, f, sg.tile, r0 + 32 + lane).info.stored;
      const __half* s0 = js.scales + c.kb_first / 2 + (size_t)max(row0, 0) * G;
      const __half* z0 = js.zeros + c.kb_first / 2 + (size_t)max(row0, 0) * G;
      const __half* s1 = js.scales + c.kb_first / 2 + (size_t)max(row1, 0) * G;
      const __half* z1 = js.zeros + c.kb_first / 2 + (size_t)max(row1, 0) * G;
      // this lane's box (warp 2): blocks beyond the family's last are left out
      const int tl = sg.tile - f.tile_begin;
      const CUtensorMap* tm = &c.wmap[&f - c.fam];
      int boxes, by = 0, bz = 0;
      if (f.per_tile == 0) {
        const int h = tl / f.tpb;
        by = (tl - h * f.tpb) * (f.mode == kBPlain ? BMW : BMW / 2);
        boxes = f.mode == kBPlain ? 1 : 2;
        bz = f.mode == kBRope ? 2 * h + lane : h;
        if (f.mode == kBSwiglu && lane == 1) tm = &c.wmap_up;
      } else {
        const int h0 = tl * f.per_tile, nb = min(f.per_tile, f.count - h0);
        boxes = f.mode == kBRope ? 2 * nb : nb;
        bz = (f.mode == kBRope ? 2 * h0 : h0) + lane;
      }
      for (int st = sg.s0; st < sg.s1; ++st, ++it) {
        if (it >= c.wst && !pmbar_wait_warp(w_empty + 8 * s, par, abort_flag)) { failed = true; break; }
        const uint32_t dst = sbase + (uint32_t)(c.off_w + s * WSTAGE);
        if (warp == LD_WARP0) {
          if (lane == 0) pmbar_expect_tx(w_full + 8 * s, (uint32_t)(boxes * f.box_rows) * 128u);
          __syncwarp();
          if (lane < boxes) tma_box_3d(dst + (uint32_t)(lane * f.box_rows) * 128u, tm, c.kb_first * 32 + st * 128, by, bz, w_full + 8 * s);
        }
        if (!sz_waited) {
          asm volatile("griddepcontrol.wait;" ::: "memory");
          sz_waited = true;
        }
        const uint32_t sd = dst + WST_BYTES + (uint32_t)((r0 + lane) * 4);
        if (row0 >= 0) {
          bcp_async4(sd, s0 + st * 2);
          bcp_async4(sd + BMW * 4, z0 + st * 2);
        }
        if (row1 >= 0) {
          bcp_async4(sd + 128, s1 + st * 2);
          bcp_async4(sd + BMW * 4 + 128, z1 + st * 2);
        }
        bcp_async_arrive(w_full + 8 * s);
        if (++s == c.wst) { s = 0; par ^= 1; }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (failed) {                           // let the copies still armed land before the block goes away
      for (int j = it > c.wst ? it - c.wst : 0; j < it; ++j)
        for (int i = 0; i < kPWait && !pmbar_try(w_full + 8 * (j % c.wst), (j / c.wst) & 1); ++i) {}
    }
  } else {
    // ===================================================================== de-quantisers, then the tile's epilogue
    // The tcgen05.st of a half stage completes while the first part of the next is converted.
    const int q = warp & 3, half = (warp - DQ0) >> 2;
    const int r = 32 * q + lane;
    const uint32_t s_off = (uint32_t)(WST_BYTES + r * 4 + half * 2);
    const uint32_t a_lane = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)c.a_base;
    int ws = 0; uint32_t wpar = 0;
    int as = half, use = 0;                      // this warp's next A slot, the slot's earlier uses (n_ast >= 2)
    int stored_as = -1;                          // A slot whose tcgen05.st is still to be announced
    auto announce = [&]() {
      if (stored_as < 0) return;
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) pmbar_arrive(a_full + 8 * stored_as);
      stored_as = -1;
    };
    float sum[16], g_s = 0.f, g_cz = 0.f;        // EXACT: the tile's sums, scale and offset of the group whose sums are due
    bool due = false;
    auto add_group = [&]() {                     // (behind the wait for the slot whose MMAs these are)
#pragma unroll
      for (int k0 = 0; k0 < 16; k0 += 8) {
        uint32_t v[8], u[8];
        tmem_ld8(a_lane - (uint32_t)c.a_base + kExP + 32 * half + k0, v);
        tmem_ld8(a_lane - (uint32_t)c.a_base + kExP + 32 * half + 16 + k0, u);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 8; ++k) sum[k0 + k] = fmaf(g_s, __uint_as_float(v[k]), fmaf(g_cz, __uint_as_float(u[k]), sum[k0 + k]));
      }
    };
    if (EXACT && half == 0) {                    // (complete before this warp's first arrival for the MMA warp)
      const uint32_t t = a_lane - (uint32_t)c.a_base + kExOnes;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(t + 8 * k), "r"(k ? 0u : 0x3c003c00u) : "memory");
      tmem_st_wait();
      tc_fence_before();
    }
    for (int count = 0; !failed && si.next(sg); ++count) {
      if (EXACT) {
        due = false;
#pragma unroll
        for (int k = 0; k < 16; ++k) sum[k] = 0.f;
      }
      const int sr = batch_row(c, p, fam_of_tile(c, sg.tile), sg.tile, r).smem_row;
      const uint32_t x_row = (uint32_t)(sr * 128), x_sw = (uint32_t)((half * 4) ^ (sr & 7)) * 16;   // piece i: x_sw ^ (16 i)
      uint32_t w[16];
      __half sc, zp;
      auto fetch = [&]() -> bool {               // codes, scale and zero-point of the next stage of the ring
        if (!pmbar_wait_warp(w_full + 8 * ws, wpar, abort_flag)) return false;
        const uint32_t src = sbase + (uint32_t)(c.off_w + ws * WSTAGE);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[4 * i]), "=r"(w[4 * i + 1]), "=r"(w[4 * i + 2]), "=r"(w[4 * i + 3])
                       : "r"(src + x_row + (x_sw ^ (16 * i))) : "memory");
        unsigned short sh, zh;
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(sh) : "r"(src + s_off) : "memory");
        asm volatile("ld.shared.u16 %0, [%1];" : "=h"(zh) : "r"(src + s_off + BMW * 4) : "memory");
        sc = __ushort_as_half(sh); zp = __ushort_as_half(zh);
        return true;
      };
      // The slot goes back only after its values are in registers: an arrival issued behind the loads can overtake them, and
      // the next stage's copy then lands under the reads (wrong rows in contractions long enough for the ring to wrap).  So the
      // arrival stands behind the tcgen05.st that takes the last of the converted codes (without EXACT the scale and the
      // zero-point are in those too, with it the arrival takes its address through them): a dependency, where the order of the
      // conversions, which are plain arithmetic, was the compiler's to choose.  Loading the next stage before that store instead
      // took 3 % (M = 64) to 5 % (M = 16) longer per
      // Llama-3-8B layer; launches of one or two stages per block were 0.05 - 0.1 us of 5 - 8 us shorter so.
      auto release = [&]() {
        const uint32_t seen = EXACT ? (__float_as_uint(g_s) | __float_as_uint(g_cz)) & c.never : 0u;
        __syncwarp();
        if (lane == 0) pmbar_arrive(w_empty + 8 * ws + seen);
        if (++ws == c.wst) { ws = 0; wpar ^= 1; }
      };
      if (!fetch()) { failed = true; break; }
      for (int st = sg.s0; st < sg.s1; ++st) {
        const __half2 s2 = __half2half2(sc);
        const __half2 cz2 = __float2half2_rn((8.f - __half2float(zp)) * __half2float(sc));
        uint32_t o[32];
        HeadSpan hs[2] = {{0, 0, BK}, {0, 0, BK}};                 // of the half stage's k-blocks
        if (HEADS) { hs[0] = head_span<HEADS == 2>(c, st * KS + 2 * half); hs[1] = head_span<HEADS == 2>(c, st * KS + 2 * half + 1); }
        auto convert = [&](int j0) {             // words j0 .. j0 + 3 of the sixteen
#pragma unroll
          for (int i = j0; i < j0 + 4; ++i) {
            const int k = i & 7, b = i >> 3;
            uint32_t wi = w[i];
            if (HEADS == 2)                      // (k-block b is a head's first unless heads have two and b is 1)
              wi = __funnelshift_l(k > 0 || (b == 1 && hs[1].lead != hs[1].shift) ? w[i > 0 ? i - 1 : 0] : 0u, w[i], 4 * hs[b].shift);
            const uint4 d = HEADS && k * 8 >= hs[b].end ? make_uint4(0, 0, 0, 0) : EXACT ? codes_word(wi) : dequant_word(wi, s2, cz2);
            const bool no_lo = HEADS == 2 && k == 0 && hs[b].lead != 0, no_hi = HEADS == 2 && k * 8 + 4 == hs[b].end;
            o[4 * k] = no_lo ? 0u : d.x; o[4 * k + 1] = no_lo ? 0u : d.y; o[4 * k + 2] = no_hi ? 0u : d.z; o[4 * k + 3] = no_hi ? 0u : d.w;
          }
        };
        convert(0);
        announce();
        convert(4);
        // (the slot's previous user: the half stage n_ast earlier.  This warp wrote the half stage two earlier after a wait
        //  that implies every half stage up to 2 + n_ast earlier is done, so the parity cannot be two phases old.)
        if (use > 0 && !pmbar_wait_warp(a_empty + 8 * as, (use - 1) & 1, abort_flag)) { failed = true; break; }
        tc_fence_after();
        tmem_st32(a_lane + (uint32_t)(64 * as), o);
        if (EXACT) {
          if (due) add_group();
          g_s = __half2float(sc);
          g_cz = (8.f - __half2float(zp)) * g_s;
          due = st * KS + half * (KS / 2) < c.n_kb;
        }
        convert(8);
        convert(12);
        tmem_st32(a_lane + (uint32_t)(64 * as + 32), o);
        release();
        if (st + 1 < sg.s1 && !fetch()) { failed = true; break; }
        stored_as = as;
        as += 2;
        if (as >= c.n_ast) { as -= c.n_ast; ++use; }
      }
      if (failed) break;
      announce();
      asm volatile("griddepcontrol.wait;" ::: "memory");       // outputs, positions and workspace: after the preceding kernel
      const Store rs = row_store(sg.tile);               // (several dependent loads, while the last MMAs run)
      if (EXACT) {
        if (!pmbar_wait_warp(a_empty + 8 * as, (use - 1) & 1, abort_flag)) { failed = true; break; }
        tc_fence_after();
        if (due) add_group();
        if (count >= 1 && !pmbar_wait_warp(acc_empty, (count - 1) & 1, abort_flag)) { failed = true; break; }
        tc_fence_after();
        uint32_t v[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = __float_as_uint(sum[k]);
        tmem_st16(a_lane - (uint32_t)c.a_base + 16 * half, v);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) pmbar_arrive(acc_full);
      }
      if (!pmbar_wait_warp(acc_full, count & 1, abort_flag)) { failed = true; break; }
      epilogue_tile(rs, count, half);
    }
  }
  if (failed && lane == 0) atomicExch(c.status, UNIQL_ERR_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, kTmemCols);
  if (c.p > 1) {                        // no block leaves while a peer may still arrive at its barriers
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// -------------------------------------------------------------------------------- host side
// Row families of the launch, or 0 when there are more than it holds.
int batch_families(const Params& p, BatchCfg* c) {
  int n = 0, tiles = 0;
  for (int j = 0; j < p.n_jobs; ++j) {
    const JobDev& jb = p.job[j];
    if (jb.pair == 2) continue;                                      // its rows ride in the tiles of the job before
    const int nf = jb.rope.enabled ? 1 : jb.omap.n_fam;
    for (int k = 0; k < nf; ++k) {
      if (n == kMaxBF) return 0;
      BFam f;
      memset(&f, 0, sizeof(f));
      f.tile_begin = tiles; f.job = j;
      int rows;                                                      // rows (pairs) that a tile has room for
      if (jb.rope.enabled) {
        f.mode = kBRope; rows = BMW / 2;
        f.keep = jb.rope.head_keep / 2; f.count = jb.rope.n_heads; f.start = 0; f.period = jb.rope.head_dim;
      } else {
        const Fam& a = jb.omap.fam[k];
        f.mode = jb.pair == 1 ? kBSwiglu : kBPlain; rows = jb.pair == 1 ? BMW / 2 : BMW;
        if (jb.pair == 1 && (nf != 1 || a.count != 1)) return 0;
        f.keep = a.keep; f.count = a.count; f.start = a.start; f.period = a.count > 1 ? a.period : a.keep; f.out_base = jb.omap.base[k];
      }
      if (f.keep > rows || f.count == 1) {
        f.box_rows = rows; f.per_tile = 0; f.tpb = (f.keep + rows - 1) / rows;
        tiles += f.tpb * f.count;
      } else {
        f.box_rows = (f.keep + 7) / 8 * 8;                           // (the swizzle pattern repeats every 8 rows)
        f.per_tile = rows / f.box_rows; f.tpb = 1;
        if (f.per_tile < 1) f.per_tile = 1;
        tiles += (f.count + f.per_tile - 1) / f.per_tile;
      }
      if (c) c->fam[n] = f;
      ++n;
    }
  }
  if (c) { c->n_fam = n; c->n_tiles = tiles; }
  return n;
}

typedef void (*BatchKernel)(Params, BatchCfg);
BatchKernel batch_instance(bool bf16, int heads, bool exact) {
  if (bf16) return heads ? batch_kernel<__nv_bfloat16, 1, false> : batch_kernel<__nv_bfloat16, 0, false>;
  if (exact) return heads ? batch_kernel<__half, 1, true> : batch_kernel<__half, 0, true>;
  return heads == 2 ? batch_kernel<__half, 2, false> : heads ? batch_kernel<__half, 1, false> : batch_kernel<__half, 0, false>;
}

struct BLaunch {
  cudaLaunchConfig_t lc;
  cudaLaunchAttribute attr[2];
  BLaunch(int grid, int p, size_t smem, cudaStream_t stream) {
    memset(this, 0, sizeof(*this));
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(NTHB);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    lc.attrs = attr;
    if (p > 1) {
      attr[lc.numAttrs].id = cudaLaunchAttributeClusterDimension;
      attr[lc.numAttrs].val.clusterDim.x = p;
      attr[lc.numAttrs].val.clusterDim.y = attr[lc.numAttrs].val.clusterDim.z = 1;
      ++lc.numAttrs;
    }
    if (opt(kOptPdl)) {
      attr[lc.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[lc.numAttrs].val.programmaticStreamSerializationAllowed = 1;
      ++lc.numAttrs;
    }
  }
};

constexpr int kMaxP = 8;
// Clusters of p blocks that the device holds at once (two blocks per SM), asked once per device.
struct Residency { bool known = false; int clusters[kMaxP + 1]; };
int residency(Residency* out) {
  static std::mutex mu;
  static Residency dev_res[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return UNIQL_ERR_CUDA;
  std::lock_guard<std::mutex> lock(mu);
  Residency& r = dev_res[dev];
  if (!r.known) {
    for (int k = 0; k < 12; ++k)
      if (cudaFuncSetAttribute(batch_instance(k & 1, k >> 2, k & 2), cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemAlone) != cudaSuccess)
        return UNIQL_ERR_CUDA;
    const int sms = device_sms();
    r.clusters[0] = 0;
    r.clusters[1] = 2 * sms;
    for (int p = 2; p <= kMaxP; ++p) {
      BLaunch l(2 * sms / p * p, p, kSmemBatch, nullptr);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, batch_instance(false, 0, false), &l.lc) != cudaSuccess) { cudaGetLastError(); n = 0; }
      r.clusters[p] = n < 2 * sms / p ? n : 2 * sms / p;
    }
    r.known = true;
  }
  *out = r;
  return UNIQL_OK;
}

}  // namespace

// Up to 128 rows; an input map whose k-blocks are all visited from a 256-channel boundary on (a leading block, or heads
// that keep a part of every k-block); scale rows that can be copied two groups at a time.
int batch_supported(const Params& p) {
  if (p.M < 1 || p.M > 128 || (p.K % (2 * kGroup) != 0 && p.sz_pitch == 0) || p.imap.n_fam != 1) return 0;
  const Fam& a = p.imap.fam[0];
  if (a.count == 1) {
    if (a.start != 0) return 0;
  } else if (a.start % (KS * BK) != 0 || a.period % BK != 0 || a.keep % 4 != 0 || a.keep <= a.period - BK) {
    return 0;
  } else if (a.keep % 8 != 0 && (p.M <= 16 || p.dt != UNIQL_F16 || a.period > 2 * BK)) {
    return 0;                            // (heads of one or two k-blocks, read in place: bf16 activations are copied anyway)
  }
  if ((p.ldx % 8) != 0 || (((uintptr_t)p.x) & 15) != 0) return 0;
  for (int j = 0; j < p.n_jobs; ++j)
    if ((((uintptr_t)p.job[j].scales) | ((uintptr_t)p.job[j].zeros)) & 3) return 0;
  return batch_families(p, nullptr) > 0;
}

// What a launch cannot do without (the header and the fp16 copy of bf16 activations), and with room for every split.
size_t batch_workspace_min(bool copy_x, int M, int k_in) {
  const size_t header = (decode_workspace_header_bytes() + 255) & ~(size_t)255;
  return copy_x ? header + (size_t)M * ((k_in + 63) / 64 * 64) * 2 + 256 : header;
}
size_t batch_workspace_bytes(int M, int K) {
  const size_t n = (M + 15) / 16 * 16;
  return batch_workspace_min(true, M, K) + (size_t)2 * device_sms() * 2 * n * BMW * 4;
}

// Whether an fp16 launch of up to 16 rows goes to the EXACT instance instead of the decode kernel.  From twelve rows: the
// decode kernel's activation traffic grows with the rows (a layer 8 - 12 % from nine to sixteen), this instance's does not.
// Measured at 12 / 16 rows, decode kernel -> here, the whole layer in microseconds: Qwen2.5-7B 84.2 -> 71.7 / 90.6 -> 71.4,
// Mamba2-2.7B 29.0 -> 22.5 / 31.4 -> 22.5, Llama-3-8B 76.0 -> 71.6 / 79.6 -> 71.7, at keep 0.75 71.9 -> 63.6 / 74.9 -> 63.5, at keep
// 0.65 68.6 -> 66.6 / 72.9 -> 67.2; over five keep rates from 0.55 the decode kernel is nowhere ahead by more than 1 %.
// Not where kept blocks of output rows are no multiple of 8: the launch that reads those channels then stays on the decode
// kernel (4-channel boundaries), whose blocks need a whole SM and cannot come in beside this kernel's (Mamba2 mixer at keep
// 0.8 29.5 -> 30.7 us).  Rotated heads excepted: there the other four launches of a layer outweigh that.
int exact_batch(const Params& p) {
  if (p.dt != UNIQL_F16 || p.M < 12 || p.M > 16 || !batch_supported(p) || !prefill_supported(p)) return 0;
  // (an option of the decode kernel that is set asks for that kernel)
  if (opt(kOptDecodeKp) != 0 || opt(kOptDecodeRp) != 0 || opt(kOptDecodeStages) != 0 || opt(kOptDecodeNarrow) != -1 || opt(kOptDecodeXstream) != -1 ||
      opt(kOptDecodeXcluster) != -1 || opt(kOptDecodeI8) != 1 || opt(kOptDecodeSplitBatch) != 2)
    return 0;
  for (int j = 0; j < p.n_jobs; ++j) {
    if (p.n_jobs > 1 && p.job[0].rope.enabled) break;
    for (int k = 0; k < p.job[j].omap.n_fam; ++k)
      if (p.job[j].omap.fam[k].count > 1 && p.job[j].omap.fam[k].keep % 8 != 0) return 0;
  }
  return 1;
}

// Measured (Llama-3-8B, M = 17 / 64 / 128, against the prefill kernel): q|k|v 18.5 / 21.5 / 21.4 -> 11.5 / 13.0 / 17.2 us, o_proj
// 20.2 / 24.4 / 27.6 -> 9.1 / 13.2 / 12.0 us, down projection 36 / 36 / 40 -> 18 / 17 / 21 us, whole layer at M = 64 and keep
// 0.85 137 -> 69 us.  What bounds it now: the issue slots of SMs that hold two tiles (0.65 us per stage and block alone on
// its SM, 1.05 us for two), and 7 us per launch before the first and after the last stage.
int launch_batch(const Params& p, const LaunchCfg& cfg) {
  BatchCfg c;
  memset(&c, 0, sizeof(c));
  if (batch_families(p, &c) < 1 || c.n_tiles < 1) return UNIQL_ERR_SHAPE;
  c.n = (p.M + 15) / 16 * 16;
  const Fam& a = p.imap.fam[0];
  const int kbh = (a.keep + BK - 1) / BK;
  c.n_kb = kbh * a.count;
  c.spt = (c.n_kb + KS - 1) / KS;
  c.kb_first = a.start / BK;
  c.head_kb = a.count > 1 ? kbh : 0;
  c.head_keep = a.keep;
  c.heads = a.count == 1 ? 0 : a.keep % 8 == 0 ? 1 : 2;
  // fp32 accumulate, A and B fp16, both K-major, N tokens, 128 rows
  c.idesc = (1u << 4) | ((uint32_t)(c.n >> 3) << 17) | ((uint32_t)(BMW >> 4) << 24);
  c.exact = p.M <= 16 && p.dt != UNIQL_BF16;
  c.n_ast = c.n <= 64 && !c.exact ? 3 : 2;
  c.a_base = c.exact ? (int)kExA : c.n <= 64 ? 64 : 128;
  // shared memory: two to four half stages of activations, the rest for the codes (HBM's latency is theirs to cover)
  c.bst = c.n > 64 ? 2 : (c.n > 32 ? 3 : 4);
  c.off_w = c.bst * (KS / 2) * c.n * 128;
  const int room = kSmemBatch - 1024 - 512 - c.off_w;
  c.wst = room / WSTAGE < MAX_WST ? room / WSTAGE : MAX_WST;
  c.off_bar = c.off_w + c.wst * WSTAGE;
  size_t smem = 1024 + (size_t)c.off_bar + 512;
  c.status = reinterpret_cast<int*>(reinterpret_cast<unsigned char*>(cfg.workspace) + decode_status_offset());
  size_t used = (decode_workspace_header_bytes() + 255) & ~(size_t)255;
  const void* x = p.x;
  int ldx = p.ldx;
  const bool copy_x = p.dt == UNIQL_BF16 && !p.x_f16;
  if (copy_x) {                                 // (room for the copy was checked by the caller)
    ldx = (p.k_in + 63) / 64 * 64;
    x = reinterpret_cast<unsigned char*>(cfg.workspace) + used;
    used = (used + (size_t)p.M * ldx * 2 + 255) & ~(size_t)255;
  }
  // The split: p blocks per tile where that shortens the longest block's work.  In microseconds: the rounds of the clusters
  // that fit, a p-th of a tile's stages each at 0.65 (one block per SM) or 1.05 (two), and 3 for the exchange.
  Residency res;
  int rc = residency(&res);
  if (rc != UNIQL_OK) return rc;
  const int env_grid = opt(kOptPrefillGrid), env_split = opt(kOptPrefillStreamk);
  int best = 1, best_clusters = 1;
  double best_cost = 1e30;
  for (int k = 1; k <= kMaxP; ++k) {
    int fit = res.clusters[k];
    if (env_grid >= 1 && env_grid / k < fit) fit = env_grid / k;              // tests: several tiles per block on small problems
    if (fit < 1 || k > c.spt) continue;
    const int clusters = c.n_tiles < fit ? c.n_tiles : fit;
    if (k > 1 && (env_split == 0 || cfg.ws_bytes < used + (size_t)clusters * k * 2 * c.n * BMW * 4)) continue;
    const int rounds = (c.n_tiles + fit - 1) / fit;
    double cost = rounds * ((double)c.spt / k * (clusters * k > device_sms() ? 1.05 : 0.65) + (k > 1 ? 3.0 : 1.0));
    if (env_split >= 1 && env_split <= 3 && k > 1) cost *= 1e-3;              // tests: split wherever it is possible
    if (env_split == 10 + k) cost = 0.0;                                     // ... over k blocks
    if (cost < best_cost) { best_cost = cost; best = k; best_clusters = clusters; }
  }
  c.p = best;
  c.partials = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(cfg.workspace) + used);
  if (copy_x) {
    rc = launch_x_to_f16(p.x, p.ldx, p.M, p.k_in, const_cast<void*>(x), ldx, cfg.stream);
    if (rc != UNIQL_OK) return rc;
  }
  const int x_extent = (c.kb_first + c.n_kb) * (BK / 2);     // bytes of a row up to the last visited k-block
  for (int k = 0; k < c.n_fam; ++k) {
    const BFam& f = c.fam[k];
    const JobDev& jb = p.job[f.job];
    const bool rope = f.mode == kBRope;
    rc = encode_w_map(&c.wmap[k], jb.w + (size_t)f.start * (p.K / 2), p.K, x_extent, f.keep, rope ? 2 * f.count : f.count,
                      rope ? f.period / 2 : f.period, f.box_rows);
    if (rc == UNIQL_OK && f.mode == kBSwiglu)
      rc = encode_w_map(&c.wmap_up, p.job[f.job + 1].w + (size_t)f.start * (p.K / 2), p.K, x_extent, f.keep, 1, f.keep, f.box_rows);
    if (rc != UNIQL_OK) return rc;
  }
  rc = encode_x_map(&c.xmap, x, p.k_in, p.M, ldx, c.n, false);
  if (rc != UNIQL_OK) return rc;
  // Shared tiles of at most a block per SM, planned at the pace of one: where the launch before still holds half of some
  // SMs, the other halves are free first and the blocks came in two to an SM, at 1.05 us per stage instead of 0.65, with
  // half of the SMs empty (SwiGLU block of Llama-3-8B, M = 64, keep 0.85: 47.4 -> 43.6 us; Qwen2.5-7B layer, 100 rows 95 -> 88
  // us).  Asking for a little more than half of the SM spreads them.  Ten stages are where that pays for the later start:
  // with four to eight (q|k|v, o_proj) a launch gains more from loading beside its predecessor (9.0 against 11.5 us).
  if (c.p > 1 && best_clusters * c.p <= device_sms() && c.spt >= 10 * c.p) smem = kSmemAlone;
  for (;;) {
    BLaunch l(best_clusters * c.p, c.p, smem, cfg.stream);
    const bool refused = c.p > 1 && opt(kOptPrefillPair) == 3;                 // tests
    if (!refused && cudaLaunchKernelEx(&l.lc, batch_instance(p.dt == UNIQL_BF16, c.heads, c.exact != 0), p, c) == cudaSuccess) return UNIQL_OK;
    cudaGetLastError();
    if (c.p == 1) return UNIQL_ERR_CUDA;
    c.p = 1;                                                                   // clusters cannot be launched here: whole tiles
    best_clusters = c.n_tiles < res.clusters[1] ? c.n_tiles : res.clusters[1];
    smem = 1024 + (size_t)c.off_bar + 512;
  }
}

}  // namespace uniql
