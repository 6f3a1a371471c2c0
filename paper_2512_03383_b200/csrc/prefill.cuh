// Tensor-core kernels of the pruned 4-bit linear layer for more than 128 rows, and for smaller batches that neither the decode
// nor the batch kernel takes, sm_100a: a dense contraction on the fifth-generation tensor cores (tcgen05.mma, accumulators in
// tensor memory).  Here: what the two of them share.  Block pairs stand in prefill.cu with the planner, single blocks in
// single.cu.  They are two kernels and not one with a switch: as instances of one template the registers of the pairs' code
// and epilogue reached the loops of the others (80 registers with spills; a k-block 0.485 -> 0.52 us, the read-back of 26 parts
// of a tile 70 -> 91 us).
//
// Orientation.  The packed weights are four times smaller than the activations, so the weight side
// takes the MMA's M dimension (128 retained weight rows per tile, de-quantised once per tile and
// k-block) and the tokens its N dimension (up to 256 per tile): D[row][token] += W[row][k] x[token][k].
//
// Roles inside a block (one persistent block per SM, tiles taken round-robin):
//   warp 0       TMA producer: boxes [64 k x BN tokens] of activations into a ring (128-byte swizzle);
//                one box per k-block, or two where a tile takes both accumulators (512 tokens)
//   warp 1       allocates tensor memory; one lane issues the MMAs of a k-block (4 x K=16 per box) and commits
//                them to the "empty" barriers of what they read and, at the end of a tile, to "accumulator full"
//   warps 4..7   epilogue: tcgen05.ld the fp32 accumulators (warp w owns TMEM lanes 32(w-4).., a lane
//                is a tile row and holds 32 tokens of it per pass), bias, rotary embedding on the
//                retained pair (Section 3.2; the pair's two rows are neighbouring lanes and swap
//                values by shuffle), one rounding, stores of 32 consecutive outputs of a token per
//                warp; two accumulator buffers of 256 columns let the epilogue of tile i overlap
//                the MMAs of tile i+1 (tiles of 512 tokens use both and hand them back one by one);
//                the epilogue of a block's last tile is shared with the de-quantiser warps, idle by then
//   warps 8..23  de-quantisers: the twelve of them whose scheduler does not host the MMA warp (warp % 4 != 1), two
//                teams of six warps on alternate stages (pairs with one box per tile: all sixteen); a thread converts
//                32 codes of a weight row per item -- nibbles to fp16 by magic number, (q-8) exact, then one fp16 FMA
//                (q-8)*s + fp16(s*(8-z)) -- and writes them into the A-operand stage in the canonical K-major
//                128-byte-swizzled layout; the packed codes of the next k-block are already in registers.  All sixteen
//                share the epilogue of the block's last segment.
// Launched with programmatic stream serialization: what a block does before griddepcontrol.wait (barriers, tensor
// memory, the first weight stages) touches nothing a preceding kernel may still read or write.
// On-device pruning (Section 3.4) is index arithmetic: tile rows are compact output channels mapped to
// stored rows per thread; the input side is the leading k_in channels (the TMA tensor ends at k_in, so
// the tail of the last k-block is zero activations) or the kept channels of every head.
// bf16 activations: bf16 weights would carry 2^-9 relative rounding error each, which alone spends the
// 2e-3 error budget; instead both operands are fp16, from a converted copy of the activations in the workspace or, where
// that has no room, converted in place by the de-quantisers of the one-block kernel (exact in fp16's range, saturating beyond).
//
// Every mbarrier wait is bounded; on expiry the block raises a flag, every role leaves its loop, the
// status word of the workspace is set, tensor memory is released and the block returns.
#pragma once
#include <cuda.h>

#include "tc.cuh"

namespace uniql {

constexpr int MAXBN = 256;          // tokens per tile (MMA N), at most
constexpr int A_BYTES = BMW * BK * 2;        // 16 KB
constexpr int B_BYTES = MAXBN * BK * 2;      // 32 KB
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
// Launch of the one-block kernel (conv: activations converted in the kernel).  UNIQL_ERR_UNSUPPORTED: the clusters that
// c.pair_split asks for cannot all be resident, or were refused.
int launch_one_block(const Params& p, const PrefillCfg& c, int grid, bool conv, cudaStream_t stream);

}  // namespace uniql
