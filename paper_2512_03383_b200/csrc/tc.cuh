// What the tensor-core kernels share: PTX wrappers (barriers, TMA, tcgen05), the rows of a weight tile, nibbles to fp16,
// and the epilogue of a thread that owns one weight row of a tile.
#pragma once
#include <stdint.h>

#include "common.cuh"

namespace uniql {

constexpr int BMW = 128;            // weight rows per tile (MMA M)
constexpr int BK = 64;              // input channels per k-block: 128 bytes of fp16 / bf16, one swizzle row
constexpr int kPWait = 1 << 20;     // polls of a bounded wait

// ---------------------------------------------------------------------------------------- PTX
__device__ inline void pmbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ inline void pmbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ inline void pmbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ inline bool pmbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// A bounded wait has one answer per warp: a warp whose lanes disagreed about an expired wait -- the phase may complete between two
// lanes' last polls -- would part, and its next warp-wide instruction would wait for the missing lanes.  The vote also brings the lanes
// together in front of that instruction.  Only a thread that waits on its own takes the form without it.  (What the vote costs where it is
// asked for every k-block, the de-quantisers of the block pairs: 0.1 - 0.7 % of a pass; Llama-3-8B layer at 512 rows 193.0 -> 193.8 us.)
// `relaxed`: sleep between polls (roles that run several stages ahead and must not steal issue slots)
__device__ inline bool pmbar_wait_lane(uint32_t bar, uint32_t parity, volatile int* abort_flag, bool relaxed = false) {
  for (int i = 0; i < kPWait; ++i) {
    if (pmbar_try(bar, parity)) return true;
    if (relaxed) __nanosleep(200);
    if ((i & 63) == 63 && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
__device__ inline bool pmbar_poll_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, bool relaxed = false) {
  return __all_sync(0xffffffffu, pmbar_wait_lane(bar, parity, abort_flag, relaxed));
}
// As pmbar_try, but the hardware may suspend the thread for up to a microsecond until the phase completes.
__device__ inline bool pmbar_try_suspend(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(1000u) : "memory");
  return ok != 0;
}
// pmbar_poll_warp with these polls, for the roles whose next step hangs on the phase.
__device__ inline bool pmbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, pmbar_try(bar, parity))) return true;
  bool ok = false;
  for (int i = 0; i < kPWait && !ok; ++i) {
    ok = pmbar_try_suspend(bar, parity);                // (polling without a suspend time costs issue slots: 3 % of a launch)
    if (!ok && (i & 63) == 63 && *abort_flag) break;
  }
  if (!ok) *abort_flag = 1;
  return __all_sync(0xffffffffu, ok);
}
// ---- clusters of two (a tile's contraction split over a pair of blocks)
__device__ inline uint32_t pcluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of `addr` (shared memory of this block) in block `rank` of the cluster
__device__ inline uint32_t ppeer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// generic address of `ptr` (shared memory of this block) in block `rank` of the cluster
__device__ inline float* ppeer_generic(void* ptr, uint32_t rank) {
  unsigned long long r;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<unsigned long long>(ptr)), "r"(rank));
  return reinterpret_cast<float*>(r);
}
template <int STRIDE, int K = 0>
__device__ inline void pld_add_f32x16(uint32_t base, const uint32_t (&v)[16], float (&val)[16]) {
  if constexpr (K < 16) {
    float o;
    asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(o) : "r"(base), "n"(K * STRIDE) : "memory");
    val[K] = __uint_as_float(v[K]) + o;
    pld_add_f32x16<STRIDE, K + 1>(base, v, val);
  }
}
// Arrival on a barrier of the other block, at the scope of this one: for signals that hand over nothing but the tensor
// core's own operands and accumulators (written with fence.proxy.async, or read with tcgen05.fence, before this).  A
// release at cluster scope waits for everything the thread has in flight, which cost 0.4 us per k-block.
__device__ inline void pmbar_signal_peer(uint32_t addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ inline void pmbar_arrive_peer(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ inline bool pmbar_try_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ inline bool pmbar_wait_cluster_lane(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  for (int i = 0; i < kPWait; ++i) {
    if (pmbar_try_cluster(bar, parity)) return true;
    __nanosleep(20);
    if ((i & 63) == 63 && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
__device__ inline bool pmbar_wait_cluster_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return __all_sync(0xffffffffu, pmbar_wait_cluster_lane(bar, parity, abort_flag));
}
__device__ inline void tma_box2(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ inline void tma_box_3d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
// ---- two blocks of a cluster on one MMA (cta_group::2).  A box into this block's shared memory, counted on a barrier of
// the first block (`bar`: its address in the cluster window).
__device__ inline void tma_box2_pair(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(tm), "r"(x), "r"(y), "r"(bar) : "memory");
}
__device__ inline void tmem_alloc_pair(uint32_t smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// arrives on the barrier at this offset in both blocks (`mask`: their ranks in the cluster) when all pair MMAs issued so far
// by this thread have completed
__device__ inline void umma_commit_pair(uint32_t bar, unsigned short mask) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(bar), "h"(mask) : "memory");
}
__device__ inline void tmem_alloc(uint32_t smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_dst), "r"(ncols) : "memory");
}
__device__ inline void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ inline void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ inline void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ inline void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D[tmem] (+)= A[smem desc] * B[smem desc] over a k-block of 64: four MMAs, 32 bytes along K each (+2 in the descriptors'
// address field); accumulate == 0: the first one overwrites D.  One block of code: the issuing warp's loop is one chain of
// instructions, so every one of them counts.  PAIR: cta_group::2 -- D is 256 rows, 128 in each block's tensor memory, A 128
// rows and B half of the tokens in each block's shared memory at the same offsets; issued by the first block only.
template <bool PAIR>
__device__ inline void umma_kblock(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  if (PAIR)
    asm volatile(
        "{\n\t.reg .pred p, t;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
        "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
        "add.s64 a1, %1, 2;\n\tadd.s64 b1, %2, 2;\n\tadd.s64 a2, %1, 4;\n\tadd.s64 b2, %2, 4;\n\tadd.s64 a3, %1, 6;\n\tadd.s64 b3, %2, 6;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %3, t;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], a2, b2, %3, t;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], a3, b3, %3, t;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p, t;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
        "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
        "add.s64 a1, %1, 2;\n\tadd.s64 b1, %2, 2;\n\tadd.s64 a2, %1, 4;\n\tadd.s64 b2, %2, 4;\n\tadd.s64 a3, %1, 6;\n\tadd.s64 b3, %2, 6;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a1, b1, %3, t;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a2, b2, %3, t;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], a3, b3, %3, t;\n\t}"
        ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate) : "memory");
}
// one lane of a converged warp (always the same one)
__device__ inline bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
// arrives on `bar` when all MMAs issued so far by this thread have completed
__device__ inline void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 consecutive fp32 columns of this thread's TMEM lane
__device__ inline void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
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
__device__ inline void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ inline void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr) : "memory");
}
__device__ inline void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ inline void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major tile whose rows are 128 bytes (64 fp16/bf16), 128-byte
// swizzle: 8-row groups 1024 bytes apart (stride byte offset), leading byte offset unused (1),
// descriptor version 1 (sm_100), layout type 2 (SWIZZLE_128B).
__device__ inline uint64_t smem_desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ inline uint32_t pand_or(uint32_t a, uint32_t mask, uint32_t magic) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(mask), "r"(magic));
  return d;
}

// ---------------------------------------------------------------------------------------- tile rows
// Row r (0..127) of local weight tile `tl` of a job: stored weight row, or -1 when the row is empty.
// Rope jobs: rows 2i and 2i + 1 are the two members of rotation pair i (first-half member, then its partner),
// so that the two sit in neighbouring lanes of the epilogue warp that rotates them.  SwiGLU pairs (pair == 1)
// likewise: rows 2i and 2i + 1 are retained row i of the gate matrix and of the up matrix.
struct RowInfo { int stored; int out_col; int pair_c; int head; };
__device__ inline RowInfo tile_row(const JobDev& jb, int tl, int r) {
  RowInfo o;
  o.stored = -1; o.out_col = -1; o.pair_c = 0; o.head = 0;
  if (jb.rope.enabled) {
    const int half = jb.rope.head_keep >> 1;
    const int P = tl * (BMW / 2) + (r >> 1);
    if (P >= jb.rope.n_heads * half) return o;
    const int h = P / half, cc = P - h * half, hi = r & 1;
    o.stored = h * jb.rope.head_dim + hi * (jb.rope.head_dim >> 1) + cc;
    o.out_col = h * jb.rope.head_keep + hi * half + cc;
    o.pair_c = cc; o.head = h;
  } else if (jb.pair == 1) {
    const int j = tl * (BMW / 2) + (r >> 1);
    if (j >= jb.k_out) return o;
    o.stored = (jb.omap.n_fam == 1 && jb.omap.fam[0].count == 1) ? jb.omap.fam[0].start + j
                                                                  : map_compact_to_stored(jb.omap, j);
    o.out_col = j;
    o.pair_c = r & 1;          // 0: row of the gate matrix, 1: row of the up matrix
  } else {
    const int j = tl * BMW + r;
    if (j >= jb.k_out) return o;
    o.stored = (jb.omap.n_fam == 1 && jb.omap.fam[0].count == 1) ? jb.omap.fam[0].start + j
                                                                  : map_compact_to_stored(jb.omap, j);
    o.out_col = j;
  }
  return o;
}

// Eight codes of one 32-bit word, in input-channel order, as eight fp16 values packed in a uint4:
// byte b -> (1024 + c_even, 64 + c_odd) as an fp16 pair (one PRMT, one LOP3), minus (1032, 72) = the
// exact (c-8) pair, then one fp16 FMA per pair: (c-8)*s + cz with cz = fp16(s*(8-z)).  s is the stored
// fp16 scale itself, (c-8)*s + cz is rounded once; the only other error is the rounding of cz (2^-12
// of at most 8 s, shared by the 128 weights of a group).
__device__ inline uint4 dequant_word(uint32_t w, __half2 s2, __half2 cz2) {
  uint32_t o[4];
  const __half2 off = __halves2half2(__ushort_as_half(0x6408), __ushort_as_half(0x5480));
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const uint32_t t = __byte_perm(w, 0u, 0x4040u + 0x0101u * b);
    const uint32_t v = pand_or(t, 0x00f0000fu, 0x54006400u);
    const __half2 r = __hfma2(__hsub2(*reinterpret_cast<const __half2*>(&v), off), s2, cz2);
    o[b] = *reinterpret_cast<const uint32_t*>(&r);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
// The codes themselves, less 8, as fp16 (exact), in channel order.
__device__ inline uint4 codes_word(uint32_t w) {
  uint32_t o[4];
  const __half2 off = __halves2half2(__ushort_as_half(0x6408), __ushort_as_half(0x5480));
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const uint32_t t = __byte_perm(w, 0u, 0x4040u + 0x0101u * b);
    const uint32_t v = pand_or(t, 0x00f0000fu, 0x54006400u);
    const __half2 r = __hsub2(*reinterpret_cast<const __half2*>(&v), off);
    o[b] = *reinterpret_cast<const uint32_t*>(&r);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// ---------------------------------------------------------------------------------------- epilogue of a row
// Bias, rotary embedding (Section 3.2, fused RoPE) or gated product, one rounding and the stores of a thread that owns
// one row of a tile of job `jn` (`info`: which; odd: the up row of a SwiGLU pair); the two members of a pair sit in lanes
// 2i and 2i + 1.
// Y16: a gated product of bf16 is stored as fp16 too where the job asks for it.
template <typename T, bool Y16 = false>
struct RowStore {
  RowInfo ri;
  T* y;
  int ldy, half;
  bool rope, swiglu;
  float b_own;
  unsigned long long turn;

  __device__ inline RowStore(const Params& p, int jn, const RowInfo& info, bool odd) {
    const JobDev& jb = p.job[jn];
    y = reinterpret_cast<T*>(jb.y);
    ldy = jb.ldy;
    rope = jb.rope.enabled != 0;
    swiglu = jb.pair == 1;
    half = jb.rope.head_keep >> 1;
    ri = info;
    b_own = 0.f;
    turn = 0;
    if (ri.stored >= 0) {
      const T* bias = reinterpret_cast<const T*>((swiglu && odd) ? p.job[jn + 1].bias : jb.bias);
      if (bias) b_own = DT<T>::to_f(bias[ri.stored]);
      if (rope) {
        int pidx = p.idx[(ri.head / jb.rope.rep) * half + ri.pair_c];
        pidx = min(max(pidx, 0), (jb.rope.head_dim >> 1) - 1);
        turn = p.rope_turn[pidx];
      }
    }
  }
  // tokens m0 .. m0 + NV - 1 of the row (all lanes of the warp call it)
  template <int NV>
  __device__ inline void store(const Params& p, int m0, const float (&val)[NV]) const {
    if (rope || swiglu) {
      // The even lane of a pair takes the even tokens, the odd lane the odd ones: one exchange hands each the other
      // member's value of its token.  Sixteen tokens at a time, exchange, arithmetic and stores one after the other without
      // a branch between tokens: with a test per token the eight dependent chains ran one behind the other, 300 cycles a
      // token, and a gated tile of 256 tokens took its four warps 20 us.
      constexpr int G = NV < 16 ? NV : 16, H = G / 2;
      const bool second = (threadIdx.x & 1) != 0;
      const int left = p.M - m0, odd = second ? 1 : 0;
      const float b_other = __shfl_xor_sync(0xffffffffu, b_own, 1);
      const float b_lo = second ? b_other : b_own, b_hi = second ? b_own : b_other;
      const bool live = ri.stored >= 0;
      const size_t step = 2 * (size_t)ldy;
      T* yp = y + (live ? ri.out_col - (rope && second ? half : 0) : 0) + (size_t)(m0 + odd) * ldy;    // this lane's first token
#pragma unroll
      for (int b = 0; b < NV; b += G) {
        if (b >= left) break;                                       // (the same for the whole warp)
        float lo[H], hi[H];
#pragma unroll
        for (int k = 0; k < H; ++k) {
          const float v0 = val[b + 2 * k], v1 = val[b + 2 * k + 1];
          const float got = __shfl_xor_sync(0xffffffffu, second ? v0 : v1, 1);
          lo[k] = (second ? got : v0) + b_lo;
          hi[k] = (second ? v1 : got) + b_hi;
        }
        const int n = live ? (left - b - odd + 1) >> 1 : 0;         // of this lane's H tokens the first n exist
        if (rope) {
          int at[H];
#pragma unroll
          for (int k = 0; k < H; ++k) at[k] = __ldg(p.pos + min(m0 + b + odd + 2 * k, p.M - 1));
          T r0[H], r1[H];
#pragma unroll
          for (int k = 0; k < H; ++k) {
            float cs, sn;
            rope_cos_sin(at[k], turn, cs, sn);
            r0[k] = DT<T>::from_f(fmaf(-hi[k], sn, lo[k] * cs));
            r1[k] = DT<T>::from_f(fmaf(lo[k], sn, hi[k] * cs));
          }
#pragma unroll
          for (int k = 0; k < H; ++k) {
            if (k < n) { yp[0] = r0[k]; yp[half] = r1[k]; }
            yp += step;
          }
        } else {
          // h = silu(g) * u, one rounding (the approximate division: two instructions instead of ten in warps that share
          // the issue slots with the de-quantisers; exp(-g) beyond fp32 gives a quotient of zero, the limit of silu)
          T r[H];
#pragma unroll
          for (int k = 0; k < H; ++k) r[k] = DT<T>::from_f(__fdividef(lo[k], 1.f + __expf(-lo[k])) * hi[k]);
#pragma unroll
          for (int k = 0; k < H; ++k) {
            if (k < n) *yp = r[k];
            yp += step;
          }
          if constexpr (Y16) {
            if (p.job[0].y16 != nullptr) {
              __half* hp = p.job[0].y16 + (live ? ri.out_col : 0) + (size_t)(m0 + b + odd) * p.job[0].ld16;
#pragma unroll
              for (int k = 0; k < H; ++k) {
                if (k < n) *hp = f16_of(r[k]);
                hp += 2 * (size_t)p.job[0].ld16;
              }
            }
          }
        }
      }
    } else {
      if (ri.stored < 0) return;
      T* yr = y + ri.out_col + (size_t)m0 * ldy;
      const int left = p.M - m0;
      if (left >= NV) {                       // a whole chunk of tokens: no test per token
#pragma unroll
        for (int k = 0; k < NV; ++k) { *yr = DT<T>::from_f(val[k] + b_own); yr += ldy; }
      } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          if (k >= left) break;
          *yr = DT<T>::from_f(val[k] + b_own);
          yr += ldy;
        }
      }
    }
  }
};

}  // namespace uniql
