// Activation quantisation shared by the decode kernels (sm_100a): fp16 or bf16 activations become 16-bit fixed point
// per (batch row, 128-channel group), split in two signed bytes, so that the 4-bit codes can go to the int8
// tensor-core MMA as they lie in memory.
#pragma once
#include "common.cuh"

namespace uniql {

// 16 / U consecutive lanes hold the 128 activations of one (batch row, group), U units of eight each (`in`): 16-bit fixed
// point against the group's maximum, x_i = rint(x * 2^e) = 256 * hi + lo with both bytes signed.  Returns the units'
// bytes in the order the nibbles leave a weight word (even codes first), the group's integer sum and 2^-e (NaN when the
// group holds a non-finite activation).  Every lane of the warp must call it (shuffles over the lanes of a group).
// T = bf16: 8 significand bits, exact for every element within a factor 2^7 of its group's maximum.  The exponent e is
// capped at 120 so that 2^e and 2^-e stay normal fp32 numbers: groups whose maximum is under 2^-106 lose bits below 2^-120.
// Every block of a decode launch quantises the whole activation matrix between its predecessor's end and its own first MMA.
// Long matrices are bound by issue slots there: one unit per lane is about 110 instructions per unit, of which the
// reductions over the lanes and the exponent come once per lane; four units per lane about 50 (Llama-3-8B layer at four rows
// and keep 0.65 42.0 -> 37.1 us).  Short ones are bound by the chain of one lane (2048 activations: 4.1 us a call with one
// unit per lane, 4.8 with four).  The rule stands where the decode kernel stages its activations.
template <typename T, int U>
__device__ inline void quantise_units(const uint4 (&in)[U], uint2 (&hi)[U], uint2 (&lo)[U], int& isum_out, float& inv_scale_out) {
  using T2 = typename DT<T>::T2;
  // the group's maximum is taken on the magnitude bits as integers: Inf and NaN compare above every finite value,
  // where a floating-point maximum would drop a NaN
  auto max2 = [](uint32_t a, uint32_t b) { uint32_t d; asm("max.u16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b)); return d; };
  uint32_t mag = 0u;
#pragma unroll
  for (int k = 0; k < U; ++k)
    mag = max2(mag, max2(max2(in[k].x & 0x7fff7fffu, in[k].y & 0x7fff7fffu), max2(in[k].z & 0x7fff7fffu, in[k].w & 0x7fff7fffu)));
  mag = max2(mag, mag >> 16);
#pragma unroll
  for (int o2 = 8 / U; o2 >= 1; o2 >>= 1) mag = max2(mag, __shfl_xor_sync(0xffffffffu, mag, o2));
  const uint32_t low = mag & 0xffffu;
  const float amax = DT<T>::to_f2(*reinterpret_cast<const T2*>(&low)).x;
  const uint32_t amax_bits = __float_as_uint(amax);
  const bool finite = amax_bits < 0x7f800000u;
  int e = 0;
  if (amax_bits != 0u && finite) {
    e = min(14 - ((int)(amax_bits >> 23) - 127), 120);
    if (amax * __uint_as_float((uint32_t)(127 + e) << 23) > 32639.f) --e;     // keep the high byte of x_i + 128 signed
  }
  // a group that holds an Inf or a NaN gets a NaN factor: every output that uses the group becomes NaN
  const float scale = __uint_as_float((uint32_t)(127 + e) << 23);
  inv_scale_out = finite ? __uint_as_float((uint32_t)(127 - e) << 23) : __uint_as_float(0x7fc00000u);
  // t = x_i + 128 through the float adder: x * 2^e + (1.5 * 2^23 + 128) is rounded to an integer (nearest even, as
  // rint) whose low 16 mantissa bits are those of t.  Byte 1 of t is hi, byte 0 of t xor 0x80 is lo; the bytes are
  // gathered with byte permutes, and their sums give the sum of the x_i.
  int s_hi = 0, s_lo = 0;
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const uint32_t w[4] = {in[k].x, in[k].y, in[k].z, in[k].w};
    uint32_t te[4], to[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 v = DT<T>::to_f2(*reinterpret_cast<const T2*>(&w[i]));
      te[i] = __float_as_uint(fmaf(v.x, scale, 12582912.f + 128.f));
      to[i] = __float_as_uint(fmaf(v.y, scale, 12582912.f + 128.f));
    }
    hi[k].x = __byte_perm(__byte_perm(te[0], te[1], 0x0051), __byte_perm(te[2], te[3], 0x0051), 0x5410);
    hi[k].y = __byte_perm(__byte_perm(to[0], to[1], 0x0051), __byte_perm(to[2], to[3], 0x0051), 0x5410);
    lo[k].x = __byte_perm(__byte_perm(te[0], te[1], 0x0040), __byte_perm(te[2], te[3], 0x0040), 0x5410) ^ 0x80808080u;
    lo[k].y = __byte_perm(__byte_perm(to[0], to[1], 0x0040), __byte_perm(to[2], to[3], 0x0040), 0x5410) ^ 0x80808080u;
    s_hi = __dp4a((int)hi[k].x, 0x01010101, __dp4a((int)hi[k].y, 0x01010101, s_hi));
    s_lo = __dp4a((int)lo[k].x, 0x01010101, __dp4a((int)lo[k].y, 0x01010101, s_lo));
  }
  int isum = 256 * s_hi + s_lo;
#pragma unroll
  for (int o2 = 8 / U; o2 >= 1; o2 >>= 1) isum += __shfl_xor_sync(0xffffffffu, isum, o2);
  isum_out = isum;
}

}  // namespace uniql
