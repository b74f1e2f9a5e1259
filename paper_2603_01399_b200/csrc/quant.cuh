// Q(v, delta) of Section 3.2 Eq. 6 for eight values at a time, bit for bit: round_half_even of the IEEE fp32 quotient v / delta.
#pragma once

#include "common.cuh"

namespace quasar {

#ifdef __CUDACC__
struct QuantStep {
  float delta, inv;
  bool quick;   // the form without a division applies to the row
};
__device__ __forceinline__ QuantStep quant_step(float delta, bool has_nan) {
  QuantStep s;
  s.delta = delta;
  s.inv = __frcp_rn(delta);
  // (about 2^-100 .. 2^100: no remainder below loses bits to underflow where it decides anything)
  s.quick = !has_nan && delta >= 7.9e-31f && delta <= 1.2e30f;
  return s;
}

// f[e]: a float whose low mantissa bits hold round_half_even(v[e] / delta) in two's complement.
// The quotient is the correctly rounded one by Markstein's theorem (IBM J. Res. Dev. 34, 1990): with y the rounded reciprocal
// of b, q an approximation of a / b within one unit in the last place and r = a - b q, exact by a fused multiply-add,
// q + r y rounded once is a / b rounded.  The first step brings a y (within three units) to q, the second is the theorem's.
// |v| <= limit * delta up to a rounding, so the integer needs no clamp.
__device__ __forceinline__ void quantize8(const float (&v)[8], const QuantStep& s, int limit, float (&f)[8]) {
  constexpr float kMagic = 12582912.f;   // 1.5 * 2^23: adding it leaves the nearest integer, ties to even, in the low bits
  if (s.quick) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float q = __fmul_rn(v[e], s.inv);
      q = __fmaf_rn(__fmaf_rn(-q, s.delta, v[e]), s.inv, q);
      q = __fmaf_rn(__fmaf_rn(-q, s.delta, v[e]), s.inv, q);
      f[e] = __fadd_rn(q, kMagic);
    }
  } else {   // rows of extreme magnitude, or holding a NaN: the definition as it stands
#pragma unroll 1
    for (int e = 0; e < 8; ++e) {
      float r = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k == e) r = v[k];
      const int q = max(-limit, min(limit, __float2int_rn(__fdiv_rn(r, s.delta))));
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (k == e) f[k] = kMagic + (float)q;
    }
  }
}

// the low bytes of eight such floats
__device__ __forceinline__ uint2 pack_codes8(const float (&f)[8]) {
  uint32_t p[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) p[e] = __byte_perm(__float_as_uint(f[2 * e]), __float_as_uint(f[2 * e + 1]), 0x0040);
  return make_uint2(__byte_perm(p[0], p[1], 0x5410), __byte_perm(p[2], p[3], 0x5410));
}
// the low nibbles, element 0 lowest
__device__ __forceinline__ uint32_t pack_nibbles8(const float (&f)[8]) {
  uint32_t p = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) p |= (__float_as_uint(f[e]) & 0xFu) << (4 * e);
  return p;
}
__device__ __forceinline__ void unpack_bf16x8(const uint4& v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    f[2 * e] = __uint_as_float(w[e] << 16);
    f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
  }
}

// A maximum that ignores NaNs (what the step size is defined by) and whether one was met: the largest magnitude among the
// numbers, and the largest bit pattern of all.
struct AbsMax {
  float num;
  uint32_t bits;
  __device__ __forceinline__ AbsMax() : num(0.f), bits(0u) {}
  __device__ __forceinline__ void take(float v) {
    const float a = fabsf(v);
    num = fmaxf(num, a);
    bits = max(bits, __float_as_uint(a));
  }
  __device__ __forceinline__ bool has_nan() const { return bits > 0x7f800000u; }
};
#endif

}  // namespace quasar
