// FP64 <-> FP32 conversions by integer arithmetic.
//
// GB300 converts from and to 64-bit types at the rate of its FP64 pipe (about 2
// per clock and SM), so a layout pass that converts 24 reals per site is bound
// by that and not by memory.  These do the same conversion (round to nearest
// even, exact the other way, signed zeros kept) on the integer pipes for
// normal results and zeros; anything else -- subnormal or overflowing results,
// infinities, NaN -- raises `other`, and the caller converts again with the
// cast.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define MGLMA_HD __host__ __device__ __forceinline__
#else
#define MGLMA_HD static inline
#endif

namespace mglma {

// FP32 bits of the FP64 with high word hi and low word lo
MGLMA_HD uint32_t d2f_bits(uint32_t hi, uint32_t lo, bool& other) {
  const uint32_t a = hi & 0x7fffffffu, sign = hi & 0x80000000u;
  // exponent field 897 .. 1150: the FP32 exponent is 1 .. 254 before rounding
  // (a carry out of 254 gives infinity, as rounding does)
  const bool normal = a - 0x38100000u < 0x47f00000u - 0x38100000u;
  const bool zero = (a | lo) == 0;
  other |= !(normal || zero);
  const uint32_t t = (a << 3) | (lo >> 29);  // exponent modulo 2^9, 23 mantissa bits
  // 29 bits are dropped; add one unit when they exceed half, or equal half and
  // the kept part is odd
  const uint32_t up = ((lo & 0x1fffffffu) + 0x0fffffffu + (t & 1u)) >> 29;
  const uint32_t f = t + 0x40000000u + up;  // 0x40000000 = -(896 << 23) mod 2^32
  return sign | (zero ? 0u : f & 0x7fffffffu);
}

// high and low word of the FP64 with FP32 bits f
MGLMA_HD void f2d_bits(uint32_t f, uint32_t& hi, uint32_t& lo, bool& other) {
  const uint32_t a = f & 0x7fffffffu, sign = f & 0x80000000u;
  const bool normal = a - 0x00800000u < 0x7f800000u - 0x00800000u;
  other |= !(normal || a == 0);
  hi = sign | (a == 0 ? 0u : (a >> 3) + 0x38000000u);  // 896 << 20
  lo = f << 29;
}

#ifdef __CUDACC__
__device__ __forceinline__ float d2f_fast(double d, bool& other) {
  return __uint_as_float(d2f_bits((uint32_t)__double2hiint(d), (uint32_t)__double2loint(d), other));
}
__device__ __forceinline__ double f2d_fast(float f, bool& other) {
  uint32_t hi, lo;
  f2d_bits(__float_as_uint(f), hi, lo, other);
  return __hiloint2double((int)hi, (int)lo);
}
#endif

}  // namespace mglma
