// FP64 multiplication on the integer pipe, correctly rounded.
//
// An FP64 instruction occupies a GB300 SM's FP64 pipe for 64 cycles per warp
// and SM quarter (2 lanes per clock and SM), while its integer and FP32 pipes
// are nearly idle in the stencils, whose FP64 instructions bound them.  A
// correctly rounded FP64 product takes about 35 integer instructions (four of
// them 32 x 32 -> 64 multiplications): measured alone, 0.78 of the native
// multiplication's time (0.741 against 0.952 ms for 125M products), and both
// run side by side, two emulated products cost no more time than the two
// native operations beside them (0.499 ms for 62M of each).  Moving a part of
// a kernel's products here so that both pipes finish together nearly halves
// its FP64 time.  (Sums do not pay: 1.16 of a native one for operands of one
// sign, 1.5 in general, as the alignment and cancellation need shifts.)
//
// The functions follow the definition of IEEE 754 round-to-nearest-even
// multiplication for finite operands that are zero or normal with a product
// that is zero or normal; results are bit-identical to __dmul_rn there.  The
// callers test their inputs' exponents first (soft_window) and use native
// instructions otherwise.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__

__device__ __forceinline__ unsigned dbl_hi(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned dbl_lo(double x) { return (unsigned)__double2loint(x); }

// positive x with 2^-64 <= x < 2^64: products of the few such values that a
// face or a cell forms (at most cubes, their reciprocals and one more factor)
// stay normal
__device__ __forceinline__ bool soft_window(double x) {
  return dbl_hi(x) - ((1023u - 64u) << 20) < (128u << 20);
}

// |x| |y| for normal x, y, as the bits of a positive double.  The two 53-bit
// significands, each moved to the top of 64 bits, give a 128-bit product
// whose upper half holds the 53 result bits and at least 10 more; the lower
// half only matters as a sticky bit.  Rounding adds half a unit less one plus
// the kept lsb (ties go to even); a carry out of the significand runs into
// the exponent field, as it should.
__device__ __forceinline__ uint64_t soft_mul_bits(double x, double y) {
  const unsigned xh = dbl_hi(x), yh = dbl_hi(y), xl = dbl_lo(x), yl = dbl_lo(y);
  const unsigned a1 = __funnelshift_l(xl, xh | 0x100000u, 11), a0 = xl << 11;
  const unsigned b1 = __funnelshift_l(yl, yh | 0x100000u, 11), b0 = yl << 11;
  const uint64_t p00 = (uint64_t)a0 * b0;
  const uint64_t p01 = (uint64_t)a0 * b1 + (p00 >> 32);
  const uint64_t p10 = (uint64_t)a1 * b0 + (unsigned)p01;
  const uint64_t p11 = (uint64_t)a1 * b1 + (p01 >> 32) + (p10 >> 32);
  const unsigned sticky = ((unsigned)p10 | (unsigned)p00) ? 1u : 0u;
  const unsigned c = (unsigned)(p11 >> 63);                // the product's top bit is 63 or 62
  const unsigned sh = 10u + c;
  const uint64_t m = p11 >> sh;                            // 53 bits, the implicit one included
  const unsigned half1 = (0x1ffu << c) | c;                // 2^(sh - 1) - 1
  const unsigned rem = ((unsigned)p11 | sticky) & ((half1 << 1) | 1u);
  const unsigned rnd = (rem + half1 + ((unsigned)m & 1u)) >> sh;
  // biased exponent: ex + ey - 1023 + c; the implicit bit in m adds one more
  const unsigned e = (xh & 0x7ff00000u) + (yh & 0x7ff00000u) - (1024u << 20) + (c << 20);
  return m + rnd + ((uint64_t)e << 32);
}

// x y for positive normal x, y with a normal product
__device__ __forceinline__ double soft_mul_pos(double x, double y) {
  return __longlong_as_double((long long)soft_mul_bits(x, y));
}

// x y of either sign, each zero or normal, with a zero or normal product
__device__ __forceinline__ double soft_mul(double x, double y) {
  const unsigned xh = dbl_hi(x), yh = dbl_hi(y);
  const bool zero = (xh << 1) == 0u || (yh << 1) == 0u;
  const uint64_t r = zero ? 0u : soft_mul_bits(x, y);
  return __longlong_as_double(
      (long long)(r | ((uint64_t)((xh ^ yh) & 0x80000000u) << 32)));
}

// 2 x for x zero or normal and below the largest exponent: an exponent
// increment
__device__ __forceinline__ double soft_twice(double x) {
  const unsigned h = dbl_hi(x);
  return __hiloint2double((int)((h << 1) ? h + 0x100000u : h), (int)dbl_lo(x));
}

// x y for any x, y: on the integer pipe where both lie within 2^(+-480) (the
// product is then normal), else one native multiplication behind a call (a
// predicated one would take its FP64 slot in every warp)
static __device__ __noinline__ double native_mul(double x, double y) { return __dmul_rn(x, y); }
__device__ __forceinline__ double soft_mul_any(double x, double y) {
  const unsigned xm = dbl_hi(x) & 0x7fffffffu, ym = dbl_hi(y) & 0x7fffffffu;
  constexpr unsigned lo = (1023u - 480u) << 20, w = 960u << 20;
  if (xm - lo >= w || ym - lo >= w) return native_mul(x, y);
  return __longlong_as_double((long long)(soft_mul_bits(x, y) |
      ((uint64_t)((dbl_hi(x) ^ dbl_hi(y)) & 0x80000000u) << 32)));
}

// the products of a face's or a cell's formulas, on the integer pipe (SOFT)
// or native; the same bits either way
template <bool SOFT>
struct Mul {
  static __device__ __forceinline__ double pos(double x, double y) {
    return SOFT ? soft_mul_pos(x, y) : __dmul_rn(x, y);
  }
  static __device__ __forceinline__ double any(double x, double y) {
    return SOFT ? soft_mul(x, y) : __dmul_rn(x, y);
  }
  static __device__ __forceinline__ double twice(double x) {
    return SOFT ? soft_twice(x) : __dadd_rn(x, x);
  }
};

#endif
