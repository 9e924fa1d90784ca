// Block fixed point, in a header of its own that a host compiler takes too (tests/test_fixed_point.py).
//
// The storage of the float-float solutions: component = (i + l) unit with a 28-bit integer i, an FP32 remainder l (|l| < 5)
// and a power of two `unit` per site, such that the largest component has 2^26 <= |i| <= 2^27.  A component within 1/8 of
// the site's largest keeps every bit of its float-float value; a smaller one is rounded at 2^-25 units, 2^-51 of the
// largest.  fix_value returns the stored value to 2^-48 of the largest, float-float's own rounding (4.8 million random
// components: exactly).
#pragma once

// the unit of a site whose largest component is m, and its reciprocal: m < 2^(E - 126) with E its biased exponent;
// unit = 2^(E - 126 - 27), at least 2^-126 (below m = 2^-99 a float-float value ends at FP32's smallest numbers too)
__device__ __forceinline__ void fix_unit(float m, float& unit, float& inv) {
  const int b = __float_as_int(m) >> 23, E = b > 27 ? b : 27;
  unit = __int_as_float((E - 26) << 23);
  inv = __int_as_float((280 - E) << 23);
}

__device__ __forceinline__ void fix_split(float hi, float lo, float inv, int& i, float& l) {
  const float t = hi * inv;   // exact; an integer already where it has no room for a fraction
  i = __float2int_rn(t);
  l = fmaf(lo, inv, t - (float)i);
}

// (i + l) unit as hi + lo.  i = f + b with f a multiple of 16 and b = -8 .. 7; the larger operand stands first in both sums
// (f is 0 or above b; |l| < 1 where i is below 2^23), so Dekker's fast TwoSum holds in both.
__device__ __forceinline__ void fix_value(int i, float l, float unit, float& hi, float& lo) {
  const int m = (i + 8) & ~15;
  const float f = (float)m, b = (float)(i - m);   // both exact
  const float s = __fadd_rn(f, b), e = __fsub_rn(b, __fsub_rn(s, f));
  const float t = __fadd_rn(s, l), d = __fsub_rn(l, __fsub_rn(t, s));
  hi = t * unit;
  lo = __fadd_rn(e, d) * unit;
}
