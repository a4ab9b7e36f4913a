// FP64 functions shorter than the library's (an FP64 warp instruction holds its sub-partition for 64 cycles), for the
// device and, in the CPU check of their errors (tests/test_fp64math.py), for the host.  Each comment gives the method and
// its error; ulp: unit in the last place of the result.
#pragma once

#include "dword.cuh"

namespace gpsoc {

// 1/sqrt(x) from y, an approximation to 2^-20: with e = 1 - x y^2, 1/sqrt(x) = y (1 - e)^(-1/2), by the binomial series
// y (1 + e/2 + 3 e^2/8) to 5 e^3/16 < 2^-61.  Roundings: half an ulp of the sum, and 2^-54 of it through e.  Within 1
// ulp + 2^-61, the library's bound; 4 instructions.
GPSOC_DW double rsqrt_refine(double x, double y) {
  const double e = fma(-(x * y), y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}
// the x that y = rsqrtf of x rounded to FP32 is within 2^-20 for: 2^-111 <= x < 2^112
GPSOC_DW bool rsqrt_in_range(double x) {
  const int h = (int)d_hi(x);
  return h >= 0x39000000 && h < 0x46f00000;
}

// a/m for m = 1 - d: where |d| < 2^-30, a + a d, which leaves out a d^2 < 2^-60 a
GPSOC_DW double divide_near_one(double a, double m) {
  const double d = 1.0 - m;
  return (d_hi(d) & 0x7fffffffu) < 0x3e100000u ? fma(d, a, a) : a / m;
}
// 1/sqrt(1 + d): where |d| < 2^-20, the binomial series 1 - d/2 + 3 d^2/8, which leaves out 5 d^3/16 < 2^-61
GPSOC_DW bool rsqrt1_in_range(double d) { return (d_hi(d) & 0x7fffffffu) < 0x3eb00000u; }
GPSOC_DW double rsqrt1(double d) { return fma(d, fma(0.375, d, -0.5), 1.0); }

// sin x (odd) or cos x for 0 <= x < 0.8 by their Taylor sums to x^19 and x^18; what is left out is below 2^-61 of the
// value.  Three roundings of the terms after the first, at most 0.11 of the sine and 0.46 of the cosine, and the sum's
// own: within 1 ulp (sine) and 2 ulp (cosine; the library's bound for both).
GPSOC_DW bool taylor_in_range(double x) { return d_hi(x) < 0x3fe99999u; }   // 0 <= x < 0.8
GPSOC_DW double taylor_sincos(double x, bool odd) {
  const double x2 = x * x;
  double r = odd ? -1.0 / 121645100408832000.0 : -1.0 / 6402373705728000.0;    // 1/19!, 1/18!
  r = fma(r, x2, odd ? 1.0 / 355687428096000.0 : 1.0 / 20922789888000.0);      // 1/17!, 1/16!
  r = fma(r, x2, odd ? -1.0 / 1307674368000.0 : -1.0 / 87178291200.0);
  r = fma(r, x2, odd ? 1.0 / 6227020800.0 : 1.0 / 479001600.0);
  r = fma(r, x2, odd ? -1.0 / 39916800.0 : -1.0 / 3628800.0);
  r = fma(r, x2, odd ? 1.0 / 362880.0 : 1.0 / 40320.0);
  r = fma(r, x2, odd ? -1.0 / 5040.0 : -1.0 / 720.0);
  r = fma(r, x2, odd ? 1.0 / 120.0 : 1.0 / 24.0);
  r = fma(r, x2, odd ? -1.0 / 6.0 : -0.5);
  const double f = odd ? x : 1.0;
  return fma(r * x2, f, f);
}

}  // namespace gpsoc
