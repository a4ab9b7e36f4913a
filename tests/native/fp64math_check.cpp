// Host build of csrc/fp64math.cuh for tests/test_fp64math.py: largest errors over the arguments given, in ulp of the
// exact result (long double: 64 bits or more).
#include <math.h>

#include "fp64math.cuh"

using namespace gpsoc;
typedef long double Q;

static double ulps(Q error, Q exact) {
  int e;
  frexpl(exact, &e);
  return (double)(fabsl(error) / ldexpl(1.0L, e - 53));
}

extern "C" {
// x and the step in FP32 ulp by which its start is off
double fm_rsqrt(double x, int off) {
  if (!rsqrt_in_range(x)) return -1.0;
  const double y = widen_f(f_from(f_bits((float)(1.0L / sqrtl((Q)narrow_f(x)))) + off));
  const Q want = 1.0L / sqrtl((Q)x);
  return ulps((Q)rsqrt_refine(x, y) - want, want);
}
double fm_divide(double a, double m) { return ulps((Q)divide_near_one(a, m) - (Q)a / m, (Q)a / m); }
double fm_rsqrt1(double d) {
  if (!rsqrt1_in_range(d)) return -1.0;
  const Q want = 1.0L / sqrtl(1.0L + d);
  return ulps((Q)rsqrt1(d) - want, want);
}
double fm_taylor(double x, int odd) {
  if (!taylor_in_range(x)) return -1.0;
  const Q want = odd ? sinl(x) : cosl(x);
  return ulps((Q)taylor_sincos(x, odd) - want, want);
}
}
