// Host build of the running double-word sums of csrc/dword.cuh for tests/test_dword_sums.py.
#include "dword.cuh"

using namespace gpsoc;

extern "C" {
// kind 0: dwa_mul, 1: dwa_sub, 2: dwa_sqd (b unused), 3: dwa_mulf (b's high word), 4: dwa_sq (a's high word), 5: dwa_add of a;
// opened by the first term when open != 0 (kinds 0 and 2)
void dwa_run(int kind, int open, int n, const float* a, const float* b, float* out) {
  DF s{0.0f, 0.0f};
  for (int i = 0; i < n; ++i) {
    const DF x{a[2 * i], a[2 * i + 1]}, y{b[2 * i], b[2 * i + 1]};
    if (open && i == 0) { s = kind == 0 ? dwa_of_mul(x, y) : dwa_of_sqd(x); continue; }
    if (kind == 0) dwa_mul(s, x, y);
    else if (kind == 1) dwa_sub(s, x, y);
    else if (kind == 2) dwa_sqd(s, x);
    else if (kind == 3) dwa_mulf(s, x, y.hi);
    else if (kind == 4) dwa_sq(s, x.hi);
    else dwa_add(s, x.hi, x.lo);
  }
  s = dwa_value(s);
  out[0] = s.hi;
  out[1] = s.lo;
}
float dwa_narrow(double x) { return narrow_f(x); }
void dwa_split(double x, float* fast, float* any) {
  const DF f = dw_of(x), g = dw_of_any(x);
  fast[0] = f.hi; fast[1] = f.lo;
  any[0] = g.hi; any[1] = g.lo;
}
}
