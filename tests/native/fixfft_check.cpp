// Host build of csrc/fixfft.cuh for tests/test_fixfft.py: the transform of one line, the passes in
// the order of fx_fft with E elements per thread, one group after another.
#include <stdlib.h>

#include "fixfft.cuh"

using namespace gpsoc;

static const FxTable g_table = fx_make_table();

static double to(long long v, int s) {
  if (fx_plain(s)) return fx_to(v, 1086 + s);
  const FxUnit u = fx_unit(s);
  return (fx_to(v, 1086) * u.f1) * u.f2;
}

template <bool INV, int R, int E>
static void pass(const FxC* in, FxC* out, int n, int Ns, bool first) {
  const int NR = n / R, shift = kFxShift<E>;
  for (int g = 0; g < NR; ++g) {
    FxC v[R];
    const int k = g & (Ns - 1);
    for (int r = 0; r < R; ++r) {
      v[r] = in[g + r * NR];
      if (first) continue;
      if (r == 0) {
        v[r] = fx_shift(v[r], shift);
        continue;
      }
      const int at = r * k * (n / (Ns * R)) * (kFxTable / n);
      FxW w;
      fx_split(g_table.c[2 * at], E == 8 ? 3 : 2, w.xh, w.xl);
      fx_split(g_table.c[2 * at + 1], E == 8 ? 3 : 2, w.yh, w.yl);
      v[r] = fx_cmul<INV, E == 2>(v[r], w);
    }
    fx_dft<INV, R>(v);
    for (int q = 0; q < R; ++q) out[(g - k) * R + k + q * Ns] = v[q];
  }
}

template <bool INV, int E>
static void line(double* d, int n) {
  int key = 0;
  for (int i = 0; i < 2 * n; ++i) key = fx_key(d[i]) > key ? fx_key(d[i]) : key;
  const int em = (key >> 20) > 1 ? key >> 20 : 1;
  constexpr int LE = (E == 8) ? 3 : (E == 4) ? 2 : 1;
  int L = 0;
  while ((1 << L) < n) ++L;
  const int rem = L % LE, lr = rem ? rem : LE;
  const int F = lr == 1 ? kFxBits<2> : lr == 2 ? kFxBits<4> : kFxBits<8>;
  FxC* a = (FxC*)aligned_alloc(16, sizeof(FxC) * n);
  FxC* b = (FxC*)aligned_alloc(16, sizeof(FxC) * n);
  for (int i = 0; i < n; ++i) { a[i].x = fx_of(d[2 * i], em, F); a[i].y = fx_of(d[2 * i + 1], em, F); }
  int sc = em - 1022 - F, Ns = 1 << lr;
  if (lr == 1) pass<INV, 2, E>(a, b, n, 1, true);
  else if (lr == 2) pass<INV, (E >= 4 ? 4 : 2), E>(a, b, n, 1, true);
  else pass<INV, E, E>(a, b, n, 1, true);
  for (; Ns < n; Ns *= E) {
    FxC* t = a; a = b; b = t;
    pass<INV, E, E>(a, b, n, Ns, false);
    sc += kFxShift<E>;
  }
  for (int i = 0; i < n; ++i) {
    d[2 * i] = to(b[i].x, em == 0x7ff ? 4096 : sc);
    d[2 * i + 1] = to(b[i].y, em == 0x7ff ? 4096 : sc);
  }
  free(a);
  free(b);
}

extern "C" {
// in place, unnormalised, n a power of two in [8, 1024], E = 2, 4 or 8
void fx_line(double* d, int n, int e, int inverse) {
  if (e == 8) inverse ? line<true, 8>(d, n) : line<false, 8>(d, n);
  else if (e == 4) inverse ? line<true, 4>(d, n) : line<false, 4>(d, n);
  else inverse ? line<true, 2>(d, n) : line<false, 2>(d, n);
}
// table entry k as (re, im) in units of 2^-62
void fx_table(int k, long long* out) { out[0] = g_table.c[2 * k]; out[1] = g_table.c[2 * k + 1]; }
// d -> fixed point at exponent field em with f bits -> FP64
double fx_round_trip(double d, int em, int f) { return to(fx_of(d, em, f), em - 1022 - f); }
double fx_widen(long long v, int s) { return to(v, s); }
}
