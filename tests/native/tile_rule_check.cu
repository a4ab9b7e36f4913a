// Host program of tests/test_tile_rule.py: asks the built-in tile rule for every grid and batch given, and prints
// each tile that its passes could not be launched with.
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <string>

#include "gpsoc_internal.cuh"

using namespace gpsoc;

static long long g_asked = 0, g_bad = 0;

template <class T> static void ask(const Geo& g, int nsolve) {
  for (int axis = 0; axis < g.d; ++axis) {
    int lines, ept, threads, la[64], ea[64];
    tile_shape<T>(g, axis, nsolve, lines, ept, threads);
    const int n = tile_candidates<T>(g, axis, la, ea, 64);
    bool ok = threads <= 384 && threads % 32 == 0 && n <= 64;
    if (axis > 0) ok = ok && threads % std::min(lines, threads) == 0;   // a thread stays on one column
    bool listed = false;
    for (int k = 0; k < n; ++k) listed = listed || (la[k] == lines && ea[k] == ept);
    ++g_asked;
    if (ok && listed) continue;
    if (++g_bad <= 20)
      printf("%dx%dx%d batch %d FP%d axis %d: %d lines, %d elements, %d threads%s\n", g.n[0], g.n[1], g.n[2], nsolve,
             (int)sizeof(T) * 8, axis, lines, ept, threads, listed ? "" : ", not a candidate");
  }
}

// arguments: dimensions, the log2 of the most points of one solve, batches...
int main(int argc, char** argv) {
  const int d = atoi(argv[1]), most = atoi(argv[2]);
  for (int a = 3; a <= 10; ++a)
    for (int b = 3; b <= 10; ++b)
      for (int c = (d == 3 ? 3 : 0); c <= (d == 3 ? 10 : 0); ++c) {
        if (a + b + c > most) continue;
        Geo g{};
        g.d = d;
        const int l[3] = {a, b, c};
        g.npts = 1;
        for (int i = 0; i < 3; ++i) { g.log2n[i] = l[i]; g.n[i] = 1 << l[i]; g.npts *= g.n[i]; }
        for (int k = 3; k < argc; ++k) { ask<double>(g, atoi(argv[k])); ask<float>(g, atoi(argv[k])); }
      }
  printf("%lld tiles, %lld bad\n", g_asked, g_bad);
  return g_bad != 0;
}
