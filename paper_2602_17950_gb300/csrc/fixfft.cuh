// The transforms of the FP64 passes, computed in 64-bit fixed point.
//
// This part issues one FP64 warp instruction per 64 cycles and SM sub-partition (clock64
// measurements), but a 64-bit integer add takes 2-3 cycles and a 32 x 32 -> 64 bit
// multiply-add 4.  A Stockham transform is additions and multiplications by numbers of modulus
// 1, so it loses nothing in fixed point as long as each line is scaled to its own largest value:
// a line's values are held to 2^-59 of that value and better (FP64 products and sums round at
// 2^-53 of each value, and their errors add up over the passes all the same).  Against exact
// transforms the error measured over the solver's states is a third to a half of that of the
// FP64 butterflies these replace (tests/test_fixfft.py).
//
// Scaling.  A line whose values are below 2^m is held as X = x 2^(F - m) with |X| < 2^F.  With
// F = 62 - log2 R the R-point DFT of the first pass stays below 2^62.5 (|X| <= sqrt2 2^F as a
// complex number, times R), and every later pass multiplies by its twiddles times 2^-LE
// (LE = log2 of its radix) first, so it stays below 2^62.5 as well.  That factor costs
// nothing: the twiddles are tabled as w 2^(64 - LE), and the product keeps its upper 64 bits.
// The values of a line are complex numbers of one transform, so one exponent per line is what
// FP64 butterflies would meet too: they add its largest value into every output.
//
// Lines holding an infinity or a NaN come back as NaN.
#pragma once

#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define GPSOC_FX __host__ __device__ __forceinline__
#else
#define GPSOC_FX inline
#endif

namespace gpsoc {

// complex fixed-point value, and a twiddle split into signed 32-bit halves: w = xh 2^32 + xl
struct alignas(16) FxC { long long x, y; };
struct alignas(16) FxW { int xh, xl, yh, yl; };

// ------------------------------------------------------------------ twiddle table
// W_1024^k = exp(-2 pi i k / 1024) in units of 2^-62, built at compile time: Taylor sums of
// sine and cosine on the first octant in 128-bit integer arithmetic, the rest by symmetry.
constexpr int kFxTable = 1024;
struct FxTable { long long c[2 * kFxTable]; };

constexpr long long fx_mul62(long long a, long long b) {
  return (long long)(((__int128)a * b + ((__int128)1 << 61)) >> 62);
}
constexpr FxTable fx_make_table() {
  FxTable t{};
  long long co[kFxTable / 8 + 1] = {}, si[kFxTable / 8 + 1] = {};
  const long long pi60 = 0x3243F6A8885A308DLL;           // pi 2^60
  const long long one = 1LL << 62;
  for (int k = 0; k <= kFxTable / 8; ++k) {
    const long long a = (long long)(((__int128)pi60 * k) >> 7);   // 2 pi k / 1024 in units of 2^-62
    const long long a2 = fx_mul62(a, a);
    long long c = one, s = a, tc = one, ts = a;
    for (int j = 1; j <= 12; ++j) {
      tc = -fx_mul62(tc, a2) / ((2 * j - 1) * (2 * j));
      ts = -fx_mul62(ts, a2) / ((2 * j) * (2 * j + 1));
      c += tc;
      s += ts;
    }
    co[k] = c;
    si[k] = s;
  }
  for (int k = 0; k < kFxTable; ++k) {
    const int quarter = k / (kFxTable / 4), m = k % (kFxTable / 4);
    const long long c = m <= kFxTable / 8 ? co[m] : si[kFxTable / 4 - m];
    const long long s = m <= kFxTable / 8 ? si[m] : co[kFxTable / 4 - m];
    // exp(-i a) times (-i)^quarter
    long long x = c, y = -s;
    for (int q = 0; q < quarter; ++q) { const long long u = x; x = y; y = -u; }
    t.c[2 * k] = x;
    t.c[2 * k + 1] = y;
  }
  return t;
}

// bits dropped by the twiddle product of a pass of E = 2, 4 or 8 elements per thread, and bits F of a
// line's values before a first pass of radix R
template <int E> constexpr int kFxShift = (E == 8) ? 3 : (E == 4) ? 2 : 1;
template <int R> constexpr int kFxBits = 62 - ((R == 8) ? 3 : (R == 4) ? 2 : 1);

// table entry (units of 2^-62) as the split twiddle in units of 2^-(64 - shift), shift 2 or 3 (E = 2: 2, as
// units of 2^-63 would not hold w = 1, and fx_cmul doubles its product); the low half stays above -2^31, so
// that its negative is an int too
GPSOC_FX void fx_split(long long w, int shift, int& hi, int& lo) {
  long long v = (w + ((1LL << (shift - 2)) >> 1)) >> (shift - 2);
  lo = (int)(unsigned)v;
  if (lo == (int)0x80000000) { v += 1; lo += 1; }
  hi = (int)((v - lo) >> 32);
}

// ------------------------------------------------------------------ conversions (integer only)
GPSOC_FX unsigned long long fx_bits(double d) {
#if defined(__CUDA_ARCH__)
  return (unsigned long long)__double_as_longlong(d);
#else
  unsigned long long b;
  memcpy(&b, &d, 8);
  return b;
#endif
}
GPSOC_FX double fx_double(unsigned long long b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}
GPSOC_FX int fx_clz(unsigned v) {   // v != 0
#if defined(__CUDA_ARCH__)
  return __clz((int)v);
#else
  return __builtin_clz(v);
#endif
}
// the upper word without its sign: its maximum over a line gives the line's exponent field
GPSOC_FX int fx_key(double d) { return (int)((unsigned)(fx_bits(d) >> 32) & 0x7fffffffu); }

// shifts of a 64-bit value held as two words, by any distance >= 0
GPSOC_FX void fx_shr(unsigned& h, unsigned& l, int n) {
  if (n >= 32) { l = h; h = 0; n -= 32; }
#if defined(__CUDA_ARCH__)
  l = __funnelshift_rc(l, h, n);
  h = __funnelshift_rc(h, 0u, n);
#else
  if (n >= 32) { l = h; h = 0; if (n > 32) l = 0; return; }
  if (n) { l = (l >> n) | (h << (32 - n)); h >>= n; }
#endif
}
GPSOC_FX unsigned fx_shl(unsigned h, unsigned l, int n) {   // upper word, 0 <= n < 32
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(l, h, n);
#else
  return n ? (h << n) | (l >> (32 - n)) : h;
#endif
}
// d in units of 2^(em - 1022 - f): em the line's exponent field (>= 1), |result| < 2^f, f in [53, 62]
GPSOC_FX long long fx_of(double d, int em, int f) {
  const unsigned long long b = fx_bits(d);
  const unsigned H = (unsigned)(b >> 32), L = (unsigned)b;
  const int e = (int)(H >> 20) & 0x7ff;
  unsigned h = H & 0xfffffu;
  if (e) h |= 0x100000u;
  h = fx_shl(h, L, f - 53);
  unsigned l = L << (f - 53);
  fx_shr(h, l, em - (e ? e : 1));
  const unsigned long long sg = (unsigned long long)(long long)((int)H >> 31);
  return (long long)(((((unsigned long long)h << 32) | l) ^ sg) - sg);
}
// The unit 2^s of a line's results: fx_to(v, 1086 + s) where s is plain; for exponents at the ends of the
// FP64 range (or a line with an infinity or a NaN, s >= 2048) fx_to(v, 1086) and the two factors of 2^s
struct FxUnit { double f1, f2; };
GPSOC_FX bool fx_plain(int s) { return s > 64 - 1086 && s < 2047 - 1086; }
GPSOC_FX double fx_pow2(int e) {
  return e >= 1024 ? fx_double(0x7ff0000000000000ULL) : e < -1022 ? 0.0 : fx_double((unsigned long long)(e + 1023) << 52);
}
GPSOC_FX FxUnit fx_unit(int s) {
  FxUnit u;
  u.f1 = s >= 2048 ? fx_double(0x7ff8000000000000ULL) : fx_pow2(s / 2);
  u.f2 = fx_pow2(s - s / 2);
  return u;
}
// v 2^(base - 1086) rounded to FP64, 64 < base < 2047
GPSOC_FX double fx_to(long long v, int base) {
  const unsigned sg = (unsigned)((int)(v >> 32) >> 31);
  const unsigned long long m = (unsigned long long)((v ^ (v >> 63)) - (v >> 63));
  unsigned l = (unsigned)m, h = (unsigned)(m >> 32);
  if (h == 0) { h = l; l = 0; base -= 32; }
  const int lz = fx_clz(h | 1u);
  const unsigned mh = fx_shl(h, l, lz), ml = l << lz;
  const unsigned rl = fx_shl(mh, ml, 21), up = (ml >> 10) & 1u;   // bits 42..11, and the first one dropped
  // the leading one adds 1 to the exponent field, and so does a carry out of the rounding
  unsigned long long b = ((((unsigned long long)((mh >> 11) + ((unsigned)(base - lz - 1) << 20))) << 32) | rl) + up;
  if (h == 0) b = 0;
  return fx_double(b | ((unsigned long long)(sg & 0x80000000u) << 32));
}
// ------------------------------------------------------------------ arithmetic
// signed halves of a value: a = h 2^32 + l
GPSOC_FX void fx_halves(long long a, int& h, int& l) {
  l = (int)(unsigned)a;
  h = (int)(a >> 32) + (int)((unsigned)a >> 31);
}
// a w 2^-shift for a complex value below 2^62.5 and a split twiddle (conj: its conjugate).  The
// product of the low halves is left out (below one unit), the middle ones are rounded.  TWICE: 2 a w 2^-shift.
template <bool CONJ, bool TWICE = false>
GPSOC_FX FxC fx_cmul(FxC a, FxW w) {
  int xh, xl, yh, yl;
  fx_halves(a.x, xh, xl);
  fx_halves(a.y, yh, yl);
  const int ph = CONJ ? w.yh : -w.yh, pl = CONJ ? w.yl : -w.yl;   // of a.y in the real part
  const int qh = -ph, ql = -pl;                                     // of a.x in the imaginary part
  const long long half = TWICE ? 1LL << 30 : 1LL << 31;
  const long long mr = half + (long long)xh * w.xl + (long long)xl * w.xh + (long long)yh * pl + (long long)yl * ph;
  const long long mi = half + (long long)yh * w.xl + (long long)yl * w.xh + (long long)xh * ql + (long long)xl * qh;
  FxC r;
  if (TWICE) {
    r.x = (mr >> 31) + 2 * ((long long)xh * w.xh + (long long)yh * ph);
    r.y = (mi >> 31) + 2 * ((long long)yh * w.xh + (long long)xh * qh);
    return r;
  }
  r.x = (mr >> 32) + (long long)xh * w.xh + (long long)yh * ph;
  r.y = (mi >> 32) + (long long)yh * w.xh + (long long)xh * qh;
  return r;
}
// sqrt(1/2) - 1 in units of 2^-64, as signed halves
constexpr long long kFxH1 = -0x4AFB0CCC06219B7CLL;
constexpr int fx_lo(long long k) { return (int)(unsigned)k; }
constexpr int fx_hi(long long k) { return (int)((k - fx_lo(k)) >> 32); }
GPSOC_FX FxC fx_shift(FxC a, int shift) {   // a 2^-shift, rounded
  a.x = (a.x + (1LL << (shift - 1))) >> shift;
  a.y = (a.y + (1LL << (shift - 1))) >> shift;
  return a;
}
// v sqrt(1/2), as v + v (sqrt(1/2) - 1)
GPSOC_FX long long fx_mul_h(long long v) {
  constexpr int kh = fx_hi(kFxH1), kl = fx_lo(kFxH1);
  int h, l;
  fx_halves(v, h, l);
  const long long m = (1LL << 31) + (long long)h * kl + (long long)l * kh;
  return v + (m >> 32) + (long long)h * kh;
}

GPSOC_FX FxC fx_add(FxC a, FxC b) { a.x += b.x; a.y += b.y; return a; }
GPSOC_FX FxC fx_sub(FxC a, FxC b) { a.x -= b.x; a.y -= b.y; return a; }
template <bool INV> GPSOC_FX FxC fx_mi(FxC a) {   // times -i (forward) or +i (inverse)
  FxC r;
  if (INV) { r.x = -a.y; r.y = a.x; } else { r.x = a.y; r.y = -a.x; }
  return r;
}
// times W_8 = (1 - i)/sqrt2 (forward), W_8^3 = (-1 - i)/sqrt2, conjugated for the inverse
template <bool INV> GPSOC_FX FxC fx_w8(FxC a) {
  FxC r;
  if (INV) { r.x = fx_mul_h(a.x - a.y); r.y = fx_mul_h(a.x + a.y); }
  else { r.x = fx_mul_h(a.x + a.y); r.y = fx_mul_h(a.y - a.x); }
  return r;
}
template <bool INV> GPSOC_FX void fx_dft4(FxC& v0, FxC& v1, FxC& v2, FxC& v3) {
  const FxC a0 = fx_add(v0, v2), a1 = fx_sub(v0, v2);
  const FxC a2 = fx_add(v1, v3), a3 = fx_mi<INV>(fx_sub(v1, v3));
  v0 = fx_add(a0, a2);
  v2 = fx_sub(a0, a2);
  v1 = fx_add(a1, a3);
  v3 = fx_sub(a1, a3);
}
// R-point DFT in place on R values, natural order
template <bool INV, int R> GPSOC_FX void fx_dft(FxC* v) {
  if constexpr (R == 2) {
    const FxC t = v[0];
    v[0] = fx_add(t, v[1]);
    v[1] = fx_sub(t, v[1]);
  } else if constexpr (R == 4) {
    fx_dft4<INV>(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    FxC e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    FxC o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    fx_dft4<INV>(e0, e1, e2, e3);
    fx_dft4<INV>(o0, o1, o2, o3);
    const FxC t1 = fx_w8<INV>(o1), t2 = fx_mi<INV>(o2), t3 = fx_mi<INV>(fx_w8<INV>(o3));
    v[0] = fx_add(e0, o0); v[4] = fx_sub(e0, o0);
    v[1] = fx_add(e1, t1); v[5] = fx_sub(e1, t1);
    v[2] = fx_add(e2, t2); v[6] = fx_sub(e2, t2);
    v[3] = fx_add(e3, t3); v[7] = fx_sub(e3, t3);
  }
}

#if defined(__CUDACC__)
// ------------------------------------------------------------------ transforms in shared memory
__device__ const FxTable g_fx_table = fx_make_table();

// Twiddles for transforms of length n with E elements per thread: entry (r, j) = W_n^(r j) 2^-shift,
// r < E, j < n/E, at the padded index pad(r n/E + j).
template <class Pad>
__device__ __forceinline__ void fx_load_tw(FxW* s_tw, int n, int ept, Pad pad) {
  const int lc = __ffs(n / ept) - 1, step = kFxTable / n, shift = (ept == 8) ? 3 : 2;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int r = i >> lc, j = i & ((1 << lc) - 1);
    const longlong2 w = reinterpret_cast<const longlong2*>(g_fx_table.c)[r * j * step];
    FxW o;
    fx_split(w.x, shift, o.xh, o.xl);
    fx_split(w.y, shift, o.yh, o.yl);
    s_tw[pad(i)] = o;
  }
}

// largest key of the G threads (a power of two) that share a line, over their warp
__device__ __forceinline__ int fx_line_max(int key, int G) {
  if (G >= 32) return __reduce_max_sync(0xffffffffu, key);
  for (int o = 1; o < G; o <<= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
  return key;
}
// the warp's barrier or the block's.  One opaque instruction pair: with a branch around the two the
// compiler makes two copies of the passes, and doubles their registers
__device__ __forceinline__ void fx_sync(bool warp) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %0, 0;\n\t@p bar.warp.sync 0xffffffff;\n\t@!p bar.sync 0;\n\t}"
               :: "r"((int)warp) : "memory");
}

// One pass of radix R (see stockham_pass) over the line at p: FIRST reads FP64 values and scales
// the line, `last` writes FP64 values; between passes the line holds fixed-point values in the
// same places.  sc: exponent of a unit of the line; the results are scaled by 2^-down (the 1/n of
// inverse transforms, for nothing).
template <int R, int E, bool FIRST, class Pad>
__device__ __forceinline__ void fx_pass(FxC* p, bool act, int g0, int N, int Ns, const FxW* tw, bool last, int& sc,
                                        int down, int* s_key, bool warp, Pad pad) {
  constexpr int PER = E / R;
  const int NR = N / R, G = N / E;
  FxC v[E];
  int key = 0;
  if (act) {
#pragma unroll
    for (int u = 0; u < PER; ++u)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const FxC z = p[pad(g0 + u * G + r * NR)];
        v[u * R + r] = z;
        if (FIRST) {
          key = max(key, (int)((unsigned)(z.x >> 32) & 0x7fffffffu));
          key = max(key, (int)((unsigned)(z.y >> 32) & 0x7fffffffu));
        }
      }
  } else {
    // defined on this path too, or the values of every pass stay live around the loop over lines
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = FxC{0, 0};
  }
  if (FIRST) {
    key = fx_line_max(key, G);
    if (!warp && (threadIdx.x & 31) == 0) s_key[threadIdx.x >> 5] = key;
  }
  fx_sync(warp);
  if (act) {
    constexpr int F = kFxBits<R>;
    if (FIRST) {
      if (!warp) {
        const int w0 = (threadIdx.x / G) * (G >> 5);
        for (int w = 0; w < (G >> 5); ++w) key = max(key, s_key[w0 + w]);
      }
      const int em = max(key >> 20, 1);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        v[e].x = fx_of(__longlong_as_double(v[e].x), em, F);
        v[e].y = fx_of(__longlong_as_double(v[e].y), em, F);
      }
      sc = em == 0x7ff ? 4096 : em - 1022 - F - down;
    } else {
      sc += kFxShift<E>;
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int g = g0 + u * G;
      const int k = g & (Ns - 1);
      if (!FIRST) {
        // W_N^(r k N / (Ns R)) 2^-shift: entry (r, k N / (Ns R)) of the table (R = E)
        const int j = k * (N / (Ns * R));
        v[u * R] = fx_shift(v[u * R], kFxShift<E>);
#pragma unroll
        for (int r = 1; r < R; ++r) v[u * R + r] = fx_cmul<false, E == 2>(v[u * R + r], tw[pad(r * G + j)]);
      }
      fx_dft<false, R>(&v[u * R]);
      const int ob = (g - k) * R + k;
      if (last) {
        const int base = fx_plain(sc) ? 1086 + sc : 1086;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          FxC z = v[u * R + q];
          z.x = __double_as_longlong(fx_to(z.x, base));
          z.y = __double_as_longlong(fx_to(z.y, base));
          p[pad(ob + q * Ns)] = z;
        }
        if (!fx_plain(sc)) {   // rare, and not unrolled: exponents at the ends of the FP64 range, infinities, NaN
          const FxUnit unit = fx_unit(sc);
#pragma unroll 1
          for (int q = 0; q < R; ++q) {
            double2* z = reinterpret_cast<double2*>(&p[pad(ob + q * Ns)]);
            *z = make_double2((z->x * unit.f1) * unit.f2, (z->y * unit.f1) * unit.f2);
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < R; ++q) p[pad(ob + q * Ns)] = v[u * R + q];
      }
    }
  }
  fx_sync(warp);
}

// The transform of length N = 2^L of one line per G = N/E threads: FP64 values in and out.
template <int E, class Pad>
__device__ __forceinline__ void fx_fft(FxC* p, bool act, int g0, int L, int down, const FxW* tw, int* s_key, bool warp,
                                       Pad pad) {
  const int N = 1 << L;
  constexpr int LE = (E == 8) ? 3 : (E == 4) ? 2 : 1;
  const int rem = L % LE, full = L / LE;
  int Ns = E, n = 1, sc = 0;
  if (rem == 1) { fx_pass<2, E, true>(p, act, g0, N, 1, tw, full == 0, sc, down, s_key, warp, pad); Ns = 2; n = 0; }
  else if (LE == 3 && rem == 2) { fx_pass<4, E, true>(p, act, g0, N, 1, tw, full == 0, sc, down, s_key, warp, pad); Ns = 4; n = 0; }
  else fx_pass<E, E, true>(p, act, g0, N, 1, tw, full == 1, sc, down, s_key, warp, pad);
#pragma unroll 1
  for (; n < full; ++n) {
    fx_pass<E, E, false>(p, act, g0, N, Ns, tw, n == full - 1, sc, down, s_key, warp, pad);
    Ns *= E;
  }
}
#endif  // __CUDACC__

}  // namespace gpsoc
