// Shared-memory Stockham FFTs, radix 16 or 8 (plus one smaller pass when log2 N
// is not a multiple of 4 or 3), natural order in and out.
//
// Transform convention (Section 3.2): forward X_k = sum_m x_m exp(-2 pi i k m / N),
// inverse with exp(+...) and no 1/N (callers fold the 1/N into their epilogues).
//
// A pass of radix R with Ns = product of the radices of the earlier passes
// treats group g in [0, N/R): it reads x[g + r N/R] (r < R), multiplies element r
// by W_N^(r k N / (Ns R)) with k = g mod Ns, takes the R-point DFT and writes
// output q to x[(g / Ns) Ns R + k + q Ns].  Every pass reads all values into
// registers, synchronises, then writes: the transform runs in place.
//
// Lines are padded in shared memory, element e at e + (e >> 4) for 8-byte and
// e + (e >> 3) for 16-byte complex values: the contiguous reads of every pass
// and the strided writes of the first pass then avoid bank conflicts.  tw holds
// W_N^(r j) = exp(-2 pi i r j / N) for r < E, j < N/E at the padded index
// fft_pad(r N/E + j) (E = elements per thread, the radix of the last pass).
#pragma once

#include "fixfft.cuh"
#include "gpsoc_internal.cuh"

namespace gpsoc {

// one gap per 16 elements for 8-byte complex values (a half-warp's 16 consecutive
// elements fill one 128-byte wavefront), one per 8 for 16-byte values
template <class C> constexpr int kPadShift = (sizeof(C) == 8) ? 4 : 3;
template <class C> __host__ __device__ __forceinline__ int fft_pad(int e) { return e + (e >> kPadShift<C>); }
template <class C> __host__ __device__ __forceinline__ int fft_padded_len(int n) { return n + (n >> kPadShift<C>); }

// multiply by -i
template <class C> __device__ __forceinline__ C mul_mi(C a) {
  C r;
  r.x = a.y;
  r.y = -a.x;
  return r;
}

template <class C> __device__ __forceinline__ void dft2(C& a, C& b) {
  const C t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

// 4-point DFT of (v0, v1, v2, v3) in place, natural output order
template <class C> __device__ __forceinline__ void dft4(C& v0, C& v1, C& v2, C& v3) {
  const C a0 = cadd(v0, v2), a1 = csub(v0, v2);
  const C a2 = cadd(v1, v3), a3 = mul_mi<C>(csub(v1, v3));
  v0 = cadd(a0, a2);
  v2 = csub(a0, a2);
  v1 = cadd(a1, a3);
  v3 = csub(a1, a3);
}

// 8-point DFT in place: two 4-point DFTs (even / odd inputs) combined with W_8^q
template <class C> __device__ __forceinline__ void dft8(C (&v)[8]) {
  using R = decltype(v[0].x);
  C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
  C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<C>(e0, e1, e2, e3);
  dft4<C>(o0, o1, o2, o3);
  const R h = (R)0.70710678118654752440;
  // W_8^1 = (1 - i)/sqrt2, W_8^2 = -i, W_8^3 = (-1 - i)/sqrt2
  C t1, t3;
  t1.x = h * (o1.x + o1.y); t1.y = h * (o1.y - o1.x);
  t3.x = h * (o3.y - o3.x); t3.y = -h * (o3.x + o3.y);
  const C t2 = mul_mi<C>(o2);
  v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
  v[1] = cadd(e1, t1); v[5] = csub(e1, t1);
  v[2] = cadd(e2, t2); v[6] = csub(e2, t2);
  v[3] = cadd(e3, t3); v[7] = csub(e3, t3);
}

// v * exp(-i a) for a constant angle with cos a = c, sin a = s
template <class C, class R> __device__ __forceinline__ C rot_const(C v, R c, R s) {
  C r;
  r.x = v.x * c + v.y * s;
  r.y = v.y * c - v.x * s;
  return r;
}

// 16-point DFT in place: four 4-point DFTs over n1 (stride 4), the twiddles
// W_16^(n2 k1), four 4-point DFTs over n2; output k = k1 + 4 k2 in natural order
template <class C> __device__ __forceinline__ void dft16(C (&v)[16]) {
  using R = decltype(v[0].x);
  const R c1 = (R)0.92387953251128675613, s1 = (R)0.38268343236508977173, h = (R)0.70710678118654752440;
  C a[4][4];   // a[n2][k1]
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    C x0 = v[n2], x1 = v[4 + n2], x2 = v[8 + n2], x3 = v[12 + n2];
    dft4<C>(x0, x1, x2, x3);
    a[n2][0] = x0; a[n2][1] = x1; a[n2][2] = x2; a[n2][3] = x3;
  }
  // W_16^m for m = n2 k1: 1, 2, 3 (n2 = 1); 2, 4, 6 (n2 = 2); 3, 6, 9 (n2 = 3)
  a[1][1] = rot_const<C>(a[1][1], c1, s1);
  a[1][2] = rot_const<C>(a[1][2], h, h);
  a[1][3] = rot_const<C>(a[1][3], s1, c1);
  a[2][1] = rot_const<C>(a[2][1], h, h);
  a[2][2] = mul_mi<C>(a[2][2]);
  a[2][3] = rot_const<C>(a[2][3], -h, h);
  a[3][1] = rot_const<C>(a[3][1], s1, c1);
  a[3][2] = rot_const<C>(a[3][2], -h, h);
  a[3][3] = rot_const<C>(a[3][3], -c1, -s1);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    C y0 = a[0][k1], y1 = a[1][k1], y2 = a[2][k1], y3 = a[3][k1];
    dft4<C>(y0, y1, y2, y3);
    v[k1] = y0; v[k1 + 4] = y1; v[k1 + 8] = y2; v[k1 + 12] = y3;
  }
}

// DFT of radix R on the R values starting at v[off] (R in {2, 4, 8, 16})
template <class C, int R, int E> __device__ __forceinline__ void dftR(C (&v)[E], int off) {
  if constexpr (R == 16) {
    C w[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) w[r] = v[off + r];
    dft16<C>(w);
#pragma unroll
    for (int r = 0; r < 16; ++r) v[off + r] = w[r];
  } else if constexpr (R == 8) {
    C w[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) w[r] = v[off + r];
    dft8<C>(w);
#pragma unroll
    for (int r = 0; r < 8; ++r) v[off + r] = w[r];
  } else if constexpr (R == 4) {
    dft4<C>(v[off], v[off + 1], v[off + 2], v[off + 3]);
  } else {
    dft2<C>(v[off], v[off + 1]);
  }
}

// One Stockham pass of radix R over the line at p, E elements per thread (E >= R): this thread's
// E/R groups are g0 + u N/E (u < E/R).  Inactive threads only synchronise.
template <class C, int R, int E>
__device__ __forceinline__ void stockham_pass(C* p, bool act, int g0, int N, int Ns, const C* tw, bool warp) {
  constexpr int PER = E / R;   // radix-R groups of one thread
  C v[E];
  const int NR = N / R;
  if (act) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int g = g0 + u * (N / E);
#pragma unroll
      for (int r = 0; r < R; ++r) v[u * R + r] = p[fft_pad<C>(g + r * NR)];
    }
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = mk<C>(0.0f, 0.0f);   // as in fx_pass
  }
  fx_sync(warp);
  if (act) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int g = g0 + u * (N / E);
      const int k = g & (Ns - 1);
      if (k != 0) {
        // W_N^(r k N / (Ns R)): entry (r, k N / (Ns R)) of the table (R = E here:
        // only the first pass, with k = 0, can have a smaller radix)
        const int j = k * (N / (Ns * R));
#pragma unroll
        for (int r = 1; r < R; ++r) v[u * R + r] = cmul(v[u * R + r], tw[fft_pad<C>(r * (N / E) + j)]);
      }
      dftR<C, R, E>(v, u * R);
      const int ob = (g - k) * R + k;
#pragma unroll
      for (int q = 0; q < R; ++q) p[fft_pad<C>(ob + q * Ns)] = v[u * R + q];
    }
  }
  fx_sync(warp);
}

// The transform of length N = 2^L (N >= E) of one line per N/E threads (E in {2, 4, 8, 16}:
// radix-E passes plus one smaller pass when log2 N is not a multiple of log2 E).
template <class C, int E>
__device__ __forceinline__ void stockham_fft(C* p, bool act, int g0, int L, const C* tw, bool warp) {
  const int N = 1 << L;
  int Ns = 1;
  constexpr int LE = (E == 16) ? 4 : (E == 8) ? 3 : (E == 4) ? 2 : 1;
  const int rem = L % LE;
  if (rem == 1) { stockham_pass<C, 2, E>(p, act, g0, N, Ns, tw, warp); Ns *= 2; }
  else if (rem == 2) { if constexpr (E >= 4) { stockham_pass<C, 4, E>(p, act, g0, N, Ns, tw, warp); Ns *= 4; } }
  else if constexpr (E == 16) {
    if (rem == 3) { stockham_pass<C, 8, E>(p, act, g0, N, Ns, tw, warp); Ns *= 8; }
  }
#pragma unroll 1
  for (int n = 0; n < L / LE; ++n) { stockham_pass<C, E, E>(p, act, g0, N, Ns, tw, warp); Ns *= E; }
}

struct FftPad16 { __device__ __forceinline__ int operator()(int e) const { return fft_pad<double2>(e); } };

// Forward transforms, in place, of nlines lines of padded length NP that start `off` values behind
// the start of the dynamic shared memory, which holds the twiddle table.  Every thread of the
// block calls it, the lines complete in shared memory; they are complete again on return.  FP64 results
// are scaled by 2^-down.
//
// A line belongs to N/E consecutive threads.  When these are within one warp (N/E <= 32: lines up
// to 256 with 8 elements per thread) its passes need no block barrier, only the warp's; before,
// each pass waited twice for the whole block (24-27% of the stalls of the 256^2 passes).
//
// The inverse transform is the forward one read at index -j mod n, so that one inlined copy serves
// every transform of a kernel: unrolled passes are 10 to 20 KB of instructions, run once or twice by a block, and a third of
// the stalls of the FP64 column passes was waiting for them (ncu, no_instruction) with three.
template <class C, int E>
__device__ __forceinline__ void fft_lines_e(int off, int nlines, int NP, int L, int down) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_key[32];
  const C* tw = reinterpret_cast<const C*>(smem_raw);
  C* buf = reinterpret_cast<C*>(smem_raw) + off;
  const int LG = L - (E == 16 ? 4 : E == 8 ? 3 : E == 4 ? 2 : 1);   // log2 of the threads of a line
  const int per = blockDim.x >> LG;
  const int q0 = threadIdx.x >> LG, g0 = threadIdx.x & ((1 << LG) - 1);
  const bool warp = LG <= 5;
#pragma unroll 1
  for (int b = 0; b < nlines; b += per) {
    const int q = b + q0;
    const bool act = q0 < per && q < nlines;
    C* p = buf + (act ? q : 0) * NP;
    int g = g0;
    asm volatile("" : "+r"(g));   // keeps every pass's addresses from being computed ahead of the loop, into spills
    if constexpr (sizeof(C) == 16)
      fx_fft<E>(reinterpret_cast<FxC*>(p), act, g, L, down, reinterpret_cast<const FxW*>(tw), s_key, warp, FftPad16{});
    else
      stockham_fft<C, E>(p, act, g, L, tw, warp);
  }
  __syncthreads();
}

}  // namespace gpsoc
