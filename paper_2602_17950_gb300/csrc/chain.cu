// Spectral passes of the Hamiltonian and preconditioner chains.
//
// A d-dimensional transform is a sequence of 1-D axis passes; each pass loads
// a tile into shared memory, runs Stockham FFTs there and stores back with
// coalesced accesses.  Row passes (x, contiguous) take R whole rows of all
// three components; column passes (y or z, strided) take a tile of TC
// consecutive inner indices across the whole axis for all three components,
// so the 3x3 spin-orbit symbol and the pointwise spin terms see every
// component of a point in one block.
//
// Chains (Section 3.2 symbols; Section 2.2 operators; Section 3.4 preconditioner):
//   H chain 2D:  X fwd -> Y (fwd, symbol, inv, rotation pieces) -> X inv + pointwise
//   H chain 3D:  X fwd -> Y fwd -> Z (fwd, symbol, inv) -> Y inv + rotation -> X inv + pointwise
//   P_C chain:   X fwd of P_V^{1/2} r -> [Y fwd] -> last axis (fwd, divide, inv) -> [Y inv] -> X inv, P_V^{1/2}
// Rotation term -Omega Lz phi = Omega y D_x phi - Omega x D_y phi with D = -i d:
// the y D_x piece is folded into the spectral-in-x array before the last x
// inverse (y is constant along an x row), the x D_y piece is carried as a
// second array G = F_y^{-1}[v_y F_y A] and multiplied by x after the x inverse.
#include <map>
#include <type_traits>
#include <mutex>

#include "gpsoc_internal.cuh"
#include "hypoint.cuh"
#include "scalar.cuh"
#include "fft.cuh"

namespace gpsoc {

static constexpr int kThreads = 384;
// reduction scratch (doubles) behind the tiles: block_reduce needs 16 per warp + 16
static constexpr int kRedDoubles = 16 * (kThreads / 32) + 16;

// elements per thread of the FP64 transforms of a tile of ept (see fft_lines)
__device__ __forceinline__ int fx_ept(int ept, int n) { return (ept == 2 && n > 64) ? 4 : ept; }

// Twiddle table in shared memory for transforms with E elements per thread:
// entry (r, j) = W_n^(r j), r < E, j < n/E, at the padded index fft_pad(r n/E + j).
// The last pass (radix E, Ns = n/E) reads j = k for consecutive groups k:
// consecutive addresses; earlier passes read j = k n/(Ns E) for few distinct k.
// FP64 passes transform in fixed point (fixfft.cuh) with a table of their own.
template <class T>
__device__ __forceinline__ void load_tw(cx_t<T>* s_tw, const cx_t<T>* tw, int n, int ept) {
  if constexpr (sizeof(T) == 8) {
    fx_load_tw(reinterpret_cast<FxW*>(s_tw), n, fx_ept(ept, n), FftPad16{});
  } else {
    const int lc = __ffs(n / ept) - 1;   // log2(n / E): n and E are powers of two
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int r = i >> lc, j = i & ((1 << lc) - 1);
      s_tw[fft_pad<cx_t<T>>(i)] = tw[r * j];
    }
  }
}

// transforms of nlines lines at offset off (see fft_lines_e).  R16: the kernel may run radix-16 passes
// (FP32 column passes only: the code path sets the register allocation of the whole kernel).
// FP64 tiles of 2 elements per thread transform lines of more than 64 points with half their threads, 4
// elements each: radix-2 passes are twice as many and pay only where a solve is bound by the latency of
// one warp per line (one 64^2 solve, 31 iterations, takes 6% less with 2 than with 4; one 128^2 solve,
// which keeps 4, takes 0.6% more with this rule, for a reason not found).
template <class C, bool R16 = false>
__device__ __forceinline__ void fft_lines(int off, int nlines, int NP, int L, int ept, int down = 0) {
  if constexpr (R16 && sizeof(C) == 8) {
    if (ept == 16) { fft_lines_e<C, 16>(off, nlines, NP, L, down); return; }
  }
  if (ept == 8) fft_lines_e<C, 8>(off, nlines, NP, L, down);
  else if (ept == 4 || (sizeof(C) == 16 && L > 6)) fft_lines_e<C, 4>(off, nlines, NP, L, down);
  else fft_lines_e<C, 2>(off, nlines, NP, L, down);
}

// padded length of a column line in shared memory
template <class C> __host__ __device__ __forceinline__ int col_line_len(int n, int tc) {
  // tiles are loaded with consecutive threads on consecutive columns, then on
  // consecutive rows: S complex values fill a 128-byte wavefront, so the line
  // stride is made S / tc modulo S (tc < S) or odd (tc >= S), which puts the
  // values one half-warp (FP32) or quarter-warp (FP64) touches on distinct banks
  constexpr int S = (sizeof(C) == 8) ? 16 : 8;
  const int base = fft_padded_len<C>(n);
  if (tc >= S) return base | 1;
  const int want = S / tc;
  return base + ((want - base % S) + S) % S;
}

// spin terms shared by the pointwise epilogues (working precision W):
//   a = conj(p0) p1 + conj(pm) p0  so that F_-/sqrt2 = a, F_+/sqrt2 = conj(a),
//   F_x = sqrt2 Re a, F_y = -sqrt2 Im a, F_z = |p1|^2 - |pm|^2, |F|^2 = 2|a|^2 + F_z^2.
template <class W, class C1, class C2, class C3>
__device__ __forceinline__ void spin_a(C1 p1, C2 p0, C3 pm, W& ar, W& ai) {
  ar = (W)p0.x * (W)p1.x + (W)p0.y * (W)p1.y + (W)pm.x * (W)p0.x + (W)pm.y * (W)p0.y;
  ai = (W)p0.x * (W)p1.y - (W)p0.y * (W)p1.x + (W)pm.x * (W)p0.y - (W)pm.y * (W)p0.x;
}

// 1/sqrt(x), x > 0.  FP64: from the FP32 value (the integer pipes convert), 4 FP64 instructions against 9 of the
// library's; outside the FP32 range the library
__device__ __forceinline__ float rsqrt_w(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_w(double x) {
  return rsqrt_in_range(x) ? rsqrt_refine(x, widen_f(rsqrtf(narrow_f(x)))) : rsqrt(x);
}
// larger of two values, the second positive: their bits are ordered alike (and a negative or
// smaller first one is below), without the FP64 pipe
__device__ __forceinline__ float max_pos(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double max_pos(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b) ? b : a;
}

// write per-thread partial sums (working precision) as a deterministic block total in FP64
// (FP32 partials are added in double-float, which carries more bits than the partials hold)
template <int K, class W>
__device__ __forceinline__ void store_partials(const W (&acc)[K], const int (&slots)[K], const bool (&mx)[K],
                                               double* red, double* part, long long sbase_slot, int pmax, int blk, int nb,
                                               unsigned* gcnt, double* tail) {
  double v[K];
  if constexpr (sizeof(W) == 4 && K >= 2) {
    block_reduce_df<K>(acc, v, red);     // FP32 partials: double-float sums on the FP32 pipes
  } else if constexpr (K == 1 && sizeof(W) == 4) {
    v[0] = mx[0] ? block_max((double)acc[0], red) : block_sum_f(acc[0], red);
  } else if (K == 1 && mx[0]) {
    v[0] = block_max(acc[0], red);
  } else {
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = (double)acc[k];
    block_reduce<K>(v, red, mx);
  }
  put_partials<K>(part, sbase_slot, pmax, blk, slots, v, mx, sizeof(W) == 4);
  using V = std::conditional_t<sizeof(W) == 4, DF, double>;
  if (K == 1 && mx[0]) group_max<V>(part + sbase_slot * pmax, pmax, slots[0], blk, nb, gcnt, tail);
  else group_sums<V, K>(part + sbase_slot * pmax, pmax, slots, blk, nb, gcnt, tail);
}

// ============================================================== row passes (x axis)
// Working precision W = T: FP64 kernels compute in double, FP32 kernels in float
// (per-thread partial sums in T, block and grid reductions in FP64).
//
// Sizes are powers of two, so indices are split by shifts (integer divisions, two of them of 64 bits
// per point, were a third of the instructions of the FP32 passes).  The twiddle table is set up before the
// wait for the kernel before; the tiles of the inverse passes come by asynchronous copies.
template <class T, int MODE>
__device__ __forceinline__ void row_pass(const ChainArgs<T>& A, int R, int ept) {
  using C = cx_t<T>;
  using W = T;
  using PV = std::conditional_t<sizeof(T) == 4, DF, double>;   // format of the sum partials
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int last_flag;
  constexpr bool fwd = (MODE == ROW_FWD_PLAIN || MODE == ROW_FWD_UPD || MODE == ROW_FWD_PROJ || MODE == ROW_FWD_PRE ||
                        MODE == ROW_FWD_PRE_HY);
  constexpr bool two = (MODE == ROW_INV_H || MODE == ROW_INV_P || MODE == ROW_INV_LIN || MODE == ROW_INV_P_HY);
  const int nx = A.g.n[0], Lx = A.g.log2n[0], Ly = A.g.log2n[1], ny = A.g.n[1];
  const long long npts = A.g.npts;
  const int bps = (int)(npts >> Lx) / R;
  const int s = blockIdx.x / bps;
  const int rb = blockIdx.x - s * bps;
  C* s_tw = (C*)smem_raw;
  load_tw<T>(s_tw, A.tw[0], nx, ept);
  pdl_wait();
  if (s >= A.nsolve || !gate_ok(A.st, A.gate, s)) return;
  const int b0 = fft_padded_len<C>(nx);   // the lines lie behind the table
  C* buf0 = s_tw + b0;
  const int per = R << Lx;            // elements of one component in the tile
  const int NP = b0, CP = R * NP;     // padded line length, component stride in smem
  C* buf1 = buf0 + 3 * CP;
  double* red = (double*)(buf1 + (two ? 3 * CP : 0));
  // scratch of a fused scalar step: over the tile, which is done with by then (32 doubles per warp are
  // at most half of its 24 or 48 bytes per element)
  double* tail = (double*)smem_raw;
  unsigned* gcnt = A.gcnt + (long long)s * A.gmax;
  // this tile's first point; component c is npts further on
  const long long base = (long long)s * 3 * npts + ((long long)rb * R << Lx);
  const int row0 = rb * R;
  const long long sslot = (long long)s * NSLOT;
  const SolveState& S = A.st[s];
  const PhysDev& ph = A.phys[s];

  if (!fwd || MODE == ROW_FWD_PLAIN) {
    for (int e = threadIdx.x; e < per; e += blockDim.x) {
      const int pos = (e >> Lx) * NP + fft_pad<C>(e & (nx - 1));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        copy_async(&buf0[c * CP + pos], A.in0 + base + c * npts + e);
        if (two) copy_async(&buf1[c * CP + pos], A.in1 + base + c * npts + e);
      }
    }
  }
  // the solve's scalars, read before the transforms
  const W c0 = pick<W>(ph.c0, ph.fc0), c1 = pick<W>(ph.c1, ph.fc1), Om = pick<W>(ph.Omega, ph.fOmega);
  const W al[3] = {pick<W>(S.alpha[0], S.falpha[0]), pick<W>(S.alpha[1], S.falpha[1]), pick<W>(S.alpha[2], S.falpha[2])};
  const int pk = A.sc.opts.precond;
  const bool use_pv = (pk == GPSOC_PRECOND_COMBINED || pk == GPSOC_PRECOND_POTENTIAL);

  if (fwd) {
    W acc[1] = {(W)0};
    const W cproj = pick<W>(S.cproj, S.fcproj), mu = A.given_r ? (W)0 : pick<W>(S.mu, S.fmu), beta = pick<W>(S.beta, S.fbeta);
    const bool use_prev = (MODE == ROW_FWD_PROJ) && beta != (W)0;
    const bool upd = (MODE == ROW_FWD_UPD) && S.pending != 0;
    const bool dphi = upd && A.sc.opts.stop == GPSOC_STOP_DPHI;   // only the stop1 test reads max |dPhi|
    const W usc = pick<W>(S.upd_scale, S.fupd_scale);
    const W uc = usc * pick<W>(S.upd_c, S.fupd_c), us = usc * pick<W>(S.upd_s, S.fupd_s);
    const double mu64 = S.mu;
    if (MODE == ROW_FWD_PLAIN) copy_wait();
    else for (int e = threadIdx.x; e < per; e += blockDim.x) {
      const int r = e >> Lx, j = e & (nx - 1);
      const long long at = base + e;
      const int pos = r * NP + fft_pad<C>(j);
      if (MODE == ROW_FWD_UPD) {
        // the step accepted by the previous iteration: Phi <- (cos t Phi + sin t P/|P|)/norm
        // (Eqs. formula-pcg, update); max |dPhi|^2 for the stop1 test
        C f[3], p[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          f[c] = A.in0[at + c * npts];
          if (upd) p[c] = A.in2[at + c * npts];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          C o = f[c];
          if (upd) {
            o = mk<C>(uc * f[c].x + us * p[c].x, uc * f[c].y + us * p[c].y);
            if (dphi) {
              const W dr = o.x - f[c].x, di = o.y - f[c].y;
              acc[0] = max_pos(acc[0], dr * dr + di * di);
            }
            A.out1[at + c * npts] = o;
          }
          buf0[c * CP + pos] = o;
        }
      } else if (MODE == ROW_FWD_PROJ) {
        // D = -z + beta P_prev, P = D - Re<D, Phi> Phi (Eq. formula-project); reduce ||P||^2
        C z[3], f[3], q[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          z[c] = A.in0[at + c * npts];
          f[c] = A.in1[at + c * npts];
          q[c] = use_prev ? A.in2[at + c * npts] : mk<C>((W)0, (W)0);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          W dr = -z[c].x, di = -z[c].y;
          if (use_prev) { dr += beta * q[c].x; di += beta * q[c].y; }
          C p;
          p.x = dr - cproj * f[c].x;
          p.y = di - cproj * f[c].y;
          A.out1[at + c * npts] = p;
          acc[0] += p.x * p.x + p.y * p.y;
          buf0[c * CP + pos] = p;
        }
      } else if (MODE == ROW_FWD_PRE_HY) {
        // GPSOC_HYBRID: r = H Phi - mu Phi in FP64 from the FP64 state and H(Phi) (the residual
        // keeps FP64 accuracy: one fused multiply-add each), stored as FP32; the preconditioner's
        // transforms then run on P_V^{1/2} r in FP32, P_V from the FP64 state's density. max |r| is
        // that of the FP64 r. 6 FP64 instructions a point (22 with the density and the conversions on that
        // pipe, which bound the pass: 308k of its 397k cycles at 64 x 256^2)
        double2 f[3], h[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          f[c] = A.phi64[at + c * npts];
          h[c] = A.hl64[at + c * npts];
        }
        const long long pt = at - (long long)s * 3 * npts;
        const W rho = A.rho32[(long long)s * npts + pt];
        const int row = row0 + r;
        const W V = trap_value<W>(A.trap, A.g, j, row & (ny - 1), row >> Ly, pt);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const DF rx = dw_of(h[c].x - mu64 * f[c].x), ry = dw_of(h[c].y - mu64 * f[c].y);
          const C rc = mk<C>(rx.hi, ry.hi);
          A.out1[at + c * npts] = rc;
          acc[0] = max_pos(acc[0], hy_square(rx, ry));
          const W den = max_pos(al[c] + (V + c0 * rho), (W)1e-12 * al[c]);
          const W sc = use_pv ? rsqrt_w(den) : (W)1;
          buf0[c * CP + pos] = mk<C>(rc.x * sc, rc.y * sc);
        }
      } else {  // ROW_FWD_PRE: r = H Phi - mu Phi, then P_V^{1/2} r (Eq. PreCondPot)
        C f[3], h[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          f[c] = A.in1[at + c * npts];
          h[c] = A.in0[at + c * npts];
        }
        W rho = (W)0;
#pragma unroll
        for (int c = 0; c < 3; ++c) rho += f[c].x * f[c].x + f[c].y * f[c].y;
        const int row = row0 + r;
        const W V = trap_value<W>(A.trap, A.g, j, row & (ny - 1), row >> Ly, at - (long long)s * 3 * npts);
        const W w = V + c0 * rho;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          C rr;
          rr.x = h[c].x - mu * f[c].x;
          rr.y = h[c].y - mu * f[c].y;
          A.out1[at + c * npts] = rr;
          acc[0] = max_pos(acc[0], rr.x * rr.x + rr.y * rr.y);
          const W sc = use_pv ? rsqrt_w(max_pos(al[c] + w, (W)1e-12 * al[c])) : (W)1;
          buf0[c * CP + pos] = mk<C>(rr.x * sc, rr.y * sc);
        }
      }
    }
    __syncthreads();
    fft_lines<C>(b0, 3 * R, NP, Lx, ept);
    for (int e = threadIdx.x; e < per; e += blockDim.x) {
      const int pos = (e >> Lx) * NP + fft_pad<C>(e & (nx - 1));
#pragma unroll
      for (int c = 0; c < 3; ++c) A.out0[base + c * npts + e] = buf0[c * CP + pos];
    }
    // GPSOC_HYBRID sums ||P||^2 with the step model, in more precision
    const bool sum = (MODE == ROW_FWD_PROJ && !(A.sc.flags & 8)) || MODE == ROW_FWD_PRE || MODE == ROW_FWD_PRE_HY ||
                     (MODE == ROW_FWD_UPD && dphi);
    if (sum) {
      const bool mx[1] = {MODE != ROW_FWD_PROJ};
      const int slots[1] = {(MODE == ROW_FWD_PROJ) ? (int)SL_P2
                            : (MODE == ROW_FWD_PRE || MODE == ROW_FWD_PRE_HY) ? (int)SL_RINF : (int)SL_DPHIINF};
      store_partials<1, W>(acc, slots, mx, red, A.part, sslot, A.pmax, rb, bps, gcnt, tail);
    }
    if ((MODE == ROW_FWD_PRE || MODE == ROW_FWD_PRE_HY) && A.fuse && last_block(A.cnt, s, bps, &last_flag))
      sc_res(A.sc, s, tail);
    return;
  }

  // ---------------------------------------------------------------- inverse passes
  // forward transforms of both arrays' lines; the inverse ones are their values at index -j
  copy_wait();
  __syncthreads();
  // the 1/npts of the whole inverse transform: FP64 transforms scale their results by powers of two for nothing
  const int Ln = Lx + Ly + A.g.log2n[2];
  fft_lines<C>(b0, two ? 6 * R : 3 * R, NP, Lx, ept, MODE == ROW_INV_PLAIN ? 0 : Ln);
  const W inv_n = sizeof(T) == 4 ? (W)1 / (W)npts : (W)1;
  if (MODE == ROW_INV_PLAIN) {
    const W sc = (W)A.scale;
    for (int e = threadIdx.x; e < per; e += blockDim.x) {
      const int pos = (e >> Lx) * NP + fft_pad<C>(-e & (nx - 1));
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const C v = buf0[c * CP + pos];
        A.out0[base + c * npts + e] = mk<C>(v.x * sc, v.y * sc);
      }
    }
    return;
  }
  if (MODE == ROW_INV_PRE) {
    // z = P_V^{1/2} F^-1[...] (Eq. PreCondMix); reduce Re<r, z>, Re<r_prev, z> (beta) and
    // Re<z, Phi>, Re<P_prev, Phi>, Re<r, P_prev> (the direction's projection and slope)
    W acc[5] = {(W)0, (W)0, (W)0, (W)0, (W)0};
    const bool use_prev = (A.in3 != nullptr) && !S.first;
    for (int e = threadIdx.x; e < per; e += blockDim.x) {
      const int r = e >> Lx, j = e & (nx - 1);
      const int pos = r * NP + fft_pad<C>(-j & (nx - 1));
      const long long at = base + e;
      W rho = (W)0;
      C f[3], rr[3], rp[3], pp[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        f[c] = A.in1[at + c * npts];
        rr[c] = A.in2[at + c * npts];
        if (use_prev) {
          rp[c] = A.in3[at + c * npts];
          pp[c] = A.in4[at + c * npts];
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) rho += f[c].x * f[c].x + f[c].y * f[c].y;
      const int row = row0 + r;
      const W V = trap_value<W>(A.trap, A.g, j, row & (ny - 1), row >> Ly, at - (long long)s * 3 * npts);
      const W w = V + c0 * rho;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const W sc = use_pv ? inv_n * rsqrt_w(max_pos(al[c] + w, (W)1e-12 * al[c])) : inv_n;
        const C v = buf0[c * CP + pos];
        const C z = mk<C>(v.x * sc, v.y * sc);
        A.out0[at + c * npts] = z;
        acc[0] += rr[c].x * z.x + rr[c].y * z.y;
        acc[2] += z.x * f[c].x + z.y * f[c].y;
        if (use_prev) {
          acc[1] += rp[c].x * z.x + rp[c].y * z.y;
          acc[3] += pp[c].x * f[c].x + pp[c].y * f[c].y;
          acc[4] += rr[c].x * pp[c].x + rr[c].y * pp[c].y;
        }
      }
    }
    const bool mx[5] = {false, false, false, false, false};
    const int slots[5] = {SL_RZ, SL_RPZ, SL_ZPHI, SL_PPHI, SL_RP};
    store_partials<5, W>(acc, slots, mx, red, A.part, sslot, A.pmax, rb, bps, gcnt, tail);
    if (A.fuse && last_block(A.cnt, s, bps, &last_flag)) sc_beta<PV>(A.sc, s, tail);
    return;
  }

  // ROW_INV_H / ROW_INV_P / ROW_INV_LIN: lin = F_x^-1(T')/npts - Omega x F_x^-1(G)/npts + V u
  const W Omn = Om * inv_n;
  double rphi = 0.0, pp = 0.0;           // ROW_INV_P_HY: Re<P, Phi> against the FP64 Phi and ||P||^2
  W acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = (W)0;
  W accR = (W)0;                         // ROW_INV_P: Re<P, Phi>
  for (int e = threadIdx.x; e < per; e += blockDim.x) {
    const int r = e >> Lx, j = e & (nx - 1);
    const int pos = r * NP + fft_pad<C>(-j & (nx - 1));
    const long long at = base + e;
    const int row = row0 + r;
    C u[3];  // Phi for ROW_INV_H, P for ROW_INV_P / ROW_INV_LIN
    C f[3], h[3];
    double2 f64[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = A.in2[at + c * npts];
      if (MODE == ROW_INV_P || MODE == ROW_INV_P_HY) {
        f[c] = A.in3[at + c * npts];
        h[c] = A.in4[at + c * npts];
      }
      if (MODE == ROW_INV_P_HY) f64[c] = A.phi64[at + c * npts];
    }
    const W ox = Omn * coord<W>(A.g, 0, j);
    const W V = trap_value<W>(A.trap, A.g, j, row & (ny - 1), row >> Ly, at - (long long)s * 3 * npts);
    W lin_r[3], lin_i[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const C t = buf0[c * CP + pos];
      const C gg = buf1[c * CP + pos];
      lin_r[c] = (t.x * inv_n - ox * gg.x) + V * u[c].x;
      lin_i[c] = (t.y * inv_n - ox * gg.y) + V * u[c].y;
    }
    if (MODE == ROW_INV_LIN) {
#pragma unroll
      for (int c = 0; c < 3; ++c) A.out0[at + c * npts] = mk<C>(lin_r[c], lin_i[c]);
      continue;
    }
    if (MODE == ROW_INV_H) {
      // nonlinear terms of Eqs. eigen1-eigen3: c0 rho phi + c1 (F.f) Phi
      W m[3];
      W rho = (W)0;
#pragma unroll
      for (int c = 0; c < 3; ++c) { m[c] = u[c].x * u[c].x + u[c].y * u[c].y; rho += m[c]; }
      W ax, ay;
      spin_a<W>(u[0], u[1], u[2], ax, ay);
      const W Fz = m[0] - m[2];
      const W c0r = c0 * rho, cz = c1 * Fz, cax = c1 * ax, cay = c1 * ay;
      // c1 (F.f)Phi: c1 [Fz p1 + a p0, conj(a) p1 + a pm, conj(a) p0 - Fz pm]
      W fr[3], fi[3];
      fr[0] = cz * u[0].x + (cax * u[1].x - cay * u[1].y);
      fi[0] = cz * u[0].y + (cax * u[1].y + cay * u[1].x);
      fr[1] = (cax * u[0].x + cay * u[0].y) + (cax * u[2].x - cay * u[2].y);
      fi[1] = (cax * u[0].y - cay * u[0].x) + (cax * u[2].y + cay * u[2].x);
      fr[2] = (cax * u[1].x + cay * u[1].y) - cz * u[2].x;
      fi[2] = (cax * u[1].y - cay * u[1].x) - cz * u[2].y;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc[0] += u[c].x * lin_r[c] + u[c].y * lin_i[c];
        A.out0[at + c * npts] = mk<C>(lin_r[c] + (c0r * u[c].x + fr[c]), lin_i[c] + (c0r * u[c].y + fi[c]));
        acc[3 + c] += V * m[c];
        acc[6 + c] += rho * m[c];
        acc[9 + c] += m[c];
      }
      acc[1] += rho * rho;
      acc[2] += (W)2 * (ax * ax + ay * ay) + Fz * Fz;
    } else {  // ROW_INV_P: step-model reductions (Eqs. an, bn and the sin/cos form of E(theta))
      if constexpr (MODE == ROW_INV_P_HY) {
        // H_lin P kept for the update of H_lin Phi by linearity; the radial part of P and ||P||^2 in FP64
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          A.out0[at + c * npts] = mk<C>(lin_r[c], lin_i[c]);
          hy_radial(rphi, pp, f64[c].x, f64[c].y, u[c].x, u[c].y);
        }
      }
      W mx_[3], mf[3], mp[3];   // Re(f conj(u)), |f|^2, |u|^2 per component
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        acc[0] += lin_r[c] * u[c].x + lin_i[c] * u[c].y;
        acc[1] += h[c].x * u[c].x + h[c].y * u[c].y;
        mx_[c] = f[c].x * u[c].x + f[c].y * u[c].y;
        mf[c] = f[c].x * f[c].x + f[c].y * f[c].y;
        mp[c] = u[c].x * u[c].x + u[c].y * u[c].y;
      }
      const W Rv = mx_[0] + mx_[1] + mx_[2], rf = mf[0] + mf[1] + mf[2], rp = mp[0] + mp[1] + mp[2];
      // spin vectors F(Phi), F(P) and the symmetric cross term Re F~(Phi, P), through
      // a(Phi + e P) = a(Phi) + e (a1 + a2) + e^2 a(P); Re F~ is half the e coefficient of F:
      // F_xy . G_xy = 2 Re(conj(a_F) a_G)
      W aFx, aFy, aPx, aPy, a1x, a1y, a2x, a2y;
      spin_a<W>(f[0], f[1], f[2], aFx, aFy);
      spin_a<W>(u[0], u[1], u[2], aPx, aPy);
      spin_a<W>(f[0], u[1], f[2], a1x, a1y);
      spin_a<W>(u[0], f[1], u[2], a2x, a2y);
      const W aXx = a1x + a2x, aXy = a1y + a2y;    // twice the cross term's a
      const W FFz = mf[0] - mf[2], FPz = mp[0] - mp[2], FXz = mx_[0] - mx_[2];
      if (MODE == ROW_INV_P) accR += Rv;
      acc[2] += rf * Rv;
      acc[3] += rf * rp;
      acc[4] += Rv * Rv;
      acc[5] += Rv * rp;
      acc[6] += rp * rp;
      acc[7] += (aFx * aXx + aFy * aXy) + FFz * FXz;
      acc[8] += (W)2 * (aFx * aPx + aFy * aPy) + FFz * FPz;
      acc[9] += (W)0.5 * (aXx * aXx + aXy * aXy) + FXz * FXz;
      acc[10] += (aXx * aPx + aXy * aPy) + FXz * FPz;
      acc[11] += (W)2 * (aPx * aPx + aPy * aPy) + FPz * FPz;
    }
  }
  if (MODE == ROW_INV_LIN) return;
  if (MODE == ROW_INV_H) {
    const bool mx12[12] = {};
    const int slots[12] = {SL_Q, SL_RHO2, SL_F2, SL_V0, SL_V1, SL_V2, SL_C0, SL_C1, SL_C2, SL_M0, SL_M1, SL_M2};
    store_partials<12, W>(acc, slots, mx12, red, A.part, sslot, A.pmax, rb, bps, gcnt, tail);
    if (A.fuse && last_block(A.cnt, s, bps, &last_flag)) sc_obs<PV>(A.sc, s, tail);
  } else {
    const int slots[14] = {SL_HPP, SL_HPHIP, SL_IFR, SL_IFP, SL_IRR, SL_IRP, SL_IPP,
                           SL_JFR, SL_JFP, SL_JRR, SL_JRP, SL_JPP, SL_RPHI, SL_P2};
    if constexpr (MODE == ROW_INV_P_HY) {
      const bool mx[14] = {};
      double v[14];
      block_reduce_df_fp64<12>(acc, rphi, pp, v, red);
      put_partials<14>(A.part, sslot, A.pmax, rb, slots, v, mx, true);
      group_sums<DF, 14>(A.part + sslot * A.pmax, A.pmax, slots, rb, bps, gcnt, tail);
    } else {
      W a13[13];
      int s13[13];
      const bool m13[13] = {};
#pragma unroll
      for (int k = 0; k < 13; ++k) { a13[k] = k < 12 ? acc[k] : accR; s13[k] = slots[k]; }
      store_partials<13, W>(a13, s13, m13, red, A.part, sslot, A.pmax, rb, bps, gcnt, tail);
    }
    if (A.fuse && last_block(A.cnt, s, bps, &last_flag)) sc_step<PV>(A.sc, s, tail);
  }
}

// Blocks of kThreads per SM each pass is compiled for: 3 (at most 56 registers, six 192-thread tiles per
// SM; the passes with fused sums spill a few values) for FP32, 2 (84 registers, four tiles) for FP64 and for
// the last pass of a hybrid iteration, whose Algorithm 2 step alone would take 113 for its grid sums.
template <class T, int MODE>
constexpr int row_blocks() { return sizeof(T) == 4 && MODE != ROW_INV_P_HY ? 3 : 2; }
template <class T, int MODE>
__global__ void __launch_bounds__(kThreads, row_blocks<T, MODE>()) k_row(ChainArgs<T> A, int R, int ept) {
  row_pass<T, MODE>(A, R, ept);
}

// ============================================================== column passes (y or z axis)
// Tile: inner indices [i0, i0 + TC) of the axis-`axis` lines at outer index o, all
// three components.  Shared memory holds every (component, column) line
// contiguously, line (c, t) at (c TC + t) NPL with the padded length NPL of
// col_line_len, so the transforms run exactly as in the row passes and the
// transposing accesses (consecutive threads on consecutive columns) fall on
// distinct banks.
// whether a pass has a second tile of three components
constexpr bool col_two(int mode) { return mode == COL_YMID_H || mode == COL_YINV_H; }

template <class T, int MODE>
__global__ void __launch_bounds__(kThreads, 2) k_col(ChainArgs<T> A, int axis, int TC, int ept) {
  using C = cx_t<T>;
  using W = T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int na = A.g.n[axis], La = A.g.log2n[axis];
  const long long npts = A.g.npts;
  const int Li = (axis == 1) ? A.g.log2n[0] : A.g.log2n[0] + A.g.log2n[1];   // log2 of the inner (faster) extent
  const int LT = __ffs(TC) - 1;
  const int Lt = Li - LT;                                        // log2 of the tiles per outer index
  const int bps = (int)(npts >> (La + LT));
  const int s = blockIdx.x / bps;
  const int tb = blockIdx.x - s * bps;
  C* s_tw = (C*)smem_raw;
  load_tw<T>(s_tw, A.tw[axis], na, ept);
  pdl_wait();
  if (s >= A.nsolve || !gate_ok(A.st, A.gate, s)) return;
  const int o = tb >> Lt;
  const int i0 = (tb - (o << Lt)) << LT;
  const int b0 = fft_padded_len<C>(na);   // the lines lie behind the table
  C* buf = s_tw + b0;
  const int NPL = col_line_len<C>(na, TC);        // padded line length
  const int CS = TC * NPL;                     // component stride in smem
  C* buf2 = buf + 3 * CS;            // second 3-component tile (YMID_H, YINV_H)
  double* red = (double*)(col_two(MODE) ? buf2 + 3 * CS : buf2);
  const SolveState& S = A.st[s];
  const PhysDev& ph = A.phys[s];
  const W piA = geo_piL<W>(A.g, axis);
  const int nx = A.g.n[0];
  // a thread stays on one column of the tile (the block is a multiple of TC threads): column t, from
  // row j0 in steps of dj; its first point, and element j of component c in shared memory
  const int t = threadIdx.x & (TC - 1), j0 = threadIdx.x >> LT, dj = blockDim.x >> LT;
  const long long col = (long long)s * 3 * npts + ((long long)o << (La + Li)) + i0 + t;
  const int lt = t * NPL;
  auto sidx = [&](int c, int j) { return c * CS + lt + fft_pad<C>(j); };

  // the in0 tile (and in1 for YINV_H) in natural order, by asynchronous copies
  for (int j = j0; j < na; j += dj) {
    const long long at = col + ((long long)j << Li);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      copy_async(&buf[sidx(c, j)], A.in0 + at + c * npts);
      if (MODE == COL_YINV_H) copy_async(&buf2[sidx(c, j)], A.in1 + at + c * npts);
    }
  }
  // wavenumbers of the column's inner index (the inputs are spectral along the faster axes)
  W kx, kyc;
  {
    const int ii = i0 + t;
    kx = wavenum<W>(ii & (nx - 1), nx, geo_piL<W>(A.g, 0));
    kyc = axis == 1 ? (W)0 : wavenum<W>(ii >> A.g.log2n[0], A.g.n[1], geo_piL<W>(A.g, 1));
  }
  const W k2c = (W)0.5 * (kx * kx + kyc * kyc);
  const W Om = pick<W>(ph.Omega, ph.fOmega), g = pick<W>(ph.gamma, ph.fgamma);
  const W al[3] = {pick<W>(S.alpha[0], S.falpha[0]), pick<W>(S.alpha[1], S.falpha[1]), pick<W>(S.alpha[2], S.falpha[2])};
  copy_wait();
  __syncthreads();

  constexpr int NK = sizeof(T) == 4 ? 9 : 3;
  W acc[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) acc[k] = (W)0;
  // one transform, or (the middle passes) a forward one, the work in k and the inverse one: a loop
  // around one inlined copy of the transforms.  The inverse transforms are forward ones whose values
  // are read at index -j
  constexpr bool middle = (MODE == COL_MID_H || MODE == COL_MID_PRE || MODE == COL_YMID_H || MODE == COL_YINV_H);
#pragma unroll 1
  for (int phase = 0; phase < (middle ? 2 : 1); ++phase) {
    if (MODE == COL_YINV_H && phase == 1) {
      // buf2: A -> F_y A, times v_y; then F_y^-1 of both: buf from C, buf2 -> G
      for (int j = j0; j < na; j += dj) {
        const W vy = wavenum<W>(j, na, piA);
#pragma unroll
        for (int c = 0; c < 3; ++c) buf2[sidx(c, j)] = cscale(buf2[sidx(c, j)], vy);
      }
      __syncthreads();
    } else if (phase == 1) {
      // pointwise in k: the kinetic + SOC symbol (H chains) or the kinetic preconditioner; with
      // YMID_H also G_c = F_y^-1[v_y F_y A_c] in buf2
      const bool use_pd = (A.sc.opts.precond == GPSOC_PRECOND_COMBINED || A.sc.opts.precond == GPSOC_PRECOND_KINETIC);
      const W gx = g * kx;
      // GPSOC_HYBRID P chain: buf holds the full spectrum of P.  Advance the stored spectrum of Phi by
      // the step applied this iteration (Phi_hat <- g (c Phi_hat + t P_hat_prev)), keep this P_hat, and
      // sum 1/2 |k|^2 |Phi_hat_l|^2 and 1/2 |k|^2 Re(Phi_hat_l conj P_hat_l)
      const bool hat = sizeof(T) == 4 && (MODE == COL_YMID_H || MODE == COL_MID_H) && A.xhat;
      const bool upd = hat && A.khat_upd && S.upd_applied;
      const W usc = pick<W>(S.upd_scale, S.fupd_scale);
      const W uc = usc * pick<W>(S.upd_c, S.fupd_c), us = usc * pick<W>(S.upd_s, S.fupd_s);
      for (int j = j0; j < na; j += dj) {
        const int i1 = sidx(0, j), i2 = sidx(1, j), i3 = sidx(2, j);
        const long long at = col + ((long long)j << Li);
        C xv[3], po[3];
        if (hat) {
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            xv[c] = A.xhat[at + c * npts];
            if (upd) po[c] = A.phat[at + c * npts];
          }
        }
        const W ka = wavenum<W>(j, na, piA);
        const W k2h = k2c + (W)0.5 * ka * ka;
        if (MODE == COL_MID_PRE) {
          // P_Delta (Eq. PreCondKin); the potential-only and no-preconditioner variants keep
          // the coefficients (the transform pair is then the identity up to rounding)
          if (use_pd) {
            // the three reciprocals from one division (an FP64 division is a long
            // instruction sequence): 1/d0 = d1 d2 / (d0 d1 d2), and so on
            const W d0 = al[0] + k2h, d1 = al[1] + k2h, d2 = al[2] + k2h;
            const W d01 = d0 * d1;
            const W inv = (W)1 / (d01 * d2);
            const W r01 = d2 * inv;
            buf[i1] = cscale(buf[i1], d1 * r01);
            buf[i2] = cscale(buf[i2], d0 * r01);
            buf[i3] = cscale(buf[i3], d01 * inv);
          }
        } else {
          const C p1 = buf[i1], p0 = buf[i2], pm = buf[i3];
          if (MODE == COL_YMID_H) {
            buf2[i1] = cscale(p1, ka);
            buf2[i2] = cscale(p0, ka);
            buf2[i3] = cscale(pm, ka);
          }
          if (hat) {
            const C pv[3] = {p1, p0, pm};
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              if (upd) {
                xv[c] = mk<C>(uc * xv[c].x + us * po[c].x, uc * xv[c].y + us * po[c].y);
                A.xhat[at + c * npts] = xv[c];
              }
              A.phat[at + c * npts] = pv[c];
              acc[3 + c] += k2h * (xv[c].x * xv[c].x + xv[c].y * xv[c].y);
              acc[6 + c] += k2h * (xv[c].x * pv[c].x + xv[c].y * pv[c].y);
            }
          }
          // kinetic per component (Parseval): sum 1/2 |k|^2 |phat_l|^2
          acc[0] += k2h * (p1.x * p1.x + p1.y * p1.y);
          acc[1] += k2h * (p0.x * p0.x + p0.y * p0.y);
          acc[2] += k2h * (pm.x * pm.x + pm.y * pm.y);
          // -gamma S symbol with -s0 = kx - i ky (L0), -s1 = kx + i ky (L1):
          // out_1 = K p1 - g s0 p0 ; out_0 = K p0 - g (s1 p1 + s0 pm) ; out_-1 = K pm - g s1 p0
          const W gy = g * (axis == 1 ? ka : kyc);
          const W sx = p1.x + pm.x, sy = p1.y + pm.y, dx = p1.x - pm.x, dy = p1.y - pm.y;
          buf[i1] = mk<C>(k2h * p1.x + (gx * p0.x + gy * p0.y), k2h * p1.y + (gx * p0.y - gy * p0.x));
          buf[i2] = mk<C>(k2h * p0.x + (gx * sx - gy * dy), k2h * p0.y + (gx * sy + gy * dx));
          buf[i3] = mk<C>(k2h * pm.x + (gx * p0.x - gy * p0.y), k2h * pm.y + (gx * p0.y + gy * p0.x));
        }
      }
      __syncthreads();
    }
    int first = b0, lines = 3 * TC;
    if (MODE == COL_YINV_H && phase == 0) first = b0 + 3 * CS;
    if ((MODE == COL_YINV_H || MODE == COL_YMID_H) && phase == 1) lines = 6 * TC;
    fft_lines<C, true>(first, lines, NPL, La, ept);
  }

  const W sc = (MODE == COL_INV) ? (W)A.scale : (W)1;
  // 2D: T' = F_y^-1[M F_y A] + ny Omega y v_x A; 3D: the factors of the axes transformed so far
  const W nz = (W)A.g.n[2];
  const W rx = (W)A.g.n[1] * (MODE == COL_YINV_H ? nz : (W)1) * Om * kx;
  for (int j = j0; j < na; j += dj) {
    const long long at = col + ((long long)j << Li);
    const int jr = (MODE == COL_FWD) ? j : (-j & (na - 1));
    if (MODE == COL_YMID_H || MODE == COL_YINV_H) {
      const W rot = rx * coord<W>(A.g, 1, j);
      C a[3];
#pragma unroll
      for (int c = 0; c < 3; ++c) a[c] = (MODE == COL_YINV_H ? A.in1 : A.in0)[at + c * npts];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const C v = buf[sidx(c, jr)], gv = buf2[sidx(c, jr)];
        A.out0[at + c * npts] = mk<C>(v.x + rot * a[c].x, v.y + rot * a[c].y);
        A.out1[at + c * npts] = (MODE == COL_YINV_H) ? mk<C>(gv.x * nz, gv.y * nz) : gv;
      }
    } else {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const C v = buf[sidx(c, jr)];
        A.out0[at + c * npts] = (MODE == COL_INV) ? mk<C>(v.x * sc, v.y * sc) : v;
      }
    }
  }
  if (MODE == COL_MID_H || MODE == COL_YMID_H) {
    const int slots[9] = {SL_KIN0, SL_KIN1, SL_KIN2, SL_KPHI0, SL_KPHI1, SL_KPHI2, SL_KX0, SL_KX1, SL_KX2};
    W aa[NK];
    int ss[NK];
    const bool mx[NK] = {};
#pragma unroll
    for (int k = 0; k < NK; ++k) { aa[k] = acc[k]; ss[k] = slots[k]; }
    store_partials<NK, W>(aa, ss, mx, red, A.part, (long long)s * NSLOT, A.pmax, tb, bps,
                          A.gcnt + (long long)s * A.gmax, (double*)smem_raw);
  }
}

// ============================================================== launch helpers
// Tile shapes: the largest tile (up to 512 elements per row tile, 1024 per
// column tile and component) that still gives the launch at least kTargetBlocks
// blocks over all solves, so small grids and single solves spread over the SMs
// while large batches keep long coalesced line segments.
//
// FP32 differs where its sweeps did: row tiles are worth halving only below 176 blocks (16 x 64^2 hybrid:
// 2 rows 1493 us, 4 rows 1410); column tiles keep 4 columns, the 32 bytes of a sector, however few
// blocks that leaves (one 512^2 solve, 1 column 1944 us, 4 columns 1650; 256^2 1611 and 1493; 3 x 128^2 1546 and
// 1389), and take 8 when 8 blocks per SM remain (64 x 256^2 24.7 ms and 23.4).
static constexpr int kTargetBlocks = 304;   // two blocks per SM of a 152-SM GB300
static constexpr int kTargetRows32 = 176;

// Tuned tiles (gpsoc_tuning_set / gpsoc_autotune) override the rule below for one
// grid, batch and precision; every launch and every block count of that key reads the
// same table entry, so the passes feeding one fused scalar step always agree.
namespace {
struct TileKey {
  int n0, n1, n2, nsolve, fp32;
  bool operator<(const TileKey& o) const {
    if (n0 != o.n0) return n0 < o.n0;
    if (n1 != o.n1) return n1 < o.n1;
    if (n2 != o.n2) return n2 < o.n2;
    if (nsolve != o.nsolve) return nsolve < o.nsolve;
    return fp32 < o.fp32;
  }
};
struct TileEntry { int lines[3] = {0, 0, 0}, ept[3] = {0, 0, 0}; };
std::map<TileKey, TileEntry> g_tiles;
std::mutex g_tiles_mu;

template <class T> TileKey tile_key(const Geo& g, int nsolve) {
  return TileKey{g.n[0], g.n[1], g.n[2], nsolve, sizeof(T) == 4 ? 1 : 0};
}
// tuned (lines, ept) of an axis, or (0, 0)
template <class T> void tuned(const Geo& g, int axis, int nsolve, int& lines, int& ept) {
  std::lock_guard<std::mutex> lk(g_tiles_mu);
  auto it = g_tiles.find(tile_key<T>(g, nsolve));
  lines = 0; ept = 0;
  if (it != g_tiles.end()) { lines = it->second.lines[axis]; ept = it->second.ept[axis]; }
}
}  // namespace

template <class T> bool tile_valid(const Geo& g, int axis, int lines, int ept);

// elements per thread of the FFT passes: 16 (radix-16 passes, FP32 column passes) or 8,
// unless the tile would then have fewer than 128 threads or a line is shorter,
// in which case fewer (more threads, more passes); and the matching thread
// count (multiple of 32, >= 64).  Rows: where the blocks fill the SMs, 8 (FP32: 16 x 64^2 hybrid
// 1493 us with 2, 1386 with 8) or at least 4 (FP64: 16 x 64^2 3118 us with 2, 3013 with 4) whatever the threads.
template <class T>
static int pick_ept(int work /* complex elements of the three components */, int n /* line length */, bool column,
                    long long blocks) {
  int e = (sizeof(T) == 4 && column) ? 16 : 8;
  const bool full = !column && blocks >= kTargetBlocks;
  const int least = full ? (sizeof(T) == 4 ? 8 : 4) : 2;
  while (e > 2 && ((work / e < 128 && e > least) || e > n)) e >>= 1;
  return e;
}

template <class T>
int row_rows_per_block(const Geo& g, int nsolve) {
  int tl, te;
  tuned<T>(g, 0, nsolve, tl, te);
  if (tl > 0) return tl;
  const int nx = g.n[0];
  const int rows = (int)(g.npts / nx);
  int R = 512 / nx;
  if (R < 1) R = 1;
  if (R > rows) R = rows;
  const int target = sizeof(T) == 4 ? kTargetRows32 : kTargetBlocks;
  while (R > 1 && (long long)nsolve * (rows / R) < target) R >>= 1;
  return R;
}

template <class T>
int col_tc(const Geo& g, int axis, int nsolve) {
  int tl, te;
  tuned<T>(g, axis, nsolve, tl, te);
  if (tl > 0) return tl;
  const int na = g.n[axis];
  const int ni = (axis == 1) ? g.n[0] : g.n[0] * g.n[1];
  const int no = (int)(g.npts / ((long long)na * ni));
  int tc = 1024 / na;
  if (tc < 1) tc = 1;
  if (tc > ni) tc = ni;
  const long long columns = (long long)nsolve * ni * no;
  while (tc > 1 && columns / tc < kTargetBlocks) tc >>= 1;
  if (sizeof(T) == 4) {
    if (tc < 4) tc = ni < 4 ? ni : 4;
    else if (2 * tc <= ni && 2 * tc * na <= 2048 && columns / (2 * tc) >= 4 * kTargetBlocks) tc *= 2;
  }
  // no more than the kernels run: 4 columns of 1024 points are 768 threads, as are 256 of 8 points (one 1024^2
  // hybrid iteration: 617 us with the 2 columns this leaves, 738 with 1)
  while (tc > 1 && !tile_valid<T>(g, axis, tc, pick_ept<T>(3 * tc * na, na, true, 0))) tc >>= 1;
  return tc;
}

static int round_threads(int t) {
  if (t < 64) t = 64;
  return (t + 31) & ~31;
}

template <class T>
static int row_ept(const Geo& g, int nsolve) {
  int tl, te;
  tuned<T>(g, 0, nsolve, tl, te);
  if (tl > 0 && te > 0) return te;
  const int R = row_rows_per_block<T>(g, nsolve);
  return pick_ept<T>(3 * R * g.n[0], g.n[0], false, (long long)nsolve * (g.npts / g.n[0]) / R);
}

template <class T>
static void col_cfg(const Geo& g, int axis, int nsolve, int& tc, int& ept, int& threads) {
  tc = col_tc<T>(g, axis, nsolve);
  const int work = 3 * tc * g.n[axis];
  int tl, te;
  tuned<T>(g, axis, nsolve, tl, te);
  ept = (tl > 0 && te > 0) ? te : pick_ept<T>(work, g.n[axis], true, 0);
  threads = round_threads(work / ept);
}

template <class T>
void tile_shape(const Geo& g, int axis, int nsolve, int& lines, int& ept, int& threads) {
  if (axis == 0) {
    lines = row_rows_per_block<T>(g, nsolve);
    ept = row_ept<T>(g, nsolve);
    threads = round_threads(3 * lines * g.n[0] / ept);
  } else {
    col_cfg<T>(g, axis, nsolve, lines, ept, threads);
  }
}

// A tile (lines, ept) for the passes along `axis` is valid when the FFT layout fits
// (ept a supported radix no longer than the line; every line of the tile has its
// threads), the block stays within the kernels' thread bound and the shared memory
// of its largest mode stays within the attribute chain_prepare sets.
template <class T>
bool tile_valid(const Geo& g, int axis, int lines, int ept) {
  using C = cx_t<T>;
  const int n = g.n[axis];
  if (lines < 1 || (lines & (lines - 1)) || n < 2) return false;
  const bool r16 = (sizeof(T) == 4 && axis > 0);
  if (!(ept == 2 || ept == 4 || ept == 8 || (ept == 16 && r16)) || ept > n) return false;
  const long long work = 3LL * lines * n;
  if (work / ept > kThreads) return false;
  size_t sm;
  if (axis == 0) {
    const int rows = (int)(g.npts / n);
    if (lines > rows) return false;
    sm = sizeof(C) * (fft_padded_len<C>(n) + 6 * (size_t)lines * fft_padded_len<C>(n)) + kRedDoubles * sizeof(double);
  } else {
    const int ni = (axis == 1) ? g.n[0] : g.n[0] * g.n[1];
    if (lines > ni) return false;
    sm = sizeof(C) * (fft_padded_len<C>(n) + 6 * (size_t)lines * col_line_len<C>(n, lines)) + kRedDoubles * sizeof(double);
  }
  return sm <= 200 * 1024;
}

// set (lines > 0) or clear (lines = 0) the tuned tile of one axis
template <class T>
bool tile_set(const Geo& g, int nsolve, int axis, int lines, int ept) {
  if (axis < 0 || axis >= g.d) return false;
  if (lines > 0 && !tile_valid<T>(g, axis, lines, ept)) return false;
  std::lock_guard<std::mutex> lk(g_tiles_mu);
  TileEntry& e = g_tiles[tile_key<T>(g, nsolve)];
  e.lines[axis] = lines > 0 ? lines : 0;
  e.ept[axis] = lines > 0 ? ept : 0;
  return true;
}

// every valid tile of an axis: powers of two for the lines, each supported radix
template <class T>
int tile_candidates(const Geo& g, int axis, int* lines, int* ept, int cap) {
  int k = 0;
  for (int l = 1; l <= 4096; l <<= 1)
    for (int e = 2; e <= 16; e <<= 1)
      if (tile_valid<T>(g, axis, l, e)) {
        if (k < cap) { lines[k] = l; ept[k] = e; }
        ++k;
      }
  return k;
}

template <class T>
int row_blocks_per_solve(const Geo& g, int nsolve) {
  return (int)(g.npts / g.n[0]) / row_rows_per_block<T>(g, nsolve);
}

template <class T>
int col_blocks_per_solve(const Geo& g, int axis, int nsolve) {
  const int na = g.n[axis];
  const int ni = (axis == 1) ? g.n[0] : g.n[0] * g.n[1];
  const int no = (int)(g.npts / ((long long)na * ni));
  return (ni / col_tc<T>(g, axis, nsolve)) * no;
}

template <class T>
static size_t row_smem(const Geo& g, int mode, int nsolve) {
  using C = cx_t<T>;
  const int R = row_rows_per_block<T>(g, nsolve);
  const bool two = (mode == ROW_INV_H || mode == ROW_INV_P || mode == ROW_INV_LIN || mode == ROW_INV_P_HY);
  const int CP = R * fft_padded_len<C>(g.n[0]);
  return sizeof(C) * (fft_padded_len<C>(g.n[0]) + 3 * CP * (two ? 2 : 1)) + kRedDoubles * sizeof(double);
}

template <class T>
static size_t col_smem(const Geo& g, int axis, int nsolve, int mode) {
  using C = cx_t<T>;
  const int tc = col_tc<T>(g, axis, nsolve);
  const int CS = col_line_len<C>(g.n[axis], tc) * tc;
  return sizeof(C) * (fft_padded_len<C>(g.n[axis]) + (col_two(mode) ? 6 : 3) * CS) + kRedDoubles * sizeof(double);
}

template <class T, int MODE>
static void row_go(const ChainArgs<T>& a, cudaStream_t st) {
  const int R = row_rows_per_block<T>(a.g, a.nsolve);
  const int nb = row_blocks_per_solve<T>(a.g, a.nsolve) * a.nsolve;
  const size_t sm = row_smem<T>(a.g, MODE, a.nsolve);
  const int ept = row_ept<T>(a.g, a.nsolve);
  const int threads = round_threads(3 * R * a.g.n[0] / ept);
  launch_pdl(k_row<T, MODE>, nb, threads, sm, st, a, R, ept);
}

template <class T>
void launch_row(int mode, const ChainArgs<T>& a, int, const Launch&, cudaStream_t st) {
  switch (mode) {
    case ROW_FWD_PLAIN: row_go<T, ROW_FWD_PLAIN>(a, st); break;
    case ROW_FWD_PROJ: row_go<T, ROW_FWD_PROJ>(a, st); break;
    case ROW_FWD_PRE: row_go<T, ROW_FWD_PRE>(a, st); break;
    case ROW_INV_H: row_go<T, ROW_INV_H>(a, st); break;
    case ROW_INV_P: row_go<T, ROW_INV_P>(a, st); break;
    case ROW_INV_PRE: row_go<T, ROW_INV_PRE>(a, st); break;
    case ROW_INV_PLAIN: row_go<T, ROW_INV_PLAIN>(a, st); break;
    case ROW_INV_LIN: row_go<T, ROW_INV_LIN>(a, st); break;
    case ROW_FWD_UPD: row_go<T, ROW_FWD_UPD>(a, st); break;
    case ROW_FWD_PRE_HY: if constexpr (sizeof(T) == 4) row_go<T, ROW_FWD_PRE_HY>(a, st); break;
    case ROW_INV_P_HY: if constexpr (sizeof(T) == 4) row_go<T, ROW_INV_P_HY>(a, st); break;
  }
}

template <class T, int MODE>
static void col_go(int axis, const ChainArgs<T>& a, cudaStream_t st) {
  int tc, ept, threads;
  col_cfg<T>(a.g, axis, a.nsolve, tc, ept, threads);
  const int nb = col_blocks_per_solve<T>(a.g, axis, a.nsolve) * a.nsolve;
  const size_t sm = col_smem<T>(a.g, axis, a.nsolve, MODE);
  launch_pdl(k_col<T, MODE>, nb, threads, sm, st, a, axis, tc, ept);
}

template <class T>
void launch_col(int mode, int axis, const ChainArgs<T>& a, const Launch&, cudaStream_t st) {
  switch (mode) {
    case COL_FWD: col_go<T, COL_FWD>(axis, a, st); break;
    case COL_INV: col_go<T, COL_INV>(axis, a, st); break;
    case COL_MID_H: col_go<T, COL_MID_H>(axis, a, st); break;
    case COL_MID_PRE: col_go<T, COL_MID_PRE>(axis, a, st); break;
    case COL_YMID_H: col_go<T, COL_YMID_H>(axis, a, st); break;
    case COL_YINV_H: col_go<T, COL_YINV_H>(axis, a, st); break;
  }
}

template <class T>
cudaError_t chain_prepare() {
  const int big = 200 * 1024;
  cudaError_t e = cudaSuccess;
#define GPSOC_ATTR(K) \
  if (e == cudaSuccess) e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, big);
  GPSOC_ATTR((k_row<T, ROW_FWD_PLAIN>)) GPSOC_ATTR((k_row<T, ROW_FWD_PROJ>)) GPSOC_ATTR((k_row<T, ROW_FWD_PRE>))
  GPSOC_ATTR((k_row<T, ROW_INV_H>)) GPSOC_ATTR((k_row<T, ROW_INV_P>)) GPSOC_ATTR((k_row<T, ROW_INV_PRE>))
  GPSOC_ATTR((k_row<T, ROW_INV_PLAIN>)) GPSOC_ATTR((k_row<T, ROW_INV_LIN>)) GPSOC_ATTR((k_row<T, ROW_FWD_UPD>))
  GPSOC_ATTR((k_col<T, COL_FWD>)) GPSOC_ATTR((k_col<T, COL_INV>)) GPSOC_ATTR((k_col<T, COL_MID_H>))
  GPSOC_ATTR((k_col<T, COL_MID_PRE>)) GPSOC_ATTR((k_col<T, COL_YMID_H>)) GPSOC_ATTR((k_col<T, COL_YINV_H>))
  if constexpr (sizeof(T) == 4) {
    GPSOC_ATTR((k_row<T, ROW_FWD_PRE_HY>)) GPSOC_ATTR((k_row<T, ROW_INV_P_HY>))
  }
#undef GPSOC_ATTR
  return e;
}

template void launch_row<double>(int, const ChainArgs<double>&, int, const Launch&, cudaStream_t);
template void launch_row<float>(int, const ChainArgs<float>&, int, const Launch&, cudaStream_t);
template void launch_col<double>(int, int, const ChainArgs<double>&, const Launch&, cudaStream_t);
template void launch_col<float>(int, int, const ChainArgs<float>&, const Launch&, cudaStream_t);
template bool tile_set<double>(const Geo&, int, int, int, int);
template bool tile_set<float>(const Geo&, int, int, int, int);
template int tile_candidates<double>(const Geo&, int, int*, int*, int);
template int tile_candidates<float>(const Geo&, int, int*, int*, int);
template void tile_shape<double>(const Geo&, int, int, int&, int&, int&);
template void tile_shape<float>(const Geo&, int, int, int&, int&, int&);
template int row_blocks_per_solve<double>(const Geo&, int);
template int row_blocks_per_solve<float>(const Geo&, int);
template int col_blocks_per_solve<double>(const Geo&, int, int);
template int col_blocks_per_solve<float>(const Geo&, int, int);
template cudaError_t chain_prepare<double>();
template cudaError_t chain_prepare<float>();

}  // namespace gpsoc
