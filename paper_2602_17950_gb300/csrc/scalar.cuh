// Scalar steps of the PCG iteration (Section 3.1, Algorithms 1 and 2), run by one
// thread block per solve: either by a separate kernel or fused into the last
// block of the array pass that produced their sums.  Every thread of the block
// calls the function (grid sums); its first warp then does the step and updates
// the solve's state.  Sums of block partials are taken in a fixed order (deterministic).
//
// One SM runs such a step while the others wait, and an FP64 warp instruction holds its
// sub-partition for 64 cycles, for one lane as for 32.  So every lane of the warp computes the
// step's common chain, values that come in threes or tens (alpha, masses, FP32 copies) take a
// lane each, the density and the spin integrals are combined before they are transformed, and
// divisions, roots, sines and finiteness tests are avoided where something shorter is as exact:
// the Algorithm 2 step went from about 330 FP64 instructions to 120.  With the four steps of an iteration
// written this way, an iteration of one 64^2 FP64 solve went from 126 to 116.5 us, of one 128^2 hybrid
// solve from 94 to 85 us.
#pragma once

#include "gpsoc_internal.cuh"

namespace gpsoc {

// ------------------------------------------------------------------ grid sums
// Totals of K <= 32 slots over the block partials of solve s into scratch[k], and the maximum of the
// slot `max_slot` (if >= 0; its values are not negative) into scratch[32].  Slots k < K0 and the
// maximum have nb0 partials, the other slots nb1.  Every thread of the block calls it; the results are
// for warp 0, which runs the scalar step alone.
//
// All the partials of a thread are loaded together (one memory round trip), added in the order
// of the blocks, then a warp adds by reduce-scatter -- at each halving step a lane keeps one half
// of its slots and adds the partner lane's copy of that half, KP - 1 sums for KP slots
// instead of 5 K -- and the warps' sums are added in the order of the warps: a fixed order.
// V = DF: double-word partials, added as double words on the FP32 pipes, the totals rounded to FP64
// once; V = double: FP64 partials, added in FP64.
// scratch: 32 * (blockDim.x / 32) + 1 doubles.
template <class V> struct TotOps;
template <> struct TotOps<double> {
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double load(const double* p) { return __ldcg(p); }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
  static __device__ __forceinline__ double from(double a) { return a; }
  static __device__ __forceinline__ double pack(double a) { return a; }
  static __device__ __forceinline__ double value(double a) { return a; }
};
template <> struct TotOps<DF> {
  static __device__ __forceinline__ DF zero() { return DF{0.0f, 0.0f}; }
  static __device__ __forceinline__ DF load(const double* p) { return get_sum_partial(p); }
  static __device__ __forceinline__ DF add(DF a, DF b) { return dw_add(a, b); }
  static __device__ __forceinline__ DF shfl(DF a, int o) { return df_shfl_xor(a, o); }
  static __device__ __forceinline__ DF from(double a) {
    const float2 f = *reinterpret_cast<const float2*>(&a);
    return DF{f.x, f.y};
  }
  static __device__ __forceinline__ double pack(DF a) {
    const float2 f = make_float2(a.hi, a.lo);
    return *reinterpret_cast<const double*>(&f);
  }
  static __device__ __forceinline__ double value(DF a) { return (double)a.hi + (double)a.lo; }
};
// A pass of more than kGroupFrom blocks per solve leaves one partial per group of kGroup blocks, at the
// place of the group's first (group_sums): the scalar step of a 128^3 pass would otherwise read thousands,
// 20 round trips to memory on one SM while the others wait (65 us of a 176 us row_inv_p_hy).
constexpr int kGroup = 64, kGroupFrom = 1024;
__host__ __device__ __forceinline__ int part_groups(int nb) { return (nb + kGroup - 1) / kGroup; }
__device__ __forceinline__ int part_stride(int nb) { return nb > kGroupFrom ? kGroup : 1; }
__device__ __forceinline__ int part_entries(int nb) { return nb > kGroupFrom ? part_groups(nb) : nb; }

// sums of one warp's share: n0 entries (slots k < K0) or n1 from `base` on, st0 or st1 apart, dealt to the
// threads tid < nt; the warp's sums go to scratch[warp * 32 + k]
template <class V, int K, int K0>
__device__ __forceinline__ void totals_of(const double* base, int pmax, const int (&slots)[K], int n0, int st0, int n1,
                                          int st1, int nt, double* scratch) {
  using O = TotOps<V>;
  constexpr int KP = (K <= 4) ? 4 : (K <= 8) ? 8 : (K <= 16) ? 16 : 32;
  constexpr int LB = (KP == 4) ? 2 : (KP == 8) ? 3 : (KP == 16) ? 4 : 5;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  V x[KP];
  const double* p0 = base + (int)threadIdx.x * st0;
  const double* p1 = base + (int)threadIdx.x * st1;
#pragma unroll
  for (int k = 0; k < KP; ++k)
    x[k] = (k < K && (int)threadIdx.x < (k < K0 ? n0 : n1))
               ? O::load((k < K0 ? p0 : p1) + (long long)slots[k < K ? k : 0] * pmax) : O::zero();
  for (int b = threadIdx.x + nt; b < max(n0, n1); b += nt) {
    V t[K];
    p0 += nt * st0;
    p1 += nt * st1;
#pragma unroll
    for (int k = 0; k < K; ++k) t[k] = b < (k < K0 ? n0 : n1) ? O::load((k < K0 ? p0 : p1) + (long long)slots[k] * pmax) : O::zero();
#pragma unroll
    for (int k = 0; k < K; ++k) x[k] = O::add(x[k], t[k]);
  }
#pragma unroll
  for (int st = 0; st < LB; ++st) {
    const int ofs = 1 << st, half = (KP / 2) >> st;
    const bool up = (lane & ofs) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const V keep = up ? x[i + half] : x[i];
      const V send = up ? x[i] : x[i + half];
      x[i] = O::add(keep, O::shfl(send, ofs));
    }
  }
#pragma unroll
  for (int ofs = KP; ofs < 32; ofs <<= 1) x[0] = O::add(x[0], O::shfl(x[0], ofs));
  int slot = 0;   // a lane's slot: its low LB bits reversed (bit 0 chose between the halves first)
#pragma unroll
  for (int b = 0; b < LB; ++b) slot |= ((lane >> b) & 1) << (LB - 1 - b);
  if (lane < KP) scratch[warp * 32 + slot] = O::pack(x[0]);
}
// PLAIN: partials of an elementwise pass, which are not grouped
template <class V, int K, int K0, bool PLAIN = false>
__device__ __forceinline__ void slot_totals(const ScalarCtx& X, int s, const int (&slots)[K], int nb0, int nb1,
                                            int max_slot, double* scratch) {
  __shared__ unsigned long long s_max[32];
  const int nw = (blockDim.x + 31) >> 5;
  const double* base = X.part + (long long)s * NSLOT * X.pmax;
  const int n0 = PLAIN ? nb0 : part_entries(nb0), st0 = PLAIN ? 1 : part_stride(nb0);
  totals_of<V, K, K0>(base, X.pmax, slots, n0, st0, part_entries(nb1), part_stride(nb1), blockDim.x, scratch);
  if (max_slot >= 0) {
    unsigned long long m = 0;   // values that are not negative (or NaN) are ordered as their bits
    const double* p = base + (long long)max_slot * X.pmax;
    for (int b = threadIdx.x; b < n0; b += blockDim.x) {
      const unsigned long long v = (unsigned long long)__double_as_longlong(__ldcg(p + (long long)b * st0));
      m = v > m ? v : m;
    }
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const int k = threadIdx.x;
    V a = TotOps<V>::from(scratch[k]);
    for (int w = 1; w < nw; ++w) a = TotOps<V>::add(a, TotOps<V>::from(scratch[w * 32 + k]));
    __syncwarp();
    scratch[k] = TotOps<V>::value(a);
    if (max_slot >= 0) {
      const unsigned long long m = warp_max(k < nw ? s_max[k] : 0ull);
      if (k == 0) scratch[32] = __longlong_as_double((long long)m);
    }
    __syncwarp();
  }
}

// The partials of block blk's group into one, by the last of its blocks to arrive: K sums (slots) and, if
// max_slot >= 0, a maximum.  Every thread of every block calls it, once in a kernel (the counters know one
// arrival per block), when the block's own partials are written; gcnt: the solve's group counters (zero;
// they are left zero); scratch: 66 doubles.  Out of line: inlined it cost the passes that have no groups 2-3%.
template <class V, int K>
__device__ __noinline__ void group_sums_of(double* base, int pmax, const int* slots, int max_slot, int blk, int nb,
                                           unsigned* gcnt, double* scratch) {
  __shared__ int s_last;
  const int g = blk / kGroup, n = min(kGroup, nb - g * kGroup);
  if (!last_block(gcnt, g, n, &s_last)) return;
  double* p = base + g * kGroup;
  const int t = threadIdx.x;
  if (max_slot >= 0 && t < kGroup) {
    const unsigned long long m =
        warp_max(t < n ? (unsigned long long)__double_as_longlong(__ldcg(p + (long long)max_slot * pmax + t)) : 0ull);
    if ((t & 31) == 0) scratch[64 + (t >> 5)] = __longlong_as_double((long long)m);
  }
  // slot after slot (few registers): a warp adds 32 partials of a slot at a time
  using O = TotOps<V>;
  for (int k = t >> 5; k < 2 * K; k += blockDim.x >> 5) {
    const int b = (k & 1) * 32 + (t & 31);
    V x = b < n ? O::load(p + (long long)slots[k >> 1] * pmax + b) : O::zero();
    for (int ofs = 16; ofs > 0; ofs >>= 1) x = O::add(x, O::shfl(x, ofs));
    if ((t & 31) == 0) scratch[k] = O::pack(x);
  }
  __syncthreads();
  if (t < K) p[(long long)slots[t] * pmax] = O::pack(O::add(O::from(scratch[2 * t]), O::from(scratch[2 * t + 1])));
  if (max_slot >= 0 && t == 0) {
    // as bits: a NaN stays the maximum
    const long long m0 = __double_as_longlong(scratch[64]), m1 = __double_as_longlong(scratch[65]);
    p[(long long)max_slot * pmax] = __longlong_as_double(m0 > m1 ? m0 : m1);
  }
}
template <class V, int K>
__device__ __forceinline__ void group_sums(double* base, int pmax, const int (&slots)[K], int blk, int nb, unsigned* gcnt,
                                           double* scratch, int max_slot = -1) {
  if (nb > kGroupFrom) group_sums_of<V, K>(base, pmax, slots, max_slot, blk, nb, gcnt, scratch);
}
template <class V>
__device__ __forceinline__ void group_max(double* base, int pmax, int max_slot, int blk, int nb, unsigned* gcnt,
                                          double* scratch) {
  if (nb > kGroupFrom) group_sums_of<V, 0>(base, pmax, nullptr, max_slot, blk, nb, gcnt, scratch);
}

__device__ __forceinline__ void deactivate(SolveState& S, int status) {
  S.active = 0;
  if (S.status == GPSOC_OK) S.status = status;
}

// The solve state of a step is copied to shared memory by the block (one round of loads, before the
// grid sums), updated there by the first warp, and copied back by it.
__device__ __forceinline__ void state_load(SolveState& dst, const SolveState* src) {
  static_assert(sizeof(SolveState) % 8 == 0, "state is copied in 8-byte words");
  auto* d = reinterpret_cast<unsigned long long*>(&dst);
  const auto* q = reinterpret_cast<const unsigned long long*>(src);
  for (int i = threadIdx.x; i < (int)(sizeof(SolveState) / 8); i += blockDim.x) d[i] = __ldcg(q + i);
}
__device__ __forceinline__ void state_store_warp(SolveState* dst, const SolveState& src) {
  __syncwarp();
  auto* d = reinterpret_cast<unsigned long long*>(dst);
  const auto* q = reinterpret_cast<const unsigned long long*>(&src);
  for (int i = threadIdx.x; i < (int)(sizeof(SolveState) / 8); i += 32) d[i] = q[i];
}
// the FP32 copies, a lane each
__device__ __forceinline__ void mirror32_warp(SolveState& S) {
  __syncwarp();
  const int l = threadIdx.x;
  if (l < 9) {
    const double* src = l == 0 ? &S.mu : l == 1 ? &S.beta : l == 2 ? &S.cproj : l == 3 ? &S.upd_c : l == 4 ? &S.upd_s
                      : l == 5 ? &S.upd_scale : &S.alpha[l - 6];
    (&S.fmu)[l] = (float)*src;   // fmu, fbeta, fcproj, fupd_c, fupd_s, fupd_scale, falpha[3]
  }
  __syncwarp();
}
// sign and finiteness from the bits (an FP64 comparison holds the FP64 pipe like an addition)
__device__ __forceinline__ bool fin(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool pos(double x) { return __double_as_longlong(x) > 0; }            // x > 0, x not NaN
__device__ __forceinline__ bool zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ bool neg(double x) { return __double_as_longlong(x) < 0 && !zero(x); }   // x < 0, x not NaN

// E, mu (Eqs. energy, muphi), alpha_l (Eq. PreCnstAlpha), masses of the current iterate
template <class V>
__device__ __forceinline__ void sc_obs(const ScalarCtx& X, int s, double* scratch) {
  __shared__ SolveState sS;
  state_load(sS, X.st + s);      // visible after the barrier of the grid sums
  const PhysDev ph = X.phys[s];
  const int slots[15] = {SL_Q, SL_RHO2, SL_F2, SL_V0, SL_V1, SL_V2, SL_C0, SL_C1, SL_C2, SL_M0, SL_M1, SL_M2,
                         SL_KIN0, SL_KIN1, SL_KIN2};
  // GPSOC_HYBRID: the kinetic part of alpha_l is in the state (an exact FP64 recomputation of H_lin Phi,
  // advanced with the steps); the slots hold sums of another pass
  const bool hy = (X.flags & 8) != 0;
  slot_totals<V, 15, 12>(X, s, slots, X.nb_row, hy ? 0 : X.nb_col, SL_DPHIINF, scratch);
  if (threadIdx.x >= 32) return;
  const int l = threadIdx.x;
  const double dV = X.dV, *v = scratch;
  const double Q = dV * v[0], rho2 = dV * v[1], F2 = dV * v[2];
  const double I = ph.c0 * rho2, J = ph.c1 * F2;
  const double mu = Q + I + J, E = Q + 0.5 * (I + J);
  // lanes 0-2: alpha_l and the mass of their component
  const int c = l < 3 ? l : 0;
  double al = dV * ((hy ? sS.kin[c] : v[12 + c]) * X.inv_npts + v[3 + c] + ph.c0 * v[6 + c]);
  const double m = dV * v[9 + c];
  const double a0 = __shfl_sync(0xffffffffu, al, 0), a1 = __shfl_sync(0xffffffffu, al, 1), a2 = __shfl_sync(0xffffffffu, al, 2);
  const bool ok = fin(E) && fin(mu) && fin(a0) && fin(a1) && fin(a2);
  al = fmax(al, 1e-12 * fmax(fabs(a0), fmax(fabs(a1), fabs(a2))) + 1e-300);
  const bool had_step = sS.pending != 0;
  __syncwarp();
  if (l < 3) {
    sS.alpha[c] = al;
    sS.mass[c] = m;
  }
  if (l == 0) {
    sS.Q = Q;
    sS.rho2 = rho2;
    sS.F2 = F2;
    sS.E = E;
    sS.mu = mu;
    // max |dPhi| is read by the stop1 test only
    if (had_step && X.opts.stop == GPSOC_STOP_DPHI) sS.dphi_inf = sqrt(v[32]);
    sS.upd_applied = had_step ? 1 : 0;
    sS.pending = 0;
    if (!ok) deactivate(sS, GPSOC_ENONFINITE);
  }
  mirror32_warp(sS);
  state_store_warp(X.st + s, sS);
}

constexpr int kStallWindow = 256;

// max_l ||r_l||_inf and the stopping test (Eqs. stop1-stop3); the partials hold max |r|^2
__device__ __forceinline__ void sc_res(const ScalarCtx& X, int s, double* scratch) {
  SolveState& S = X.st[s];
  unsigned long long m = 0;
  const double* p = X.part + ((long long)s * NSLOT + SL_RINF) * X.pmax;
  const int n = part_entries(X.nb_row), st = part_stride(X.nb_row);
  for (int b = threadIdx.x; b < n; b += blockDim.x) {
    const unsigned long long v = (unsigned long long)__double_as_longlong(__ldcg(p + (long long)b * st));
    m = v > m ? v : m;
  }
  m = warp_max(m);
  auto* sm = reinterpret_cast<unsigned long long*>(scratch);
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  m = warp_max(threadIdx.x < (blockDim.x >> 5) ? sm[threadIdx.x] : 0ull);
  if (threadIdx.x != 0) return;
  const double rinf = sqrt(__longlong_as_double((long long)m));
  const OptsDev& O = X.opts;
  S.res_inf = rinf;
  if (!fin(rinf)) { deactivate(S, GPSOC_ENONFINITE); return; }
  if (O.no_stop) return;
  // FP32 phase: once the residual is this small the FP32 rounding floor is near, so
  // the level continues in FP64 (also at iteration 0: a level that starts converged
  // takes no FP32 step)
  if (O.phase32 && O.res32 > 0.0 && rinf < O.res32) { S.active = 0; return; }
  if (S.iters >= 1 || O.stop == GPSOC_STOP_RES) {
    bool conv;
    if (O.stop == GPSOC_STOP_ENERGY) conv = fabs(S.dE_last) < O.tol + O.tol_rel * fabs(S.E);
    else if (O.stop == GPSOC_STOP_RES) conv = rinf < O.tol;
    else conv = S.dphi_inf < O.tol;
    if (conv && O.res_tol > 0.0) conv = rinf < O.res_tol;
    if (conv) { S.active = 0; return; }
  }
  // FP32 phase: per-iteration energy changes carry rounding noise that can stay
  // above tol_rel |E| for ever; hand over to FP64 once the energy fell by less
  // than tol_rel |E| per iteration on average over a window of kStallWindow.
  if (O.phase32 && S.iters - S.it_win >= kStallWindow) {
    if (!(S.E_win - S.E >= kStallWindow * O.tol_rel * fabs(S.E))) { S.active = 0; return; }
    S.E_win = S.E;
    S.it_win = S.iters;
  }
  if (S.iters >= O.max_iter) {
    if (O.phase32) S.active = 0;
    else deactivate(S, GPSOC_ENOTCONV);
  }
}

// Polak-Ribiere+ beta = max(Re<r - r_prev, P r> / Re<r_prev, P_prev r_prev>, 0), the
// tangent projection coefficient c = Re<D, Phi> of D = -P r + beta P_prev (Eq. formula-
// project) and Algorithm 2 Step 2, all from the sums of the preconditioner's last pass:
// D is linear in beta, so Re<D, Phi> = -Re<z, Phi> + beta Re<P_prev, Phi> and the slope
// Re<r, D> = -Re<r, z> + beta Re<r, P_prev> (b_n has its sign: Re<H Phi, P> = Re<r, D>
// for the tangent P).  If the slope is not negative the step restarts from D = -P r.
template <class V>
__device__ __forceinline__ void sc_beta(const ScalarCtx& X, int s, double* scratch) {
  SolveState& S = X.st[s];
  const bool first = S.first != 0;          // read ahead of the sums
  const double s_prev = S.s_prev;
  const int slots[5] = {SL_RZ, SL_RPZ, SL_ZPHI, SL_PPHI, SL_RP};
  slot_totals<V, 5, 5>(X, s, slots, X.nb_row, 0, -1, scratch);
  if (threadIdx.x != 0) return;
  const double dV = X.dV, *w = scratch;
  const double rz = dV * w[0], zphi = dV * w[2];
  S.s_cur = rz;
  double beta = 0.0;
  if (!first) {
    beta = (rz - dV * w[1]) / s_prev;
    if (!(beta > 0.0)) beta = 0.0;   // max(beta, 0), NaN -> 0
  }
  double cD = -zphi + beta * dV * w[3];
  if (beta != 0.0 && !(-rz + beta * dV * w[4] < 0.0)) {
    beta = 0.0;
    S.beta_resets++;
    cD = -zphi;
  }
  S.beta = beta;
  S.cproj = cD;
  S.fbeta = (float)beta;
  S.fcproj = (float)cD;
}

// E(cos t Phi + sin t P/||P||) - E(Phi) from the reduced integrals (unnormalised P),
// given sn = sin t, cs = cos t: quadratic part -s^2 Q + 2cs/|P| Re<H_lin Phi,P> +
// s^2/|P|^2 <H_lin P,P>, interaction part from rho_t - rho = u rho_Phi + w1 R + w2 rho_P
// (u = -s^2, w1 = 2cs/|P|, w2 = s^2/|P|^2) and the same for the spin density
// (Section 3.1, the explicit form of E(theta)).  K[k] = c0 I[k] + c1 J[k] combines the six
// integrals of the density and of the spin density.
__device__ __forceinline__ double energy_change_sc(const SolveState& S, double sn, double cs, double inv_nP) {
  const double* K = S.K;
  const double sp = sn * inv_nP;
  const double u = -sn * sn, w1 = 2.0 * cs * sp, w2 = sp * sp;
  const double Au = 0.5 * (u * K[0]) + (w1 * K[1] + w2 * K[2]) + (S.Q + K[0]);
  const double A1 = 0.5 * (w1 * K[3]) + w2 * K[4] + S.HPhiP;
  const double A2 = 0.5 * (w2 * K[5]) + (S.HPP + K[2]);
  return u * Au + w1 * A1 + w2 * A2;
}

__device__ __forceinline__ double energy_change(const SolveState& S, double theta) {
  double sn, cs;
  sincos(theta, &sn, &cs);
  return energy_change_sc(S, sn, cs, rsqrt(S.P2));
}

// sine and cosine of the step's angle, by a whole warp: their Taylor sums on the odd and the even lanes,
// 12 FP64 instructions instead of the library's 27; larger angles (and negative ones, NaN) by the library
__device__ __forceinline__ void sincos_warp(double x, double& sn, double& cs) {
  if (!taylor_in_range(x)) {
    sincos(x, &sn, &cs);
    return;
  }
  const double r = taylor_sincos(x, threadIdx.x & 1);
  cs = __shfl_sync(0xffffffffu, r, 0);
  sn = __shfl_sync(0xffffffffu, r, 1);
}

// Eq. theta: theta_n = argmin_{theta > 0} E(cos t Phi + sin t P/|P|), on the explicit
// sin/cos form of the energy change.  With u = -s^2, v = 2cs/|P|, w = s^2/|P|^2 the change
// is a quadratic polynomial in (u, v, w) (energy_change_sc); its t-derivative follows with
// du/dt = -sin 2t, dv/dt = 2 cos 2t/|P|, dw/dt = sin 2t/|P|^2.  The minimiser taken is the
// first zero of the derivative found by doubling from the quadratic model's t0 (E has
// period pi and decreases at 0+), solved by Newton steps kept inside the bracket
// (bisection when a step leaves it).  If no sign change is met up to pi, t0 is kept.
struct TrigForm {
  double lu, l1, l2;                 // linear coefficients of u, v, w
  double huu, hu1, hu2, h11, h12, h22;   // second derivatives of the change in (u, v, w)
  double inv_nP, inv_nP2;
  // derivative (g1) and second derivative (g2) of the energy change at t
  __device__ __forceinline__ void eval(double t, double& g1, double& g2) const {
    double s2, c2;
    sincos(2.0 * t, &s2, &c2);
    const double u = -0.5 * (1.0 - c2), v = s2 * inv_nP, w = 0.5 * (1.0 - c2) * inv_nP2;
    const double du = -s2, dv = 2.0 * c2 * inv_nP, dw = s2 * inv_nP2;
    const double ddu = -2.0 * c2, ddv = -4.0 * s2 * inv_nP, ddw = 2.0 * c2 * inv_nP2;
    const double Au = lu + huu * u + hu1 * v + hu2 * w;
    const double A1 = l1 + hu1 * u + h11 * v + h12 * w;
    const double A2 = l2 + hu2 * u + h12 * v + h22 * w;
    g1 = Au * du + A1 * dv + A2 * dw;
    g2 = Au * ddu + A1 * ddv + A2 * ddw + huu * du * du + h11 * dv * dv + h22 * dw * dw +
         2.0 * (hu1 * du * dv + hu2 * du * dw + h12 * dv * dw);
  }
};

__device__ __forceinline__ double exact_theta(const SolveState& S, double inv_nP, double t0) {
  TrigForm f;
  const double* K = S.K;
  f.lu = S.Q + K[0];
  f.l1 = S.HPhiP;
  f.l2 = S.HPP + K[2];
  f.huu = K[0]; f.hu1 = K[1]; f.hu2 = K[2];
  f.h11 = K[3]; f.h12 = K[4]; f.h22 = K[5];
  f.inv_nP = inv_nP; f.inv_nP2 = inv_nP * inv_nP;
  const double PI = 3.14159265358979323846;
  double lo = 0.0, hi = fmin(t0, PI), g1, g2;
  f.eval(hi, g1, g2);
  while (g1 < 0.0 && hi < PI) {
    lo = hi;
    hi = fmin(2.0 * hi, PI);
    f.eval(hi, g1, g2);
  }
  if (g1 < 0.0) return t0;
  double t = hi;   // Newton from the right end of the bracket
  for (int it = 0; it < 100; ++it) {
    f.eval(t, g1, g2);
    if (g1 == 0.0) break;
    if (g1 < 0.0) lo = t; else hi = t;
    double tn = (g2 > 0.0) ? t - g1 / g2 : 0.5 * (lo + hi);
    if (!(tn > lo && tn < hi)) tn = 0.5 * (lo + hi);
    if (fabs(tn - t) <= 1e-15 * t || hi - lo <= 2e-16 * hi) { t = tn; break; }
    t = tn;
  }
  return t;
}

// The step-model sums of the P chain (warp 0, from the totals v in the order of kStepSlots) into S, and
// a_n, b_n of Eqs. an, bn; returns 1/|P|
__device__ __forceinline__ double step_sums(const ScalarCtx& X, int s, const double* v, SolveState& S) {
  const PhysDev ph = X.phys[s];
  const double dV = X.dV;
  // the combined integrals c0 I + c1 J, a lane each: lanes 1-5; lanes 8-11 scale P2, HPP, HPHIP, RPHI
  const int l = threadIdx.x & 31;
  const int at = (l >= 1 && l <= 5) ? 3 + l : (l >= 8 && l <= 11) ? l - 8 : 0;
  const double i_l = dV * v[at];
  const double j_l = dV * v[(l >= 1 && l <= 5) ? 8 + l : 0];
  const double k_l = ph.c0 * (l == 0 ? S.rho2 : i_l) + ph.c1 * (l == 0 ? S.F2 : j_l);
  auto lane = [](double x, int k) { return __shfl_sync(0xffffffffu, x, k); };
  const double K0 = lane(k_l, 0), K1 = lane(k_l, 1), K2 = lane(k_l, 2), K3 = lane(k_l, 3), K4 = lane(k_l, 4), K5 = lane(k_l, 5);
  const double P2 = lane(i_l, 8), HPP = lane(i_l, 9), X1 = lane(i_l, 10), RPhi = lane(i_l, 11);
  const double M = S.mass[0] + S.mass[1] + S.mass[2], Q = S.Q, mu = S.mu;
  // Re<H_lin Phi, P>: from Re<H Phi, P>, or in GPSOC_HYBRID from Re<r, P> + mu Re<P, Phi>
  const double QFP = ((X.flags & 8) ? X1 + mu * RPhi : X1) - K1;
  // Exact tangent correction: the step is taken along P_t = P - a Phi, a = Re<P, Phi>/||Phi||^2,
  // which is tangent to the sphere whatever the rounding of P (an FP32 direction carries a
  // radial part of relative size 1e-7).  Every sum transforms exactly: R -> R - a rho_Phi,
  // rho_P -> rho_P - 2a R + a^2 rho_Phi, and the same for the spin vectors.
  const double a = divide_near_one(RPhi, M);   // ||Phi||^2 is 1 up to rounding
  const double Z1 = K1 - a * K0, Z2 = K2 - a * (K1 + Z1);
  const double q = K3 - a * K1, Z3 = q - a * Z1;
  const double w = K4 - a * (K3 + q), Z4 = w - a * Z2;
  const double Z5 = K5 - a * (2.0 * (K4 + w) - a * (K2 + Z2));
  const double tHPP = HPP - a * (2.0 * QFP - a * Q), tP2 = P2 - a * RPhi;
  const double HPhiP = (QFP - a * Q) + Z1;
  const double inv = rsqrt(tP2);
  // density frozen at Phi^n in H_l(P^n)
  const double an = (tHPP + Z2 + 2.0 * Z3) * (inv * inv) - mu;
  const double bn = 2.0 * HPhiP * inv;
  __syncwarp();
  if (l == 0) {
    S.acorr = a;
    S.P2 = tP2;
    S.HPP = tHPP;
    S.HPhiP = HPhiP;
    S.K[0] = K0; S.K[1] = Z1; S.K[2] = Z2; S.K[3] = Z3; S.K[4] = Z4; S.K[5] = Z5;
    S.a = an;
    S.b = bn;
  }
  __syncwarp();
  return inv;
}
constexpr int kStepSlots = 14;
#define GPSOC_STEP_SLOTS SL_P2, SL_HPP, SL_HPHIP, SL_RPHI, SL_IFR, SL_IFP, SL_IRR, SL_IRP, SL_IPP, \
                         SL_JFR, SL_JFP, SL_JRR, SL_JRP, SL_JPP

// Algorithm 2: step size from the quadratic model, backtracking on the exact
// energy change, update coefficients of Eqs. formula-pcg / update (applied by
// the next iteration's first pass).  The whole warp, on the copy S of the state; every lane
// computes the same values, lane 0 stores them.
__device__ __forceinline__ void step_decide(const ScalarCtx& X, SolveState& S, double inv) {
  const OptsDev& O = X.opts;
  const double a = S.a, b = S.b;
  const bool one = (threadIdx.x & 31) == 0;
  int halvings = 0;
  if (!fin(a) || !fin(b)) {
    if (one) deactivate(S, GPSOC_ENONFINITE);
    return;
  }
  if (pos(b) || (zero(b) && !neg(a))) {
    if (one) {
      if (zero(S.beta)) {
        if (O.phase32) S.active = 0;   // rounding floor of the FP32 phase: hand over to FP64
        else deactivate(S, GPSOC_ESTAGNATED);
      } else {
        // the sign test before the transform missed by rounding: redo this step with
        // beta = 0 in the next iteration (same Phi, same residual: Step 2 -> Step 1)
        S.first = 1;
        S.beta_resets++;
      }
    }
    return;
  }
  double theta = (pos(a) && neg(b)) ? -b / (2.0 * a) : O.theta_trial;
  if (O.line_search == 1) theta = exact_theta(S, inv, theta);
  bool accepted = false;
  double dE = 0.0, sn = 0.0, cs = 1.0;
  for (int h = 0; h <= O.max_halvings; ++h) {
    sincos_warp(theta, sn, cs);
    dE = energy_change_sc(S, sn, cs, inv);
    if (dE < 0.0) { accepted = true; break; }
    theta *= O.sigma;
    ++halvings;
  }
  if (!accepted) {
    if (one) {
      S.halvings += halvings;
      if (O.phase32) S.active = 0;
      else deactivate(S, GPSOC_ESTAGNATED);
    }
    return;
  }
  const double sp = sn * inv;
  const double M = S.mass[0] + S.mass[1] + S.mass[2];
  // Phi' = (cos t Phi + sin t P_t/|P_t|)/norm with P_t = P - a Phi tangent: |.|^2 = c^2 M + s'^2 |P_t|^2,
  // which is 1 up to rounding
  const double d = (cs * cs * M + sp * sp * S.P2) - 1.0;
  const double g = rsqrt1_in_range(d) ? rsqrt1(d) : rsqrt(1.0 + d);
  const double uc = cs - sp * S.acorr;
  __syncwarp();
  if (one) {
    S.theta = theta;
    S.dE = dE;
    S.dE_last = dE;
    S.upd_c = uc; S.upd_s = sp; S.upd_scale = g;
    S.halvings += halvings;
    S.pending = 1;
    S.last_par = (X.flags >> 2) & 1;
    S.iters++; S.total_iters++;
    if (X.flags & 2) S.fp32_iters++; else S.fp64_iters++;
    S.first = 0;
    S.s_prev = S.s_cur;
  }
  if (X.flags & 8) {
    // GPSOC_HYBRID: the double-word coefficients the opening pass applies, a lane each
    const int l = threadIdx.x & 31;
    const double guc = g * uc, gut = g * sp, gm = guc - 1.0;
    if (l < 3) dw_split(l == 0 ? guc : l == 1 ? gut : gm, l == 0 ? S.dw_uc : l == 1 ? S.dw_ut : S.dw_ucm1);
  }
  __syncwarp();
}

template <class V>
__device__ __forceinline__ void sc_step(const ScalarCtx& X, int s, double* scratch) {
  __shared__ SolveState sS;
  state_load(sS, X.st + s);      // visible after the barrier of the grid sums
  if (X.flags & 8) {
    // GPSOC_HYBRID: also the kinetic sums of Phi, of P and their cross term from the column pass
    const int slots[kStepSlots + 9] = {GPSOC_STEP_SLOTS, SL_KPHI0, SL_KPHI1, SL_KPHI2, SL_KX0, SL_KX1, SL_KX2,
                                       SL_KIN0, SL_KIN1, SL_KIN2};
    slot_totals<V, kStepSlots + 9, kStepSlots>(X, s, slots, X.nb_row, X.nb_col, -1, scratch);
  } else {
    const int slots[kStepSlots] = {GPSOC_STEP_SLOTS};
    slot_totals<V, kStepSlots, kStepSlots>(X, s, slots, X.nb_row, 0, -1, scratch);
  }
  if (threadIdx.x >= 32) return;
  const double inv = step_sums(X, s, scratch, sS);
  step_decide(X, sS, inv);
  if (X.flags & 8) {
    // kinetic part of alpha_l at the next iterate, exactly: Phi' = g (c Phi + t P), so
    // |k|^2 |Phi'_hat|^2 sums to g^2 (c^2 K_Phi + 2 c t K_x + t^2 K_P) per component, a lane each
    const int l = threadIdx.x < 3 ? threadIdx.x : 0;
    const double* kq = scratch + kStepSlots + l;
    const double c = sS.upd_c, t = sS.upd_s, g = sS.upd_scale;
    const double k = sS.pending != 0 ? (g * g) * (c * c * kq[0] + 2.0 * c * t * kq[3] + t * t * kq[6]) : kq[0];
    __syncwarp();
    if (threadIdx.x < 3) sS.kin[l] = k;
  }
  mirror32_warp(sS);
  state_store_warp(X.st + s, sS);
}

}  // namespace gpsoc
