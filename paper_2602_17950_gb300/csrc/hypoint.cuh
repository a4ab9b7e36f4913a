// The pointwise arithmetic of the hybrid opening pass (k_hy_upd) in double words, for the device and, in the CPU
// check of its errors (tests/test_hypoint.py), for the host; and the FP64 sums of the pass that ends an iteration.
//
// Its error may not exceed that of the same formulas with dw_add for every sum, which is what the grouping is
// chosen by: products are added in pairs (dwa_mul), pairs, states and totals with dw_add; where all terms
// are positive or the products' smaller error leaves room, dwa_sum does.  Rms errors over
// random points against that form (tests/test_hypoint.py), and those of sums normalised once at their end, which were
// here before: Phi 1.00, 1.04; H_lin Phi 0.98, 1.14; rho 0.97, 1.19; spin terms 0.99, 1.42; H(Phi) 1.00, 1.26; with four
// points to a thread <H_lin Phi, Phi> 0.86, 2.70, the integrals of rho^2 0.97, 1.22 and of |F|^2 0.97, 1.64, masses 0.96,
// 1.25.  In time it costs 6% of a 64 x 256^2 solve (22.9 to 24.2 ms), 1% of a 128^2 one.
#pragma once

#include "dword.cuh"

namespace gpsoc {

// The accepted step at one value: its change (uc - 1) f + ut q, which is also max |dPhi|'s, and H_lin's update
GPSOC_DW DF hy_change(DF ucm1, DF ut, DF f, float q) { return dw_add(dw_mul(ucm1, f), dw_mulf(ut, q)); }
GPSOC_DW DF hy_linear(DF uc, DF ut, DF h, float hq) { return dw_add(dw_mul(uc, h), dw_mulf(ut, hq)); }

// a b + c d and a b - c d, products that are new (see dwa_add)
GPSOC_DW DF hy_pair(DF a, DF b, DF c, DF d) {
  DF t = dwa_of_mul(a, b);
  dwa_mul(t, c, d);
  return t;
}
GPSOC_DW DF hy_diff(DF a, DF b, DF c, DF d) {
  DF t = dwa_of_mul(a, b);
  dwa_sub(t, c, d);
  return t;
}

// |phi_l|^2, rho and the spin terms of a point (components ordered 1, 0, -1):
// a = phi_1 conj(phi_0) + phi_0 conj(phi_-1), Fz = |phi_1|^2 - |phi_-1|^2
struct HyPoint { DF m[3], rho, ar, ai, Fz; };
GPSOC_DW HyPoint hy_point(const DF (&fx)[3], const DF (&fy)[3]) {
  HyPoint p;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    p.m[c] = dwa_of_sqd(fx[c]);
    dwa_sqd(p.m[c], fy[c]);
  }
  p.rho = p.m[0];
  dwa_sum(p.rho, p.m[1]);
  dwa_sum(p.rho, p.m[2]);
  p.ar = dw_add(hy_pair(fx[1], fx[0], fy[1], fy[0]), hy_pair(fx[2], fx[1], fy[2], fy[1]));
  p.ai = dw_add(hy_diff(fx[1], fy[0], fy[1], fx[0]), hy_diff(fx[2], fy[1], fy[2], fx[1]));
  p.Fz = p.m[0];
  dwa_sum(p.Fz, dw_neg(p.m[2]));
  return p;
}

// H(Phi) = H_lin Phi + c0 rho Phi + c1 (F.f) Phi (Eqs. eigen1-eigen3), real and imaginary parts of component c at
// out[2 c] and out[2 c + 1]
GPSOC_DW void hy_hamiltonian(const HyPoint& p, DF c0, DF c1, const DF (&fx)[3], const DF (&fy)[3], const DF (&hx)[3],
                             const DF (&hy)[3], DF (&out)[6]) {
  const DF c0r = dw_mul(c0, p.rho), cz = dw_mul(c1, p.Fz), cr = dw_mul(c1, p.ar), ci = dw_mul(c1, p.ai);
  DF up = c0r, down = c0r;             // c0 rho +- c1 Fz
  dwa_sum(up, cz);
  dwa_sum(down, dw_neg(cz));
  out[0] = dw_add(dw_add(hx[0], dw_mul(up, fx[0])), hy_diff(cr, fx[1], ci, fy[1]));
  out[1] = dw_add(dw_add(hy[0], dw_mul(up, fy[0])), hy_pair(cr, fy[1], ci, fx[1]));
  DF t = hy_pair(cr, fx[0], ci, fy[0]);
  dwa_sum(t, hy_diff(cr, fx[2], ci, fy[2]));
  out[2] = dw_add(dw_add(hx[1], dw_mul(c0r, fx[1])), t);
  t = hy_diff(cr, fy[0], ci, fx[0]);
  dwa_sum(t, hy_pair(cr, fy[2], ci, fx[2]));
  out[3] = dw_add(dw_add(hy[1], dw_mul(c0r, fy[1])), t);
  out[4] = dw_add(dw_add(hx[2], dw_mul(down, fx[2])), hy_pair(cr, fx[1], ci, fy[1]));
  out[5] = dw_add(dw_add(hy[2], dw_mul(down, fy[2])), hy_diff(cr, fy[1], ci, fx[1]));
}

// the point's terms of <H_lin Phi, Phi>, the integrals of rho^2 and |F|^2, and the masses, into a thread's sums
GPSOC_DW void hy_sums(DF (&acc)[6], const HyPoint& p, const DF (&fx)[3], const DF (&fy)[3], const DF (&hx)[3],
                      const DF (&hy)[3]) {
  DF q = hy_pair(fx[0], hx[0], fy[0], hy[0]);
  q = dw_add(q, hy_pair(fx[1], hx[1], fy[1], hy[1]));
  q = dw_add(q, hy_pair(fx[2], hx[2], fy[2], hy[2]));
  acc[0] = dw_add(acc[0], q);
  acc[1] = dw_add(acc[1], dw_sqr(p.rho));
  DF f = dwa_of_sqd(p.ar);
  dwa_sqd(f, p.ai);
  f.hi += f.hi;
  f.lo += f.lo;
  dwa_sqd(f, p.Fz);
  acc[2] = dw_add(acc[2], f);
#pragma unroll
  for (int c = 0; c < 3; ++c) acc[3 + c] = dw_add(acc[3 + c], p.m[c]);
}

// |r|^2 of an FP64 residual given as double words, in FP32: the two products' roundings, u each
GPSOC_DW float hy_square(DF x, DF y) {
  return rn_fma(x.hi, x.hi, rn_fma(y.hi, y.hi, rn_fma(x.hi + x.hi, x.lo, rn_mul(y.hi + y.hi, y.lo))));
}

// a value's terms of the radial part Re<P, Phi> of the direction and of ||P||^2 (row_inv_p_hy): FP64 sums of an FP32
// direction against the FP64 Phi, for the exact tangent correction and the normalisation of the step.  As double words
// they made the totals' error two to five times as large for a 64 x 256^2 solve of 24.2 ms instead of 24.9
GPSOC_DW void hy_radial(double& rphi, double& pp, double fx, double fy, float px, float py) {
  const double x = widen_f(px), y = widen_f(py);
  rphi += fx * x + fy * y;
  pp += x * x + y * y;
}

}  // namespace gpsoc
