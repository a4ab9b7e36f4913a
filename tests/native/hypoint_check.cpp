// Host build of csrc/hypoint.cuh for tests/test_hypoint.py: its errors over random points, in u^2 of the terms'
// moduli, beside those of the same formulas with an accurate double-word sum (dw_add) and a normalised product for
// every term.
#include <math.h>

#include <random>

#include "hypoint.cuh"

using namespace gpsoc;
typedef long double Q;   // 64 bits or more: its roundings are below 2^-14 u^2

static Q q(DF a) { return (Q)a.hi + (Q)a.lo; }
static Q mod(Q x) { return x < 0 ? -x : x; }

// the reference's product: cross terms from a product and an FMA, added to the error of the leading one
static DF r_mul(DF a, DF b) {
  const float ch = a.hi * b.hi, cl = fmaf(a.hi, b.hi, -ch), t = fmaf(a.lo, b.hi, a.hi * b.lo);
  return dw_fast_two_sum(ch, cl + t);
}
static DF r_sub(DF a, DF b) { return dw_add(a, dw_neg(b)); }

enum { PHI, HLIN, MASS1, RHO, SPIN_A, SPIN_Z, HAM, SUM_Q, SUM_RHO2, SUM_F2, SUM_MASS, COUNT };
struct Stat {
  double s2 = 0, most = 0;
  long n = 0;
  void add(Q error, Q moduli) {
    if (moduli == 0) return;
    const double r = (double)(mod(error) / moduli) * ldexp(1.0, 48);
    s2 += r * r;
    if (r > most) most = r;
    ++n;
  }
};

// rms[2][COUNT] and most[2][COUNT]: 0 the header's, 1 the reference's
extern "C" int hp_errors(int seed, int threads, int points, double* rms, double* most) {
  std::mt19937_64 gen(seed);
  std::normal_distribution<double> N;
  std::uniform_real_distribution<double> U(0, 1);
  Stat st[2][COUNT];
  for (int th = 0; th < threads; ++th) {
    DF acc[6] = {}, ref[4] = {};
    Q sum[4] = {0, 0, 0, 0}, sm[4] = {0, 0, 0, 0};
    // a condensate's amplitude at the thread's points, parameters and a step angle
    const double amp = exp(-6 * U(gen)), c0d = 50 + 400 * U(gen), c1d = 10 * N(gen), angle = pow(10, -4 * U(gen));
    const DF c0 = dw_of(c0d), c1 = dw_of(c1d);
    const DF uc = dw_of(cos(angle)), ut = dw_of(2 * sin(angle)), um = dw_of(cos(angle) - 1.0);
    for (int k = 0; k < points; ++k) {
      DF fx[3], fy[3], hx[3], hy[3];
      for (int c = 0; c < 3; ++c) {
        DF* f[2] = {&fx[c], &fy[c]};
        DF* h[2] = {&hx[c], &hy[c]};
        for (int i = 0; i < 2; ++i) {
          const DF g = dw_of(amp * N(gen)), l = dw_of(30 * amp * N(gen));
          const float p = (float)(amp * N(gen)), hp = (float)(30 * amp * N(gen));
          const Q a = q(um) * q(g), b = q(ut) * (Q)p, e = q(uc) * q(l), d = q(ut) * (Q)hp;
          const DF got = dw_add(g, hy_change(um, ut, g, p));
          const DF want = dw_add(g, dw_add(r_mul(um, g), dw_mulf(ut, p)));
          st[0][PHI].add(q(got) - (a + b + q(g)), mod(a) + mod(b) + mod(q(g)));
          st[1][PHI].add(q(want) - (a + b + q(g)), mod(a) + mod(b) + mod(q(g)));
          const DF hg = hy_linear(uc, ut, l, hp), hw = dw_add(r_mul(uc, l), dw_mulf(ut, hp));
          st[0][HLIN].add(q(hg) - (e + d), mod(e) + mod(d));
          st[1][HLIN].add(q(hw) - (e + d), mod(e) + mod(d));
          *f[i] = g;
          *h[i] = l;
        }
      }
      Q X[3], Y[3], m[3];
      for (int c = 0; c < 3; ++c) { X[c] = q(fx[c]); Y[c] = q(fy[c]); m[c] = X[c] * X[c] + Y[c] * Y[c]; }
      const Q rho = m[0] + m[1] + m[2], Fz = m[0] - m[2], zm = m[0] + m[2];
      const Q ar = X[1] * X[0] + Y[1] * Y[0] + X[2] * X[1] + Y[2] * Y[1], ai = X[1] * Y[0] - Y[1] * X[0] + X[2] * Y[1] - Y[2] * X[1];
      const Q arm = mod(X[1] * X[0]) + mod(Y[1] * Y[0]) + mod(X[2] * X[1]) + mod(Y[2] * Y[1]);
      const Q aim = mod(X[1] * Y[0]) + mod(Y[1] * X[0]) + mod(X[2] * Y[1]) + mod(Y[2] * X[1]);
      // the reference
      DF rm[3];
      for (int c = 0; c < 3; ++c) rm[c] = dw_add(r_mul(fx[c], fx[c]), r_mul(fy[c], fy[c]));
      const DF rr = dw_add(dw_add(rm[0], rm[1]), rm[2]), rz = r_sub(rm[0], rm[2]);
      const DF ra = dw_add(dw_add(r_mul(fx[1], fx[0]), r_mul(fy[1], fy[0])), dw_add(r_mul(fx[2], fx[1]), r_mul(fy[2], fy[1])));
      const DF ri = dw_add(r_sub(r_mul(fx[1], fy[0]), r_mul(fy[1], fx[0])), r_sub(r_mul(fx[2], fy[1]), r_mul(fy[2], fx[1])));
      DF w[6];
      w[0] = dw_add(r_mul(rz, fx[0]), r_sub(r_mul(ra, fx[1]), r_mul(ri, fy[1])));
      w[1] = dw_add(r_mul(rz, fy[0]), dw_add(r_mul(ra, fy[1]), r_mul(ri, fx[1])));
      w[2] = dw_add(dw_add(r_mul(ra, fx[0]), r_mul(ri, fy[0])), r_sub(r_mul(ra, fx[2]), r_mul(ri, fy[2])));
      w[3] = dw_add(r_sub(r_mul(ra, fy[0]), r_mul(ri, fx[0])), dw_add(r_mul(ra, fy[2]), r_mul(ri, fx[2])));
      w[4] = r_sub(dw_add(r_mul(ra, fx[1]), r_mul(ri, fy[1])), r_mul(rz, fx[2]));
      w[5] = r_sub(r_sub(r_mul(ra, fy[1]), r_mul(ri, fx[1])), r_mul(rz, fy[2]));
      const DF rc = r_mul(c0, rr);
      for (int c = 0; c < 3; ++c) {
        w[2 * c] = dw_add(dw_add(hx[c], r_mul(rc, fx[c])), r_mul(c1, w[2 * c]));
        w[2 * c + 1] = dw_add(dw_add(hy[c], r_mul(rc, fy[c])), r_mul(c1, w[2 * c + 1]));
        ref[0] = dw_add(ref[0], dw_add(r_mul(fx[c], hx[c]), r_mul(fy[c], hy[c])));
      }
      ref[1] = dw_add(ref[1], r_mul(rr, rr));
      const DF r2 = dw_add(r_mul(ra, ra), r_mul(ri, ri));
      ref[2] = dw_add(ref[2], dw_add(dw_add(r2, r2), r_mul(rz, rz)));
      ref[3] = dw_add(ref[3], rm[0]);
      // the header
      const HyPoint p = hy_point(fx, fy);
      DF h[6];
      hy_hamiltonian(p, c0, c1, fx, fy, hx, hy, h);
      hy_sums(acc, p, fx, fy, hx, hy);
      for (int c = 0; c < 3; ++c) { st[0][MASS1].add(q(p.m[c]) - m[c], m[c]); st[1][MASS1].add(q(rm[c]) - m[c], m[c]); }
      st[0][RHO].add(q(p.rho) - rho, rho); st[1][RHO].add(q(rr) - rho, rho);
      st[0][SPIN_A].add(q(p.ar) - ar, arm); st[1][SPIN_A].add(q(ra) - ar, arm);
      st[0][SPIN_A].add(q(p.ai) - ai, aim); st[1][SPIN_A].add(q(ri) - ai, aim);
      st[0][SPIN_Z].add(q(p.Fz) - Fz, zm); st[1][SPIN_Z].add(q(rz) - Fz, zm);
      const Q C0 = q(c0), C1 = q(c1), M1 = mod(C1);
      const Q f[6] = {Fz * X[0] + ar * X[1] - ai * Y[1], Fz * Y[0] + ar * Y[1] + ai * X[1],
                      ar * X[0] + ai * Y[0] + ar * X[2] - ai * Y[2], ar * Y[0] - ai * X[0] + ar * Y[2] + ai * X[2],
                      ar * X[1] + ai * Y[1] - Fz * X[2], ar * Y[1] - ai * X[1] - Fz * Y[2]};
      const Q x = mod(X[1]), y = mod(Y[1]);
      const Q fm[6] = {zm * mod(X[0]) + arm * x + aim * y, zm * mod(Y[0]) + arm * y + aim * x,
                       arm * (mod(X[0]) + mod(X[2])) + aim * (mod(Y[0]) + mod(Y[2])),
                       arm * (mod(Y[0]) + mod(Y[2])) + aim * (mod(X[0]) + mod(X[2])),
                       zm * mod(X[2]) + arm * x + aim * y, zm * mod(Y[2]) + arm * y + aim * x};
      for (int i = 0; i < 6; ++i) {
        const Q u = i & 1 ? Y[i / 2] : X[i / 2], l = i & 1 ? q(hy[i / 2]) : q(hx[i / 2]);
        const Q e = l + C0 * rho * u + C1 * f[i], moduli = mod(l) + C0 * rho * mod(u) + M1 * fm[i];
        st[0][HAM].add(q(h[i]) - e, moduli);
        st[1][HAM].add(q(w[i]) - e, moduli);
        sum[0] += u * l;
        sm[0] += mod(u * l);
      }
      sum[1] += rho * rho; sm[1] += rho * rho;
      sum[2] += 2 * (ar * ar + ai * ai) + Fz * Fz; sm[2] += 2 * (arm * arm + aim * aim) + zm * zm;
      sum[3] += m[0]; sm[3] += m[0];
    }
    for (int k = 0; k < 4; ++k) {
      st[0][SUM_Q + k].add(q(acc[k]) - sum[k], sm[k]);
      st[1][SUM_Q + k].add(q(ref[k]) - sum[k], sm[k]);
    }
  }
  for (int v = 0; v < 2; ++v)
    for (int k = 0; k < COUNT; ++k) {
      rms[v * COUNT + k] = sqrt(st[v][k].s2 / st[v][k].n);
      most[v * COUNT + k] = st[v][k].most;
    }
  return COUNT;
}

// sums of a thread's direction p (pairs) against phi (pairs) by hy_radial, and their errors
extern "C" void hp_radial(int n, const double* phi, const float* p, double* got, double* want, double* moduli) {
  double r = 0.0, s = 0.0;
  Q er = 0, es = 0, mr = 0;
  for (int i = 0; i < n; ++i) {
    hy_radial(r, s, phi[2 * i], phi[2 * i + 1], p[2 * i], p[2 * i + 1]);
    for (int k = 2 * i; k < 2 * i + 2; ++k) {
      er += (Q)phi[k] * p[k];
      mr += mod((Q)phi[k] * p[k]);
      es += (Q)p[k] * p[k];
    }
  }
  got[0] = r; got[1] = s;
  want[0] = (double)(r - er); want[1] = (double)(s - es);
  moduli[0] = (double)mr; moduli[1] = (double)es;
}

// largest errors in u of |r|^2 by hy_square and of the density's FP32 value, over n random residuals and points
extern "C" void hp_fp32(int seed, int n, double* most) {
  std::mt19937_64 gen(seed);
  std::normal_distribution<double> N;
  std::uniform_real_distribution<double> U(0, 1);
  most[0] = most[1] = 0.0;
  for (int i = 0; i < n; ++i) {
    const double scale = exp(-20 * U(gen));
    DF f[6], fx[3], fy[3];
    for (int k = 0; k < 6; ++k) f[k] = dw_of(scale * N(gen));
    for (int c = 0; c < 3; ++c) { fx[c] = f[2 * c]; fy[c] = f[2 * c + 1]; }
    const double x = scale * N(gen), y = scale * N(gen);
    const Q r2 = (Q)x * x + (Q)y * y, got = hy_square(dw_of(x), dw_of(y));
    Q rho = 0;
    for (int k = 0; k < 6; ++k) rho += q(f[k]) * q(f[k]);
    const double e[2] = {(double)(mod(got - r2) / r2), (double)(mod(hy_point(fx, fy).rho.hi - rho) / rho)};
    for (int k = 0; k < 2; ++k) most[k] = e[k] * 16777216.0 > most[k] ? e[k] * 16777216.0 : most[k];
  }
}
