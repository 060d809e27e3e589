// The explicit pairs (ode23, ode12) for a proportional law without tangent, in
// its elastic deviatoric strain.
//
// With psi isotropic and Psi = c_Psi (s_A^2)^b_Psi, s_A the von Mises norm of
// A = -psi_y, the flow is ydot = Lambda x with x the y-components of
// dev(eps) - P y and
//   Lambda = 6 mu c_Psi b_Psi (12 mu^2 Q)^(b_Psi - 1) = L_ode (q_ode Q)^(b_Psi - 1),
//   Q = x0^2 + x1^2 + x0 x1 + (x2^2 + x3^2 + x4^2)/4     (s_A^2 = 12 mu^2 Q),
//   L_ode = 3 mu edot0 / sigma0,  q_ode = 12 mu^2 / sigma0^2:
// the power's base is (s_A / sigma0)^2, of order one wherever the law flows, so
// neither the base nor the factor leaves the FP64 range, whatever the units and
// the exponent (as one number, (12 mu^2)^(b_Psi - 1) overflows for E in Pa at n = 28).
// The strain is linear over the step, so x obeys the autonomous equation
//   xdot = edot - Lambda(x) x,
// and a Runge-Kutta method applied to x is the one applied to y (affine
// change of variable; the stage abscissae equal the row sums).  The stresses
// are sigma = kappa tr(eps) 1 + 2 mu x, and the pair's stress difference is
// 2 mu times the embedded difference of x: no stress is evaluated twice and
// the difference does not cancel.  y is carried beside x and takes the flow
// Lambda x of the accepted substeps: as dev(eps) - x a flow that is small beside
// the strain would be rounded to the strain's last place.
//
// Bound: the FP64 pipe.  The AD sweeps of ode23.cuh took about 800 FP64
// operations an attempt; this takes about 200 (odd integer n: Q^(b_Psi - 1) is
// a product of Q) or 290 (else: the table power).  Measured on 200 k voxels, n =
// 5, rtol 1e-3: 7568 -> 3502 us, 3177 with the voxels of a block taken from a
// shared counter (ode_kernel.cuh), the same with y beside x (the embedded
// difference from edot - f and the end rates pays for it).
#pragma once

// (included by ode23.cuh)

namespace gsm {

// |a| > |b| ? |a| : |b| on the integer pipe (a NaN wins).
AD_HD double absmax_bits(double a, double b) {
  const uint64_t m = 0x7fffffffffffffffull;
  const uint64_t x = fpow::bits_of(a) & m, y = fpow::bits_of(b) & m;
  return fpow::double_of(x > y ? x : y);
}

template <class Law, int PAIR> struct RayErkVoxel {
  double x[5], k1[5], ed[5];  // elastic deviatoric strain, its rate, the strain rate
  double y[5], L1;            // internal variables; Lambda at x
  double hyd0, dhyd;          // kappa tr(eps_n) and its increment
  double sig_old[6];
  double t, dt;
  int n_acc, n_rej;
  unsigned flags;
  bool last_rejected, done;

  AD_HD static double lambda(const LawParams<double>& p, const double (&v)[5]) {
    const double Q =
        p.q_ode * (fma(v[0], v[0] + v[1], v[1] * v[1]) + 0.25 * fma(v[4], v[4], fma(v[3], v[3], v[2] * v[2])));
    // b_Psi - 1 a small integer, from the bits (the same for every lane; an FP64
    // compare or conversion would occupy the FP64 pipe)
    const uint64_t b = fpow::bits_of(p.b_Psi);
    if (b == fpow::bits_of(3.0)) return p.L_ode * (Q * Q);
    if (b == fpow::bits_of(2.0)) return p.L_ode * Q;
    if (b == fpow::bits_of(1.0)) return p.L_ode;
    const int e = (int)(b >> 52) - 1023;
    if (e >= 2 && e <= 3 && (b & (0x000fffffffffffffull >> e)) == 0) {  // 4 <= b_Psi < 16, an integer
      const int m = (int)((b & 0x000fffffffffffffull) >> (52 - e)) + (1 << e) - 1;
      double r = Q;
      for (int i = 1; i < m; ++i) r *= Q;
      return p.L_ode * r;
    }
    return p.L_ode * fpow::pow_pos(Q, p.b_Psi - 1.0);
  }
  // k = edot - Lambda v; returns Lambda
  AD_HD double rate(const LawParams<double>& p, const double (&v)[5], double (&k)[5]) const {
    const double L = lambda(p, v);
#pragma unroll
    for (int a = 0; a < 5; ++a) k[a] = fma(-L, v[a], ed[a]);
    return L;
  }
  AD_HD void stress(const LawParams<double>& p, double hyd, const double (&v)[5], double (&s)[6]) const {
    const double m2 = p.mu + p.mu;
    s[0] = fma(m2, v[0], hyd);
    s[1] = fma(m2, v[1], hyd);
    s[2] = fma(-m2, v[0] + v[1], hyd);
    s[3] = p.mu * v[2];
    s[4] = p.mu * v[3];
    s[5] = p.mu * v[4];
  }

  AD_HD void init(const LawParams<double>& p, const double (&e0_)[6], const double (&e1_)[6], const double (&zn)[6],
                  const Step& hs, const void* = nullptr) {
    const double kappa = p.lam + p.mu * (2.0 / 3.0), inv_h = hs.inv_h;
    const double tr0 = e0_[0] + e0_[1] + e0_[2];
    double d[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) d[i] = e1_[i] - e0_[i];
    // deviators from differences: a hydrostatic strain leaves no rounding in them
    auto dev = [](const double (&e)[6], int a) {
      return a < 2 ? ((e[a] - e[1 - a]) + (e[a] - e[2])) * (1.0 / 3.0) : e[a + 1];
    };
    // (0 times: a non-finite increment or z_n shows in the stress from the start)
#pragma unroll
    for (int a = 0; a < 5; ++a) {
      ed[a] = dev(d, a) * inv_h;
      y[a] = zn[a < 2 ? a : a + 1];
      x[a] = fma(0.0, ed[a], dev(e0_, a) - y[a]);
    }
    dhyd = kappa * (d[0] + d[1] + d[2]);
    hyd0 = fma(0.0, dhyd + (y[0] + y[1]), kappa * tr0);
    L1 = rate(p, x, k1);
    stress(p, hyd0, x, sig_old);
    t = 0.0;
    dt = hs.h;
    n_acc = n_rej = 0;
    flags = 0;
    last_rejected = false;
    done = false;
  }

  AD_HD void attempt(const LawParams<double>& p, const Step& hs, const Ode23Ctl& ctl) {
    const double h = hs.h;
    if (n_acc + n_rej >= ctl.max_steps) {
      flags |= ST_CAP;
      done = true;
      return;
    }
    const bool clip = t + dt >= h;  // the substep that ends the interval ends at h exactly
    if (clip) dt = h - t;
    const double tn1 = clip ? h : t + dt;
    const double th1 = clip ? 1.0 : tn1 * hs.inv_h;
    // f: the pair's flow, sum of b_i Lambda_i x_i; xn = x + dt (edot - f), y takes dt f;
    // e: de times the embedded difference's rate
    constexpr double de = PAIR == ERK_BS23 ? 0.25 : 0.5;
    double xn[5], e[5], f[5], k[5], v[5], Ln;
    if constexpr (PAIR == ERK_BS23) {
      constexpr double b1 = 2.0 / 9.0, b2 = 1.0 / 3.0, b3 = 4.0 / 9.0;
      const double c2 = 0.5 * dt, c3 = 0.75 * dt, w1 = b1 * L1;
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        v[a] = fma(c2, k1[a], x[a]);
        f[a] = w1 * x[a];
      }
      const double w2 = b2 * rate(p, v, k);
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        f[a] = fma(w2, v[a], f[a]);
        v[a] = fma(c3, k[a], x[a]);
      }
      const double w3 = b3 * rate(p, v, k);
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        f[a] = fma(w3, v[a], f[a]);
        e[a] = ed[a] - f[a];  // sum of b_i k_i
        xn[a] = fma(dt, e[a], x[a]);
      }
      Ln = rate(p, xn, k);  // k1 of the next substep
      // the difference of the two weights, (-5/72, 1/12, 1/9, -1/8), is 1/4 (b, 0) - 1/8 (1, 0, 0, 1)
#pragma unroll
      for (int a = 0; a < 5; ++a) e[a] = fma(-0.5, k1[a] + k[a], e[a]);
    } else {
      // Heun (order 2) continued, explicit Euler embedded: difference dt/2 (k2 - k1)
#pragma unroll
      for (int a = 0; a < 5; ++a) v[a] = fma(dt, k1[a], x[a]);
      const double w1 = 0.5 * L1, w2 = 0.5 * rate(p, v, k);
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        f[a] = fma(w2, v[a], w1 * x[a]);
        xn[a] = fma(dt, ed[a] - f[a], x[a]);
        e[a] = k[a] - k1[a];
      }
      Ln = rate(p, xn, k);
    }
    double s[6];
    stress(p, fma(th1, dhyd, hyd0), xn, s);
    // stress difference of the pair (the hydrostatic parts are the same)
    const double md = p.mu * dt * de, m2d = md + md;
    const double d[6] = {m2d * e[0], m2d * e[1], -m2d * (e[0] + e[1]), md * e[2], md * e[3], md * e[4]};
    double sum = 0.0;
#pragma unroll
    for (int i = 0; i < 6; ++i) sum += scaled_sq(d[i], fma(ctl.rtol, absmax_bits(sig_old[i], s[i]), ctl.atol));
    // err^2, err the RMS; a trial step that overflows is rejected like one with a large error
    const double err2 = finite64(sum) ? sum * (1.0 / 6.0) : 1e300;
    // 0.9 err^(-1/3) (ode23), 0.9 err^(-1/2) (ode12)
    const double fac = err2 == 0.0 ? 1e300 : 0.9 * fpow::pow_pos(err2, PAIR == ERK_BS23 ? -1.0 / 6.0 : -1.0 / 4.0);
    const double grow = fmin(last_rejected ? 1.0 : 5.0, fmax(0.2, fac));
    if (err2 <= 1.0) {
      t = tn1;
#pragma unroll
      for (int a = 0; a < 5; ++a) {
        y[a] = fma(dt, f[a], y[a]);
        x[a] = xn[a];
        k1[a] = k[a];
      }
      L1 = Ln;
#pragma unroll
      for (int i = 0; i < 6; ++i) sig_old[i] = s[i];
      ++n_acc;
      last_rejected = false;
      if (clip) done = true;
    } else {
      ++n_rej;
      last_rejected = true;
    }
    dt *= grow;
  }

  AD_HD unsigned finish(double h, double (&sig)[6], double (&z)[6], double*) const {
#pragma unroll
    for (int i = 0; i < 6; ++i) sig[i] = sig_old[i];
    z[0] = y[0];
    z[1] = y[1];
    z[2] = -(y[0] + y[1]);
    z[3] = y[2];
    z[4] = y[3];
    z[5] = y[4];
    unsigned st = flags;
    if (t >= h && !(flags & ST_CAP)) st |= ST_CONVERGED;
    if (!finite64(sig[0]) || !finite64(z[0])) st |= ST_NONFINITE;
    st |= (unsigned)(n_acc < 0xffff ? n_acc : 0xffff);
    st |= (unsigned)(n_rej < 0x7ff ? n_rej : 0x7ff) << ST_ODE_REJ_SHIFT;
    return st;
  }
};

}  // namespace gsm
