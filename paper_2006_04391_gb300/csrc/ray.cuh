// Implicit-Euler step of a proportional law: the 5-dimensional Newton system
// of solver.cuh collapses to one scalar equation.
//
// A law declares kRay when (i) psi is quadratic and depends on y through the
// deviatoric strain e_s - P y with an isotropic stiffness, and (ii) phi =
// c_phi q^a_phi with q = (2/3) zdot:zdot, the norm of the same metric.  Then
// psi_y(e_s, 0), psi_yy d and phi_v(theta d / h) are all parallel for the
// predictor d (the increment that relaxes the deviatoric trial strain: d =
// the y-components of e_s), so R(theta d) = 0 has its root on the predictor
// segment and the segment minimisation of solver.cuh already gives it; the
// Newton polish that followed it only confirmed the root (five-direction AD
// sweeps, a 5x5 factorisation).  With A = -d.psi_y(e_s, 0) = 2 mu (e_s:e_s)
// and d.phi_v(theta d/h) = 2 mu (e_s:e_s) k(theta) the root solves
//   k(theta) = 1 - theta,   k(theta) = c0 theta (E2 theta^2)^(a_phi - 1),  E2 = e_s:e_s,
//   c0 = 2 a_phi c_phi / (3 mu h) (2 / (3 h^2))^(a_phi - 1)      (once per step;
//   where that leaves the FP64 range, n < 0.1, on E2 scaled by a power of four),
// and with t = 1 - theta
//   w = theta d,   sigma = kappa tr(eps) 1 + 2 mu t e_s,
//   C_t = kappa 1x1 + 2 mu t I_dev - 2 mu (1 - p) theta t / (p t + theta) n x n,
//   p = 2 a_phi - 1,  n = e_s / |e_s|
// (the last term from the derivative of the scalar equation, Eq.
// tangent_formula restricted to the segment).  The host tests compare this
// with the general solver (the AD-driven Newton) and the oracle over n from 1
// to 20 and trial strains from 1e-25 to 1e-1.
//
// Solution: theta in FP32 from the equation in u = log2 theta (convex and
// increasing; Newton from an upper bound decreases monotonically onto the
// root), then Halley steps in the working precision on the equation itself.
// One step cubes the seed's ~1e-7: its remainder is below 1e-18, so a voxel
// takes one power in the working precision.  FP64 operations per voxel: 74
// (33 in the FP32-bulk mode), where the line search and Newton steps took about
// 800.
//
// Bound: FP64 the FP64 pipe (74 operations at 629 G/s: 8.5 G voxel/s at 100 %;
// the pipe is 87 % busy, its maximum in any kernel here), FP32 the memory (96
// bytes a voxel).  Measured on GB300 against the general solver: FP64 3.0 M
// voxels (n = 10) 5208 -> 415 us (7.2 G voxel/s), FP64 with tangent 1.0 M voxels
// 2793 -> 233 us, FP32 5.0 M voxels 266 -> 86 us (5.6 TB/s), FP32 bulk +
// correction 2^24 voxels 3015 -> 1120 us (2450 with the correction in FP64; 2.9
// TB/s), the FP32 material kernel of the scheme at 256^3 1199 -> 294 us.
#pragma once

#include "dpow.cuh"
#include "solver.cuh"

namespace gsm {

// Constants of the scalar equation of one law and one step size.
struct RayConst {
  double c0, am1, p, mu, kappa;
  int sh;          // c0 belongs to 2^(2 sh) E2 (0 but where c0 of E2 itself is out of range)
  float am1f, pf, inv_pf, muf, kappaf;
  float lg_c0;     // log2 c0
  float c0m;       // c0 = c0m 2^c0e, c0m in [1, 2)
  int c0e;
  float lg_floor;  // log2 of 1e-140 h (2^sh): rates below 1e-140 of |d| / h are no flow
  df am1d, pd, c0d;  // am1, p and c0 2^-c0e as double-float pairs (the FP32-bulk correction)
};

AD_HD float lg2_approx(float x) {
#if defined(__CUDA_ARCH__)
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return std::log2(x);
#endif
}
AD_HD float ex2_approx(float x) {
#if defined(__CUDA_ARCH__)
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return std::exp2(x);
#endif
}
AD_HD float rcp_approx(float x) {
#if defined(__CUDA_ARCH__)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}

// floor(log2 x) of a positive normal FP32 x.
AD_HD int ilog2_pos(float x) {
#if defined(__CUDA_ARCH__)
  return (int)(__float_as_uint(x) >> 23) - 127;
#else
  unsigned b;
  std::memcpy(&b, &x, sizeof b);
  return (int)(b >> 23) - 127;
#endif
}

AD_HD RayConst make_ray(const LawParams<double>& p, double h) {
  RayConst r;
  r.am1 = p.a_phi - 1.0;
  r.p = 1.0 + 2.0 * r.am1;
  r.mu = p.mu;
  r.kappa = p.lam + p.mu * (2.0 / 3.0);
  r.c0 = 2.0 * p.a_phi * p.c_phi / (3.0 * p.mu * h) * ::pow(2.0 / (3.0 * h * h), r.am1);
  r.sh = 0;
  if (p.L_ode > 0.0 && !(r.c0 > 1e-120 && r.c0 < 1e120)) {
    // the same as C (X E2 theta^2)^(a_phi - 1) theta with C = sigma0 / (3 mu h edot0) and X = 2 / (3 h^2 edot0^2)
    const double C = 1.0 / (p.L_ode * h), X = 0.5 * p.q_ode * C * C;
    r.sh = (int)::rint(0.5 * ::log2(X));
    r.c0 = C * ::pow(::ldexp(X, -2 * r.sh), r.am1);
  }
  r.am1f = (float)r.am1;
  r.pf = (float)r.p;
  r.inv_pf = (float)(1.0 / r.p);
  r.muf = (float)r.mu;
  r.kappaf = (float)r.kappa;
  r.lg_c0 = (float)::log2(r.c0);
  r.c0e = (int)((fpow::bits_of(r.c0) >> 52) & 0x7ff) - 1023;
  r.c0m = f32_of(r.c0, -r.c0e);
  r.lg_floor = (float)(::log2(1e-140 * h) + r.sh);
  r.am1d = df_of(r.am1);
  r.pd = df_of(r.p);
  r.c0d = df_of(r.c0, -r.c0e);
  return r;
}

// log2 x of a positive normal FP64 x to FP32 accuracy, whatever its exponent.
AD_HD float lg2_of(double x) {
  const uint64_t b = fpow::bits_of(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  const float m = f32_of(x, -e);
  return (float)e + lg2_approx(m);
}

// u = log2 theta of the root of K theta^p + theta = 1, L = log2 K, p > 0.
// Both terms are at most 1 at the root, so u <= min(0, -L/p); at that bound
// the larger term is 1, and Newton on the convex increasing function of u
// decreases monotonically onto the root (three to five iterations).
AD_HD float ray_seed(float L, float p, float inv_p, int& iters) {
  float u = fminf(0.0f, -L * inv_p);
  iters = 0;
  for (int k = 0; k < 16; ++k) {
    ++iters;
    const float a = ex2_approx(L + p * u), b = ex2_approx(u);
    const float du = 1.44269504f * (1.0f - a - b) * rcp_approx(p * a + b);
    u += du;
    if (!(fabsf(du) > 2e-4f)) break;  // quadratic: the next step is below 1e-7
  }
  return fminf(u, 0.0f);
}

struct RayRoot {
  bool flows;
  bool bad;   // the trial strain is not finite, or its square is not
  bool conv;  // no flow, or the last step met its tolerance
  int n_eval, n_model;
};

// The root in FP64: theta and t = 1 - theta, each to its own rounding.
AD_HD RayRoot ray_root(const RayConst& c, double E2, bool active, double& theta, double& t) {
  RayRoot r{false, false, true, 0, 0};
  theta = 0.0;
  t = 1.0;
  // E2 = 0 (a stress-free deviatoric state), NaN or out of range: no flow
  const int e2 = (int)((fpow::bits_of(E2) >> 52) & 0x7ff), e2s = e2 + 2 * c.sh;
  r.bad = active && (e2 > 1023 + 996 || e2s > 1023 + 996);
  r.conv = !r.bad;
  if (!active || e2 < 1023 - 996 || e2s < 1023 - 996 || r.bad) return r;
  E2 = fpow::double_of(fpow::bits_of(E2) + ((uint64_t)(int64_t)(2 * c.sh) << 52));
  const float lgE = lg2_of(E2);
  const float u = ray_seed(c.lg_c0 + c.am1f * lgE, c.pf, c.inv_pf, r.n_model);
  if (!(u + 0.5f * lgE > c.lg_floor) || !(u > -1000.0f)) return r;
  r.flows = true;
  r.conv = false;
  const float uf = floorf(u);
  double th = f64_of(ex2_approx(u - uf), (int)uf);
  for (int it = 0; it < 8; ++it) {
    ++r.n_eval;
    const double s = 1.0 - th;
    const double k = c.c0 * th * fpow::pow_pos(E2 * (th * th), c.am1);
    const double pk = c.p * k;
    const double D = pk + th;  // theta d/dtheta of k + theta
    // 1/D by one Newton step from the FP32 reciprocal (relative error ~1e-14)
    const int e = (int)((fpow::bits_of(D) >> 52) & 0x7ff) - 1023;
    const float Df = f32_of(D, -e);
    const float y0 = rcp_approx(Df);
    double y = f64_of(y0, -e);
    y = fma(y, fma(-D, y, 1.0), y);
    const double eta = (s - k) * y;  // Newton step of ln theta
    // Halley: eta / (1 + eta (p - 1)/2 pk/D); the correction is O(eta^2), FP32
    const float ef = f32_of(eta);
    const float q = 0.5f * (c.pf - 1.0f) * f32_of(pk, -e) * y0 * ef;
    const double step = eta - eta * f64_of(q * rcp_approx(1.0f + q));
    const double dth = th * step;
    theta = th + dth;
    t = s - dth;
    if (!(fabsf(ef) > 8e-6f)) {  // remainder below eta^3 / 10
      r.conv = ef == ef;
      break;
    }
    th = theta > 0.0 ? theta : 0.5 * th;
  }
  return r;
}

// x 2^k as a double-float pair by integer operations alone: hi is x truncated
// to FP32, lo the 29 mantissa bits below it.
AD_HD df df_bits(double x, int k) {
  const uint64_t b = fpow::bits_of(x);
  const float lo = (float)(int)(b & 0x1fffffffu);
  const int e = (int)((b >> 52) & 0x7ff) - 1023 - 52 + k;
  const float sc = e < -126 ? 0.0f : exp2i(e, 0.0f);
  return df{f32_of(x, k), (b >> 63) ? -lo * sc : lo * sc};
}

// The root of the FP32-bulk mode: FP32 seed, then the Halley step with the
// equation's residual in double-float arithmetic (2^-45, the accuracy of this
// mode's correction), on e_s scaled by 2^-k.  FP64 operations: three inside the
// power and one per result, where ray_root takes about 45; the FP64 pipe runs
// at 1/64 of the FP32 rate.  Returns false where the pairs do not reach (a zero,
// subnormal or non-finite trial strain, a start far from the root): the caller
// takes ray_root.
AD_HD bool ray_root_df(const RayConst& c, const double (&es)[6], int k, bool active, RayRoot& r, double& theta,
                       double& t) {
  r = RayRoot{false, false, true, 0, 0};
  theta = 0.0;
  t = 1.0;
  if (!active) return true;
  // E2 = e_s:e_s, scaled: squares of the pairs, normal and shear parts apart
  df n, h;
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const df a = df_bits(es[i], -k);
    const float p = dfo::mul_rn(a.hi, a.hi);
    const float q = dfo::fma_rn(a.hi + a.hi, a.lo, dfo::fma_rn(a.hi, a.hi, -p));
    df& s = i < 3 ? n : h;
    if (i % 3 == 0) {
      s = df{p, q};
    } else {
      const df u = dfo::two_sum(s.hi, p);
      s = df{u.hi, dfo::add_rn(s.lo, dfo::add_rn(u.lo, q))};
    }
  }
  const df u2 = dfo::two_sum(n.hi, 0.5f * h.hi);
  const df E2 = dfo::fast_two_sum(u2.hi, dfo::add_rn(u2.lo, dfo::fma_rn(0.5f, h.lo, n.lo)));
  if (!(E2.hi > 0.25f && E2.hi < 64.0f)) return false;  // zero, non-finite or subnormal trial strain
  const float lgE = lg2_approx(E2.hi) + 2.0f * (float)(k + c.sh);
  const float u = ray_seed(c.lg_c0 + c.am1f * lgE, c.pf, c.inv_pf, r.n_model);
  // (no flow: the rules of ray_root)
  if (!(u + 0.5f * lgE > c.lg_floor) || !(u > -1000.0f)) return true;
  // theta = 2^et tm, tm near 1: a flow of any size takes the same FP32 pairs
  // (below 2^-40 the FP64 root took over before: n = 20, strains of 2e-5, 4.2 M
  // voxels 893 -> 336 us; a flowing batch as before)
  // (et = u rounded, by an addition: no conversion)
  constexpr float magic = 12582912.0f;  // 1.5 2^23
  const float um = u + magic;
  const int et = (int)(dpow::fbits(um) - 0x4b400000u);
  const float sc = et < -126 ? 0.0f : exp2i(et, 0.0f);
  float tm = ex2_approx(u - (um - magic));
  for (int it = 0; it < 8; ++it) {
    ++r.n_eval;
    const float t2 = dfo::mul_rn(tm, tm);
    const df x = E2 * df{t2, dfo::fma_rn(tm, tm, -t2)};
    df F;
    // (one exit: a second one at the loop's end cost a voxel 1 us of latency)
    if (!(tm > 0.25f && tm < 4.0f) ||
        !dpow::pow_scaled(x, 2 * (k + c.sh + et), c.am1, c.am1d, c.c0d, c.c0e + et, F))
      return false;
    const float th = tm * sc;
    const df kk = F * tm;
    const df s = dfo::two_sum(1.0f, -th);
    const df R = s - kk;
    const df D = kk * c.pd + th;
    // eta = R / D as a pair, then Halley's factor (FP32: second order)
    const float y0 = rcp_approx(D.hi);
    const float eta = R.hi * y0;
    const float q = 0.5f * (c.pf - 1.0f) * c.pf * kk.hi * y0 * eta;
    const float rest = dfo::fma_rn(-eta, D.hi, R.hi) + dfo::fma_rn(-eta, D.lo, R.lo);
    const df step = dfo::fast_two_sum(eta, dfo::fma_rn(rest, y0, -eta * q * rcp_approx(1.0f + q)));
    const df dth = step * tm;
    if (!(fabsf(eta) > 8e-6f)) {
      theta = fpow::double_of(fpow::bits_of(f64_of(dth + tm)) + ((uint64_t)(int64_t)et << 52));
      t = f64_of(s - df{dth.hi * sc, dth.lo * sc});
      r.flows = true;
      return true;
    }
    tm = tm + dth.hi;
  }
  return false;
}

AD_HD unsigned ray_status(const RayRoot& r, bool correction) {
  unsigned st = r.conv ? ST_CONVERGED : r.bad ? ST_NONFINITE : ST_CAP;
  st |= (unsigned)(r.n_model & 0x7f) << ST_MODEL_SHIFT;
  if (correction)
    st |= ((unsigned)r.n_eval << ST_NEWTON_SHIFT) | ((unsigned)(r.n_eval & 0xf) << ST_FIX_SHIFT);
  else
    st |= (unsigned)r.n_eval << ST_LINE_SHIFT;
  return st;
}

template <class T> AD_HD T recip_of(T x);
template <> AD_HD double recip_of(double x) { return recip_pos(x); }
template <> AD_HD float recip_of(float x) { return 1.0f / x; }

// Consistent tangent (21 packed entries) at the root.
template <class T>
AD_HD void ray_tangent(T mu, T kappa, T p, const T (&es)[6], T E2, T theta, T t, bool flows, T (&C21)[21]) {
  T m[6], cm[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) m[i] = i < 3 ? es[i] : T(0.5) * es[i];
  T c3 = T(0);
  if (flows) c3 = T(-2) * mu * (T(1) - p) * (theta * t) * recip_of<T>((p * t + theta) * E2);
#pragma unroll
  for (int i = 0; i < 6; ++i) cm[i] = c3 * m[i];
  const T g = mu * t;                                // shear modulus of the deviatoric part
  const T off = kappa - g * T(2.0 / 3.0), dia = off + T(2) * g;
  int q = 0;
#pragma unroll
  for (int i = 0; i < 6; ++i)
#pragma unroll
    for (int j = i; j < 6; ++j) {
      const T base = i == j ? (i < 3 ? dia : g) : (j < 3 ? off : T(0));
      C21[q++] = cm[i] * m[j] + base;
    }
}

// Trial state and root of one voxel in FP64 (correction: the FP32-bulk mode).
struct RayVoxel {
  double es[6], tr, theta, t;
  RayRoot r;
  AD_HD double norm2() const {
    return es[0] * es[0] + es[1] * es[1] + es[2] * es[2] + 0.5 * (es[3] * es[3] + es[4] * es[4] + es[5] * es[5]);
  }
};
template <class Law>
AD_HD void ray_solve(const RayConst& c, const double (&eps)[6], const double (&yn)[5], bool active, bool correction,
                     RayVoxel& v) {
  v.tr = Law::trial_strain(eps, yn, v.es);
  if (!correction || !ray_root_df(c, v.es, ilog2_max(v.es), active, v.r, v.theta, v.t))
    v.r = ray_root(c, v.norm2(), active, v.theta, v.t);
}
AD_HD void ray_stress(const RayConst& c, const double (&es)[6], double tr, double t, double (&sig)[6]) {
  const double hyd = c.kappa * tr, g = c.mu * t, g2 = g + g;
#pragma unroll
  for (int i = 0; i < 3; ++i) sig[i] = fma(g2, es[i], hyd);
#pragma unroll
  for (int i = 3; i < 6; ++i) sig[i] = g * es[i];
}

// One voxel in FP64 (correction: the FP32-bulk mode and its status bookkeeping).
template <class Law>
AD_HD unsigned voxel_ray(const RayConst& c, const double (&eps)[6], const double (&zn)[6], bool active,
                         bool correction, double (&sig)[6], double (&z)[6], double* C21) {
  const double yn[5] = {zn[0], zn[1], zn[3], zn[4], zn[5]};
  RayVoxel v;
  ray_solve<Law>(c, eps, yn, active, correction, v);
  ray_stress(c, v.es, v.tr, v.t, sig);
  const bool flows = v.r.flows;
  z[0] = flows ? fma(v.theta, v.es[0], yn[0]) : yn[0];
  z[1] = flows ? fma(v.theta, v.es[1], yn[1]) : yn[1];
  z[2] = -(z[0] + z[1]);
#pragma unroll
  for (int i = 3; i < 6; ++i) z[i] = flows ? fma(v.theta, v.es[i], yn[i - 1]) : yn[i - 1];
  if (C21) {
    double C[21];
    ray_tangent<double>(c.mu, c.kappa, c.p, v.es, v.norm2(), v.theta, v.t, flows, C);
#pragma unroll
    for (int q = 0; q < 21; ++q) C21[q] = C[q];
  }
  return ray_status(v.r, correction);
}

// The Newton matrix at the root, K = psi_yy + phi_vv / h, in the metric M of the
// y coordinates (z:z = y^T M y) and d, the y components of e_s:
//   K = (2 mu / theta) (M + t (p - 1)/E2 (M d)(M d)^T),
//   phi_vv / h = K - 2 mu M = (2 mu t / theta) (M + (p - 1)/E2 (M d)(M d)^T),
// for the adjoint: K^-1 by Sherman and Morrison, no factorisation.
AD_HD void metric_apply(const double (&y)[5], double (&out)[5]) {
  const double s = y[0] + y[1];
  out[0] = y[0] + s;
  out[1] = y[1] + s;
  out[2] = 0.5 * y[2];
  out[3] = 0.5 * y[3];
  out[4] = 0.5 * y[4];
}
// b = K^-1 g
AD_HD void ray_K_solve(double mu, double p, double theta, double t, double E2, const double (&d)[5],
                       const double (&g)[5], double (&b)[5]) {
  const double f = theta / (2.0 * mu);
  double dg = 0.0;
#pragma unroll
  for (int a = 0; a < 5; ++a) dg += d[a] * g[a];
  const double w = t * (1.0 - p) * dg / (E2 * (theta + p * t));
  const double m = (g[0] + g[1]) * (1.0 / 3.0);
  b[0] = f * ((g[0] - m) + w * d[0]);
  b[1] = f * ((g[1] - m) + w * d[1]);
#pragma unroll
  for (int a = 2; a < 5; ++a) b[a] = f * (2.0 * g[a] + w * d[a]);
}
// out = (phi_vv / h) b
AD_HD void ray_flow_apply(double mu, double p, double theta, double t, double E2, const double (&d)[5],
                          const double (&b)[5], double (&out)[5]) {
  double Mb[5], Md[5];
  metric_apply(b, Mb);
  metric_apply(d, Md);
  double db = 0.0;
#pragma unroll
  for (int a = 0; a < 5; ++a) db += d[a] * Mb[a];
  const double f = 2.0 * mu * t / theta, w = (p - 1.0) * db / E2;
#pragma unroll
  for (int a = 0; a < 5; ++a) out[a] = f * (Mb[a] + w * Md[a]);
}

// FP32 power (2^e m)^a with lgm = log2 m: the integer nearest the exponent is
// split off and the product a e kept with its remainder, so the result carries
// ~2^-23, not 2^-23 of the exponent.  Returns r with the power = 2^n r.
AD_HD float ray_pow(float a, int e, float lgm, int& n) {
  const float ef = (float)e;
  const float yh = a * ef;
  const float yl = fmaf(a, ef, -yh);
  const float ni = rintf(fmaf(a, lgm, yh));
  n = (int)ni;
  return ex2_approx((yh - ni) + fmaf(a, lgm, yl));
}

// a + b = s + e exactly.
AD_HD float two_sum_f32(float a, float b, float& e) {
  const float s = a + b, bb = s - a;
  e = (a - (s - bb)) + (b - bb);
  return s;
}

// One voxel in FP32.  E2 is formed on e_s scaled by 2^-k, k = the exponent of
// its largest entry, so that no trial strain under- or overflows.
//
// Rounding: the trace enters all three normal components, so its own rounding
// is carried along (tr + tr_lo = eps_11 + eps_22 + eps_33 up to one rounding of
// tr_lo), and 1/3 as a pair; a voxel past theta = 1/2 takes z = dev(eps) - t e_s, where
// z_n + theta e_s would add the rounding of e_s = dev(eps) - z_n a second time.
// Against 64 bits on the batch (n = 5, h = 0.01, 2-norm, GB300): sigma 3.4e-8, z
// 3.8e-8; the general solver 5.5e-8 and 5.1e-8 (its Newton step projects the
// trace's rounding out), a plain trial strain 5.6e-8 and 5.9e-8.  5.0 M voxels
// 87.9 -> 85.6 us; an FP32 iteration of the scheme at 256^3 1.284 -> 1.303 ms.
template <class Law>
AD_HD unsigned voxel_ray(const RayConst& c, const float (&eps)[6], const float (&zn)[6], bool active, bool,
                         float (&sig)[6], float (&z)[6], float* C21) {
  const float yn[5] = {zn[0], zn[1], zn[3], zn[4], zn[5]};
  float es[6], ss[6], tr_lo, lo2;
  const float tr = two_sum_f32(two_sum_f32(eps[0], eps[1], tr_lo), eps[2], lo2);
  tr_lo += lo2;
  constexpr float third = (float)(1.0 / 3.0), third_lo = (float)(1.0 / 3.0 - (double)third);
  const float m_lo = fmaf(third, tr_lo, third_lo * tr);
  auto dev = [&](int i) { return i < 3 ? fmaf(-third, tr, eps[i]) - m_lo : eps[i]; };
  es[0] = dev(0) - yn[0];
  es[1] = dev(1) - yn[1];
  es[2] = dev(2) + (yn[0] + yn[1]);
#pragma unroll
  for (int i = 3; i < 6; ++i) es[i] = eps[i] - yn[i - 1];
  const int k0 = ilog2_max(es);
  const int k = k0 > 126 ? 126 : k0;
  const float inv_s = exp2i(-k, 0.0f);
#pragma unroll
  for (int i = 0; i < 6; ++i) ss[i] = es[i] * inv_s;
  const float E2 = ss[0] * ss[0] + ss[1] * ss[1] + ss[2] * ss[2] +
                   0.5f * (ss[3] * ss[3] + ss[4] * ss[4] + ss[5] * ss[5]);  // in [0.5, 24)
  const bool bad = active && !(E2 < 1e30f);
  RayRoot r{false, bad, !bad, 0, 0};
  float theta = 0.0f, t = 1.0f;
  if (active && E2 > 0.0f && E2 < 1e30f) {
    const float lgE = lg2_approx(E2) + 2.0f * (float)(k + c.sh);
    const float u = ray_seed(c.lg_c0 + c.am1f * lgE, c.pf, c.inv_pf, r.n_model);
    if (u > -120.0f) {
      r.flows = true;
      r.conv = false;
      float th = ex2_approx(u);
      for (int it = 0; it < 4; ++it) {
        ++r.n_eval;
        const float s = 1.0f - th;
        // (E2 th^2)^am1 with th = tm 2^et, E2 tm^2 in [0.5, 96)
        const int et = ilog2_pos(th);
        const float tm = th * exp2i(-et, 0.0f);
        const float x = E2 * tm * tm;
        const int ex = ilog2_pos(x);
        int n;
        const float pw = ray_pow(c.am1f, ex + 2 * (k + c.sh + et), lg2_approx(x * exp2i(-ex, 0.0f)), n);
        n += c.c0e;
        n = n > 240 ? 240 : (n < -240 ? -240 : n);
        const int n1 = n / 2;
        const float kk = (c.c0m * th * exp2i(n1, 0.0f)) * (pw * exp2i(n - n1, 0.0f));
        const float pk = c.pf * kk;
        const float y0 = rcp_approx(pk + th);
        const float eta = (s - kk) * y0;
        const float q = 0.5f * (c.pf - 1.0f) * pk * y0 * eta;
        const float dth = th * (eta - eta * q * rcp_approx(1.0f + q));
        theta = th + dth;
        t = s - dth;
        if (!(fabsf(eta) > 1e-3f)) {
          r.conv = eta == eta;
          break;
        }
        th = theta > 0.0f ? theta : 0.5f * th;
      }
    }
  }
  unsigned st = ray_status(r, false);
  const float hyd = c.kappaf * tr, hyd_lo = c.kappaf * tr_lo, g = c.muf * t, g2 = g + g;
#pragma unroll
  for (int i = 0; i < 3; ++i) sig[i] = hyd + fmaf(g2, es[i], hyd_lo);
#pragma unroll
  for (int i = 3; i < 6; ++i) sig[i] = g * es[i];
  const bool past = theta > 0.5f;
  const float zs = past ? -t : theta;
  auto flow = [&](int i, float y) { return r.flows ? fmaf(zs, es[i], past ? dev(i) : y) : y; };
  z[0] = flow(0, yn[0]);
  z[1] = flow(1, yn[1]);
  z[2] = -(z[0] + z[1]);
#pragma unroll
  for (int i = 3; i < 6; ++i) z[i] = flow(i, yn[i - 1]);
  if (C21) {
    float C[21];
    // n x n is scale free: the tangent takes the scaled trial strain
    ray_tangent<float>(c.muf, c.kappaf, c.pf, ss, E2, theta, t, r.flows, C);
#pragma unroll
    for (int q = 0; q < 21; ++q) C21[q] = C[q];
  }
  return st;
}

}  // namespace gsm
