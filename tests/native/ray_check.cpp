// Test-only host build: the scalar equation of a proportional law (ray.cuh)
// against the general solver (AD-driven Newton) instantiated on the same
// potentials, in the three precision modes.
#include <cstdint>

#include "../../paper_2006_04391_gb300/csrc/common.cuh"
#include "../../paper_2006_04391_gb300/csrc/voxel.cuh"
#include "../../paper_2006_04391_gb300/csrc/ode23.cuh"

using namespace gsm;

// The same potentials without the certificate: takes the general path.
struct GeneralNorton : NortonDev {
  static constexpr bool kRay = false;
};

template <class Law>
static void run(int mode, const double* prm, int64_t n, const double* eps, const double* zn, double h, double* sig,
                double* z, double* tan, int32_t* status) {
  const LawParams<double> p = make_params(prm, 1);
  const LawParams<float> pf = to_float(p);
  const Step hs = make_step(h);
  const RayConst rc = make_ray(p, h);
  for (int64_t i = 0; i < n; ++i) {
    double e[6], zi[6], s[6], zo[6], t[21];
    for (int c = 0; c < 6; ++c) e[c] = eps[6 * i + c], zi[c] = zn[6 * i + c];
    if (mode == 0) {
      status[i] = (int32_t)voxel_fp64<Law>(p, e, zi, hs, true, s, zo, t, &rc);
    } else if (mode == 1) {
      status[i] = (int32_t)voxel_fp32_fix<Law>(p, pf, e, zi, hs, true, s, zo, t, &rc);
    } else {
      float ef[6], zf[6], sf[6], zof[6], tf[21];
      for (int c = 0; c < 6; ++c) ef[c] = (float)e[c], zf[c] = (float)zi[c];
      status[i] = (int32_t)voxel_fp32<Law>(pf, ef, zf, hs, true, sf, zof, tf, &rc);
      for (int c = 0; c < 6; ++c) s[c] = sf[c], zo[c] = zof[c];
      for (int c = 0; c < 21; ++c) t[c] = tf[c];
    }
    for (int c = 0; c < 6; ++c) sig[6 * i + c] = s[c], z[6 * i + c] = zo[c];
    for (int c = 0; c < 21; ++c) tan[21 * i + c] = t[c];
  }
}

extern "C" int ray_update(int general, int mode, const double* prm, int64_t n, const double* eps, const double* zn,
                          double h, double* sig, double* z, double* tan, int32_t* status) {
  if (general) run<GeneralNorton>(mode, prm, n, eps, zn, h, sig, z, tan, status);
  else run<NortonDev>(mode, prm, n, eps, zn, h, sig, z, tan, status);
  return 0;
}

// The explicit pairs (0: ode23, 1: ode12), in the elastic deviatoric strain
// (ode_ray.cuh) or by the AD sweeps of the general state.
template <class Law, int PAIR>
static void run_ode(const double* prm, int64_t n, const double* eps_n, const double* eps, const double* zn, double h,
                    double rtol, double atol, int max_steps, double* sig, double* z, int32_t* status) {
  const LawParams<double> p = make_params(prm, 1);
  const Step hs = make_step(h);
  const Ode23Ctl ctl{rtol, atol, max_steps};
  for (int64_t i = 0; i < n; ++i) {
    double e0[6], e1[6], zi[6], s[6], zo[6];
    for (int c = 0; c < 6; ++c) e0[c] = eps_n[6 * i + c], e1[c] = eps[6 * i + c], zi[c] = zn[6 * i + c];
    status[i] = (int32_t)voxel_ode23<Law, false, PAIR>(p, e0, e1, zi, hs, ctl, s, zo, nullptr);
    for (int c = 0; c < 6; ++c) sig[6 * i + c] = s[c], z[6 * i + c] = zo[c];
  }
}

extern "C" int ray_ode(int general, int pair, const double* prm, int64_t n, const double* eps_n, const double* eps,
                       const double* zn, double h, double rtol, double atol, int max_steps, double* sig, double* z,
                       int32_t* status) {
  if (general && pair == 0) run_ode<GeneralNorton, ERK_BS23>(prm, n, eps_n, eps, zn, h, rtol, atol, max_steps, sig, z, status);
  else if (general) run_ode<GeneralNorton, ERK_HEUN12>(prm, n, eps_n, eps, zn, h, rtol, atol, max_steps, sig, z, status);
  else if (pair == 0) run_ode<NortonDev, ERK_BS23>(prm, n, eps_n, eps, zn, h, rtol, atol, max_steps, sig, z, status);
  else run_ode<NortonDev, ERK_HEUN12>(prm, n, eps_n, eps, zn, h, rtol, atol, max_steps, sig, z, status);
  return 0;
}
