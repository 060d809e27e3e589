// Test-only host build: the status word of the scalar update (ray.cuh), with the
// start of its iteration moved off on request so that it cannot end.
#include <cstdint>

#include "../../paper_2006_04391_gb300/csrc/common.cuh"
#include "../../paper_2006_04391_gb300/csrc/voxel.cuh"

using namespace gsm;

// shift: added to log2 c0, from which the iteration's start is taken (the
// evaluations keep the right constant).
extern "C" uint32_t ray_status_word(int mode, const double* prm, const double* eps, double h, double shift,
                                    double* sig) {
  RayConst rc = make_ray(make_params(prm, 1), h);
  rc.lg_c0 += (float)shift;
  double z[6] = {0, 0, 0, 0, 0, 0}, s[6], zo[6];
  if (mode < 2) {
    double e[6];
    for (int c = 0; c < 6; ++c) e[c] = eps[c];
    const unsigned w = voxel_ray<NortonDev>(rc, e, z, true, mode == 1, s, zo, (double*)nullptr);
    for (int c = 0; c < 6; ++c) sig[c] = s[c];
    return w;
  }
  float e[6], zf[6] = {0, 0, 0, 0, 0, 0}, sf[6], zof[6];
  for (int c = 0; c < 6; ++c) e[c] = (float)eps[c];
  const unsigned w = voxel_ray<NortonDev>(rc, e, zf, true, false, sf, zof, (float*)nullptr);
  for (int c = 0; c < 6; ++c) sig[c] = sf[c];
  return w;
}
