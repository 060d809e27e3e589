// The standalone ODE material-update kernel (AutoMat, arXiv 2006.04391,
// Sec. 4.3, Corollary 1, Sec. 4.5) and its launcher, instantiated per
// integrator in ode23.cu, ode12.cu and ode23s.cu (one translation unit each,
// compiled in parallel).  One thread per voxel; fields in HBM (or page-locked
// host memory) in structure-of-arrays layout.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "ode23.cuh"

namespace gsm {

// Launch the update of n voxels with integrator PAIR (ERK_BS23, ERK_HEUN12 or
// ROS_23S) for the law of m; pointers are device addresses; tangent may be NULL.
template <int PAIR>
void ode_launch(const Material& m, int64_t n, int64_t ld, const Step& hs, const Ode23Ctl& ctl, const double* e0,
                const double* e1, const double* zi, double* so, double* zo, double* to, int32_t* sto,
                cudaStream_t s);

// Each integrator's kernels live in their own translation unit only.
#define GSM_ODE_EXTERN(PAIR)                                                                                     \
  extern template void ode_launch<PAIR>(const Material&, int64_t, int64_t, const Step&, const Ode23Ctl&,         \
                                        const double*, const double*, const double*, double*, double*, double*, \
                                        int32_t*, cudaStream_t);
GSM_ODE_EXTERN(ERK_BS23)
GSM_ODE_EXTERN(ERK_HEUN12)
GSM_ODE_EXTERN(ROS_23S)
#undef GSM_ODE_EXTERN

#ifdef GSM_ODE_KERNEL_IMPL
namespace {


constexpr int kOdeBlock = 128;
// Finished lanes of a warp that change their voxel together.  One lane's change
// (outputs, loads, first right-hand side) costs the warp as much as 32, about
// half an attempt; waiting costs idle lanes.  Measured on 200 k voxels, n = 5:
// 3645 us with 1, 3502 with 4, 3686 with 8, 4108 with 12.
constexpr int kRefill = 4;
constexpr int kOdeGroup = 8;  // voxels: whole 32-byte sectors of every component

// Per-lane scheduling (without the tangent): a lane starts its next voxel when
// its current one has finished its substeps; the warp runs while any lane has
// work.  Voxels need different substep counts, and with one voxel per lane per
// pass the finished lanes would idle until the slowest voxel of their warp is
// done.
template <class Law, bool TAN, int PAIR>
__global__ void __launch_bounds__(kOdeBlock) ode23_kernel(int64_t n, int64_t ld, LawParams<double> p, Step hs,
                                                          Ode23Ctl ctl, const double* __restrict__ epsn,
                                                          const double* __restrict__ eps,
                                                          const double* __restrict__ zn, double* __restrict__ sig,
                                                          double* __restrict__ z, double* __restrict__ tan,
                                                          int32_t* __restrict__ status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  constexpr int NZ = stored_nz<Law>();
  OdeVoxel<Law, TAN, PAIR> v;
  // with TAN: psi's second-derivative blocks, constants of the law, once per block
  __shared__ PsiBlocks<Law::NY> blk;
  if constexpr (TAN) {
    if (threadIdx.x == 0) psi_const_blocks<Law>(p, blk);
    __syncthreads();
  }
  auto start = [&](int64_t k) {
    double e0[6], e1[6], zi[NZ];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      e0[c] = __ldg(epsn + c * ld + k);
      e1[c] = __ldg(eps + c * ld + k);
    }
#pragma unroll
    for (int c = 0; c < NZ; ++c) zi[c] = __ldg(zn + c * ld + k);
    v.init(p, e0, e1, zi, hs, TAN ? &blk : nullptr);
  };
  if constexpr (TAN) {
    // with the tangent the state lives mostly in local memory (register
    // spills); there one voxel per lane per pass, warp-voted, measured faster
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < n; base += stride) {
      const int64_t k = base + threadIdx.x;
      const bool active = k < n;
      if (active) start(k);
      else v.done = true;
      for (;;) {
        if (all_done(v.done)) break;
        if (!v.done) v.attempt(p, hs, ctl);
      }
      if (active) {
        double s[6], zo[NZ], t36[36];
        const unsigned st = v.finish(hs.h, s, zo, t36);
#pragma unroll
        for (int c = 0; c < 6; ++c) sig[c * ld + k] = s[c];
#pragma unroll
        for (int c = 0; c < NZ; ++c) z[c * ld + k] = zo[c];
#pragma unroll
        for (int c = 0; c < 36; ++c) tan[c * ld + k] = t36[c];
        if (status) status[k] = (int32_t)st;
      }
    }
    return;
  }
  // a block owns every gridDim-th group of kOdeGroup voxels; its lanes take the next
  // one of them from a shared counter, so they finish together whatever their
  // substep counts (200 k voxels: 3502 -> 3177 us against a fixed stride per lane).
  // Groups and not one range: where the flow is confined to a part of the field,
  // the blocks of that part would work alone (1 M voxels, 2 % of them flowing,
  // ode23 5772 -> 1010 us, ode12 18042 -> 2392).
  __shared__ unsigned long long taken;
  if (threadIdx.x == 0) taken = blockDim.x;
  __syncthreads();
  auto voxel = [&](int64_t k) {
    return ((k / kOdeGroup) * gridDim.x + blockIdx.x) * kOdeGroup + k % kOdeGroup;
  };
  i = voxel(threadIdx.x);
  bool have = i < n;
  if (have) start(i);
  for (;;) {
    const bool busy = have && !v.done;
    if (busy) v.attempt(p, hs, ctl);
    const unsigned idle = __ballot_sync(0xffffffffu, have && v.done);
    const bool none = !__any_sync(0xffffffffu, have && !v.done);
    if (none && !idle) break;
    if (__popc(idle) >= kRefill || none) {
      if (have && v.done) {
        double s[6], zo[NZ];
        const unsigned st = v.finish(hs.h, s, zo, nullptr);
#pragma unroll
        for (int c = 0; c < 6; ++c) sig[c * ld + i] = s[c];
#pragma unroll
        for (int c = 0; c < NZ; ++c) z[c * ld + i] = zo[c];
        if (status) status[i] = (int32_t)st;
        i = voxel((int64_t)atomicAdd(&taken, 1ull));
        have = i < n;
        if (have) start(i);
      }
    }
  }
}

template <auto Kernel> int ode_grid(int64_t n) {
  static const int per_sm = [] {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, Kernel, kOdeBlock, 0) != cudaSuccess || b <= 0) b = 1;
    return b;
  }();
  const int64_t need = (n + kOdeBlock - 1) / kOdeBlock;
  const int64_t cap = (int64_t)sm_count() * per_sm;
  return (int)(need < cap ? need : cap);
}

}  // namespace

template <int PAIR>
void ode_launch(const Material& m, int64_t n_vox, int64_t ld, const Step& hs, const Ode23Ctl& ctl, const double* e0,
                const double* e1, const double* zi, double* so, double* zo, double* to, int32_t* sto,
                cudaStream_t s) {
  auto launch = [&](auto law) {
    using Law = decltype(law);
    if (to)
      ode23_kernel<Law, true, PAIR><<<ode_grid<ode23_kernel<Law, true, PAIR>>(n_vox), kOdeBlock, 0, s>>>(
          n_vox, ld, m.p64, hs, ctl, e0, e1, zi, so, zo, to, sto);
    else
      ode23_kernel<Law, false, PAIR><<<ode_grid<ode23_kernel<Law, false, PAIR>>(n_vox), kOdeBlock, 0, s>>>(
          n_vox, ld, m.p64, hs, ctl, e0, e1, zi, so, zo, nullptr, sto);
  };
  if (m.psi_kind == GSM_PSI_ELASTIC_VP_DEV) launch(NortonDev{});
  else launch(MichelSuquet{});
}
#endif

}  // namespace gsm
