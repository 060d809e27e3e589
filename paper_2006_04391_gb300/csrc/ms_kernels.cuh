// Device kernels of the Moulinec-Suquet basic scheme (AutoMat, arXiv
// 2006.04391: Sec. 1 and Sec. 3 "Material Law Evaluations").  Included by
// ms_solve.cu and (for the job views and block reductions) ms_ode.cu.
//
// Every kernel works on a batch of independent problems ("jobs") at once: a
// job's voxels (modes) are cut into chunks of a size fixed by its grid, the
// chunks of all jobs in a launch are numbered consecutively, and each block
// walks the global chunk list.  Partial sums are written per chunk and summed
// per job in chunk order, so a job's results are bit-identical whether it
// runs alone or in a batch.  A single basic-scheme solve is a batch of one.
//
// Green operator of the isotropic reference medium (lambda0, mu0), applied to
// a symmetric tau with q = tau k (homogeneous of degree 0 in k):
//   (Gamma0 : tau)_ij = (k_j q_i + k_i q_j) / (2 mu0 |k|^2)
//                       - (lambda0 + mu0) / (mu0 (lambda0 + 2 mu0)) (k.q) k_i k_j / |k|^4.
// Even N: a mode with the Nyquist index N/2 together with any other nonzero
// index has no Hermitian-consistent Gamma0; it gets Gamma0 := 0 and is left
// out of the equilibrium error.  Pure-axis Nyquist modes keep the operator.
#pragma once

#include <cufft.h>

#include "common.cuh"
#include "voxel.cuh"

namespace gsm {
namespace {

constexpr int kMaxPhases = 16;
constexpr int kMatBlock = 128;
constexpr int kGamBlock = 256;
constexpr int kVChunk = 1024;  // largest voxel chunk (8 sweeps of a material block)
constexpr int kMChunk = 2048;  // modes per chunk (8 sweeps of a gamma block)
constexpr int kMaxBatch = 256; // jobs per launch
constexpr double kTwoPi = 6.283185307179586476925286766559;

struct PhaseTable {
  int kind[kMaxPhases];  // GSM_PSI_* of each phase
  LawParams<double> p64[kMaxPhases];
  LawParams<float> p32[kMaxPhases];
};

template <class T> struct cplx;
template <> struct cplx<double> { using type = cufftDoubleComplex; };
template <> struct cplx<float> { using type = cufftComplex; };

struct double6 {
  double v[6];
};

struct Reduced {
  double e;        // equilibrium error
  double mean[6];  // <sigma>
  double res;      // sum |xi . c|^2
};

// One job of a batched launch (device copy, rebuilt by the host every tick).
struct JobView {
  RayConst ray[kMaxPhases];  // the scalar equation of each phase at this step's h (elastic: its moduli)
  int kind[kMaxPhases];      // GSM_PSI_* of each phase
  const uint8_t* phase;
  const void* eps_raw;   // [6][nvox] N^3 * strain (inverse transform's output); FP32 fields: without its mean
  const void* zn;        // [6][nvox]
  void* sig;             // [6][nvox] stress; FP32 fields: less *mean
  void* eps_out;         // [6][nvox] where the inverse transform writes the next strain
  void* z;               // [6][nvox]
  void* sig_hat;         // [6][nmodes]
  void* eps_hat;         // [6][nmodes]
  double* mat_part;      // [6][n_vch]
  double* gam_part;      // [n_mch]; fused Green pass: [7][tiles], the error and the six stress sums
  double* mean;          // [6] the mean stress of the step's last evaluation, 0 at its first (device)
  double E[6];           // mean strain
  Reduced* red;          // where the job's error and mean stress go (page-locked host memory)
  unsigned* arrived;     // blocks of the fused Green pass that are done (0 between launches), or NULL
  const PhaseTable* tab;
  int64_t nvox, nmodes;
  int64_t vchunk0, mchunk0;  // first chunk of this job in its launch
  int n_vch, n_mch;
  int N;
  int chunk;             // voxels per chunk
  int project;           // 1: the Green pass gives -Gamma0 : sig_hat alone, eps_hat is not used (adjoint)
  int n_phases;
  double h, inv_h, inv_n3, lam0, mu0;
  double inv4mu, green_b;  // constants of the fused Green pass (fft.cuh), set_reference
  // ode23 laws (Sec. 4.3): strain at t_n, the Michel-Suquet alpha, tolerances
  const double* eps_prev;  // [6][nvox]
  const double* alpha_n;   // [nvox] or NULL
  double* alpha;           // [nvox] or NULL
  double ode_rtol, ode_atol;
  int ode_max, pad2;
};

inline void set_reference(JobView& v, double lam0, double mu0) {
  v.lam0 = lam0;
  v.mu0 = mu0;
  v.inv4mu = 0.25 / mu0;
  v.green_b = 0.25 * (lam0 + mu0) / (mu0 * (lam0 + 2.0 * mu0));
}

// ------------------------------------------------------------------ helpers

// Block-wide deterministic sum of NV FP64 values (fixed shuffle order);
// thread 0 writes out[c * stride + index].  Ends with a barrier so the
// shared buffer can be reused by the next call.
template <int NV>
__device__ void block_sum_at(double (&v)[NV], double* out, int64_t stride, int64_t index) {
  __shared__ double sh[NV][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < NV; ++c)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
  if (lane == 0)
#pragma unroll
    for (int c = 0; c < NV; ++c) sh[c][warp] = v[c];
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      double s = 0.0;
      for (int w = 0; w < nw; ++w) s += sh[c][w];
      out[c * stride + index] = s;
    }
  }
  __syncthreads();
}

template <int NV> __device__ void block_sum(double (&v)[NV], double* out, int64_t stride) {
  block_sum_at<NV>(v, out, stride, blockIdx.x);
}

// Block-wide deterministic sum of six FP64 values a lane, as block_sum_at<6>: the
// lanes of a warp split the components between them as they combine (9 FP64
// additions a warp instead of 30, 18 shuffles instead of 60; an FP64 warp
// instruction holds the SM's FP64 pipe for 16 cycles).
__device__ __forceinline__ void block_sum6_at(const double (&v)[6], double* out, int64_t stride, int64_t index) {
  __shared__ double sh[6][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
  double a[4], b[2], c;  // lanes with bit 4: components 4, 5; else 0..3
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double lo = v[k], hi = k < 2 ? v[4 + k] : 0.0;
    const double r = __shfl_xor_sync(0xffffffffu, h16 ? lo : hi, 16);
    a[k] = (h16 ? hi : lo) + r;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double r = __shfl_xor_sync(0xffffffffu, h8 ? a[k] : a[2 + k], 8);
    b[k] = (h8 ? a[2 + k] : a[k]) + r;
  }
  c = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  c += __shfl_xor_sync(0xffffffffu, c, 1);
  const int comp = (h16 ? 4 : 0) + (h8 ? 2 : 0) + (h4 ? 1 : 0);
  if ((lane & 3) == 0 && comp < 6) sh[comp][warp] = c;
  __syncthreads();
  if (threadIdx.x < 6) {
    const int nw = blockDim.x >> 5;
    double s = 0.0;
    for (int w = 0; w < nw; ++w) s += sh[threadIdx.x][w];
    out[threadIdx.x * stride + index] = s;
  }
  __syncthreads();
}

// The laws of a job's phases as the material kernels read them (shared memory).
//
// FP32 fields hold what varies: the strain without its mean E (added here as a
// pair of FP32 numbers) and the stress less a uniform one (the mean of the
// evaluation before, zero at a step's first; the Green operator does not see the
// zero mode).  Their rounding, and that of the transforms, is then relative to
// the fluctuations and not to the means.
struct LawTable {
  RayConst ray[kMaxPhases];
  int kind[kMaxPhases];
  float E_hi[6], E_lo[6], sub[6];
};

// Material evaluation of voxel i.  The field precision T is also that of the
// 1/N^3 scaling and of the lane's partial stress sums (FP32 fields: no FP64
// work, a sixty-fourth of the FP32 rate on GB300; the block sums are FP64).
// All loads are issued before the phase is known: z_n of an elastic voxel is
// read for nothing, but no load waits for another.  An elastic voxel is the
// Norton voxel that does not flow (theta = 0, t = 1, z = 0): one instruction
// stream for both, where a branch cost the warps that hold both kinds both.
template <class T, int MODE>
__device__ __forceinline__ void material_voxel(int64_t i, int64_t nvox, const uint8_t* __restrict__ phase,
                                               const LawTable& law, T inv_n3,
                                               const T* __restrict__ eps_raw, const T* __restrict__ zn,
                                               T* __restrict__ sig, T* __restrict__ z, T (&acc)[6]) {
  const int ph = (int)__ldg(phase + i);
  T e[6], zi[6], s[6], zo[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) e[c] = __ldg(eps_raw + c * nvox + i);
#pragma unroll
  for (int c = 0; c < 6; ++c) zi[c] = __ldg(zn + c * nvox + i);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    if constexpr (sizeof(T) == 4) e[c] = fmaf(e[c], inv_n3, law.E_lo[c]) + law.E_hi[c];
    else e[c] *= inv_n3;
  }
  const bool vp = law.kind[ph] == GSM_PSI_ELASTIC_VP_DEV;
#pragma unroll
  for (int c = 0; c < 6; ++c) zi[c] = vp ? zi[c] : T(0);
  voxel_ray<NortonDev>(law.ray[ph], e, zi, vp, MODE == MODE_FP32_FIX, s, zo, static_cast<T*>(nullptr));
  zo[2] = vp ? zo[2] : T(0);
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    if constexpr (sizeof(T) == 4) sig[c * nvox + i] = s[c] - law.sub[c];
    else sig[c * nvox + i] = s[c];
    z[c * nvox + i] = zo[c];
    acc[c] += s[c];
  }
}

// Mode (a, b, c) of the half spectrum -> signed integer frequency.
__device__ __forceinline__ int freq(int a, int N) { return a < (N + 1) / 2 ? a : a - N; }

// Green-operator update of mode m: eps_hat -= Gamma0 : sig_hat, the updated
// eps_hat copied into sig_hat (the inverse-transform input); adds the mode's
// |k . sig_hat|^2 (Hermitian weight 1 or 2) to res.  Arithmetic in the field
// precision T, the error sum in FP64.
template <class T>
__device__ __forceinline__ void gamma_mode(int N, double inv2mu, double coef, typename cplx<T>::type* __restrict__ sig_hat,
                                           typename cplx<T>::type* __restrict__ eps_hat, int64_t nmodes, int64_t m,
                                           double& res) {
  using C = typename cplx<T>::type;
  const int Nh = N / 2 + 1;
  const bool even = (N % 2) == 0;
  const int c = (int)(m % Nh);
  const int64_t ab = m / Nh;
  const int b = (int)(ab % N);
  const int a = (int)(ab / N);
  const int kx = freq(a, N), ky = freq(b, N), kz = c;
  const int nz = (kx != 0) + (ky != 0) + (kz != 0);
  const bool nyq = even && (a == N / 2 || b == N / 2 || c == N / 2);
  const bool skip = nz == 0 || (nyq && nz >= 2);
  if (skip) {
    // Gamma0 = 0: eps_hat unchanged; the transform input gets eps_hat
#pragma unroll
    for (int q = 0; q < 6; ++q) sig_hat[q * nmodes + m] = eps_hat[q * nmodes + m];
    return;
  }
  C s[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) s[q] = sig_hat[q * nmodes + m];
  const T k1 = (T)kx, k2 = (T)ky, k3 = (T)kz;
  // q = sigma k (Voigt 11,22,33,23,13,12; tensor shears)
  T qr[3], qi[3];
  qr[0] = s[0].x * k1 + s[5].x * k2 + s[4].x * k3;
  qi[0] = s[0].y * k1 + s[5].y * k2 + s[4].y * k3;
  qr[1] = s[5].x * k1 + s[1].x * k2 + s[3].x * k3;
  qi[1] = s[5].y * k1 + s[1].y * k2 + s[3].y * k3;
  qr[2] = s[4].x * k1 + s[3].x * k2 + s[2].x * k3;
  qi[2] = s[4].y * k1 + s[3].y * k2 + s[2].y * k3;
  const double w = (c == 0 || (even && c == N / 2)) ? 1.0 : 2.0;
  res += w * ((double)(qr[0] * qr[0] + qi[0] * qi[0]) + (double)(qr[1] * qr[1] + qi[1] * qi[1]) +
              (double)(qr[2] * qr[2] + qi[2] * qi[2]));
  const T kk = k1 * k1 + k2 * k2 + k3 * k3;
  const T ik2 = T(1) / kk;
  const T a1 = (T)inv2mu * ik2;
  const T a2 = (T)coef * ik2 * ik2;
  const T kqr = k1 * qr[0] + k2 * qr[1] + k3 * qr[2];
  const T kqi = k1 * qi[0] + k2 * qi[1] + k3 * qi[2];
  const T kv[3] = {k1, k2, k3};
  const int ii[6] = {0, 1, 2, 1, 0, 0}, jj[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int i = ii[q], j = jj[q];
    const T f = q < 3 ? T(1) : T(2);  // engineering shears for strain
    const T dr = f * (a1 * (kv[j] * qr[i] + kv[i] * qr[j]) - a2 * kqr * kv[i] * kv[j]);
    const T di = f * (a1 * (kv[j] * qi[i] + kv[i] * qi[j]) - a2 * kqi * kv[i] * kv[j]);
    C e = eps_hat[q * nmodes + m];
    e.x -= dr;
    e.y -= di;
    eps_hat[q * nmodes + m] = e;
    sig_hat[q * nmodes + m] = e;
  }
}

// The Green-operator update of one FP32 mode on registers: s = sig_hat, e =
// eps_hat (in/out, the updated strain spectrum); (a, b, c) its half-spectrum
// index.  Same arithmetic as gamma_mode.
__device__ __forceinline__ void gamma_mode_f32_regs(int N, int a, int b, int c, float inv2mu, float coef,
                                                    const float2 (&s)[6], float2 (&e)[6], double& res) {
  const int Nh = N / 2 + 1;
  (void)Nh;
  const bool even = (N % 2) == 0;
  const int kx = freq(a, N), ky = freq(b, N), kz = c;
  const int nz = (kx != 0) + (ky != 0) + (kz != 0);
  const bool nyq = even && (a == N / 2 || b == N / 2 || c == N / 2);
  if (nz == 0 || (nyq && nz >= 2)) return;  // Gamma0 = 0: eps_hat unchanged
  const float k1 = (float)kx, k2 = (float)ky, k3 = (float)kz;
  float qr[3], qi[3];
  qr[0] = s[0].x * k1 + s[5].x * k2 + s[4].x * k3;
  qi[0] = s[0].y * k1 + s[5].y * k2 + s[4].y * k3;
  qr[1] = s[5].x * k1 + s[1].x * k2 + s[3].x * k3;
  qi[1] = s[5].y * k1 + s[1].y * k2 + s[3].y * k3;
  qr[2] = s[4].x * k1 + s[3].x * k2 + s[2].x * k3;
  qi[2] = s[4].y * k1 + s[3].y * k2 + s[2].y * k3;
  const double w = (c == 0 || (even && c == N / 2)) ? 1.0 : 2.0;
  res += w * ((double)(qr[0] * qr[0] + qi[0] * qi[0]) + (double)(qr[1] * qr[1] + qi[1] * qi[1]) +
              (double)(qr[2] * qr[2] + qi[2] * qi[2]));
  const float kk = k1 * k1 + k2 * k2 + k3 * k3;
  const float ik2 = 1.0f / kk;
  const float a1 = inv2mu * ik2;
  const float a2 = coef * ik2 * ik2;
  const float kqr = k1 * qr[0] + k2 * qr[1] + k3 * qr[2];
  const float kqi = k1 * qi[0] + k2 * qi[1] + k3 * qi[2];
  const float kv[3] = {k1, k2, k3};
  const int ii[6] = {0, 1, 2, 1, 0, 0}, jj[6] = {0, 1, 2, 2, 2, 1};
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int i = ii[q], j = jj[q];
    const float f = q < 3 ? 1.0f : 2.0f;
    e[q].x -= f * (a1 * (kv[j] * qr[i] + kv[i] * qr[j]) - a2 * kqr * kv[i] * kv[j]);
    e[q].y -= f * (a1 * (kv[j] * qi[i] + kv[i] * qi[j]) - a2 * kqi * kv[i] * kv[j]);
  }
}

// Two consecutive FP32 modes m0 (even) and m0 + 1 with 16-byte loads and
// stores (nmodes even, so every component's base is 16-byte aligned); the
// index (a, b, c) of m0 by 32-bit division (nmodes < 2^31), that of m0 + 1 by
// a carry.
__device__ __forceinline__ void gamma_pair_f32(int N, float inv2mu, float coef, float4* __restrict__ sig_hat,
                                               float4* __restrict__ eps_hat, int64_t nmodes, unsigned m0,
                                               double& res) {
  const unsigned Nh = (unsigned)(N / 2 + 1);
  const size_t st = (size_t)nmodes / 2, p = m0 / 2;
  float4 S[6], E[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) S[q] = sig_hat[q * st + p];
#pragma unroll
  for (int q = 0; q < 6; ++q) E[q] = eps_hat[q * st + p];
  const unsigned ab = m0 / Nh;
  int c = (int)(m0 - ab * Nh);
  int a = (int)(ab / (unsigned)N);
  int b = (int)(ab - (unsigned)a * (unsigned)N);
  float2 s0[6], e0[6], s1[6], e1[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    s0[q] = make_float2(S[q].x, S[q].y);
    s1[q] = make_float2(S[q].z, S[q].w);
    e0[q] = make_float2(E[q].x, E[q].y);
    e1[q] = make_float2(E[q].z, E[q].w);
  }
  gamma_mode_f32_regs(N, a, b, c, inv2mu, coef, s0, e0, res);
  if (++c == (int)Nh) {
    c = 0;
    if (++b == N) {
      b = 0;
      ++a;
    }
  }
  gamma_mode_f32_regs(N, a, b, c, inv2mu, coef, s1, e1, res);
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const float4 o = make_float4(e0[q].x, e0[q].y, e1[q].x, e1[q].y);
    eps_hat[q * st + p] = o;
    sig_hat[q * st + p] = o;
  }
}

// ------------------------------------------------------------------ kernels

// Single-problem material evaluation (grid-stride over voxels; one partial
// sum per block).  Used by the allocation-free entry point.
template <class T, int MODE>
__global__ void __launch_bounds__(kMatBlock) ms_material_kernel(int64_t nvox, const uint8_t* __restrict__ phase,
                                                                PhaseTable tab, double h, double inv_n3,
                                                                const T* __restrict__ eps_raw,
                                                                const T* __restrict__ zn, T* __restrict__ sig,
                                                                T* __restrict__ z, double* __restrict__ partials) {
  __shared__ LawTable law;
  if (threadIdx.x < kMaxPhases) {
    law.kind[threadIdx.x] = tab.kind[threadIdx.x];
    law.ray[threadIdx.x] = make_ray(tab.p64[threadIdx.x], h);
  }
  __syncthreads();
  T acc[6] = {0, 0, 0, 0, 0, 0};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvox; i += stride)
    material_voxel<T, MODE>(i, nvox, phase, law, (T)inv_n3, eps_raw, zn, sig, z, acc);
  double accd[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) accd[c] = (double)acc[c];
  block_sum6_at(accd, partials, gridDim.x, blockIdx.x);
}

// Index of the job owning global chunk c (starts ascending, starts[0] = 0).
__device__ __forceinline__ int owner(const int64_t* starts, int n, int64_t c) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (starts[mid] <= c) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Batched material evaluation: all jobs of the launch, chunk by chunk.
// (FP32: 40 registers, twelve blocks an SM, 20 bytes spilled; the kernel waits on
// loads: 256^3 385 us at nine blocks, 306 at ten, 294 at twelve, 346 at sixteen)
template <class T, int MODE>
__global__ void __launch_bounds__(kMatBlock, MODE == MODE_FP32 ? 12 : 1) ms_material_batch_kernel(const JobView* __restrict__ views, int n_jobs,
                                                                      int64_t total_chunks) {
  __shared__ int64_t starts[kMaxBatch];
  __shared__ LawTable law;
  for (int j = threadIdx.x; j < n_jobs; j += blockDim.x) starts[j] = views[j].vchunk0;
  __syncthreads();
  int held = -1;  // the job whose laws are in shared memory
  for (int64_t gc = blockIdx.x; gc < total_chunks; gc += gridDim.x) {
    const int job = n_jobs > 1 ? owner(starts, n_jobs, gc) : 0;
    const JobView& v = views[job];
    if (job != held) {  // (a block sum's barrier lies between the last use and this)
      static_assert(sizeof(RayConst) % 4 == 0, "");
      const int* src = reinterpret_cast<const int*>(v.ray);
      int* dst = reinterpret_cast<int*>(law.ray);
      for (int k = threadIdx.x; k < v.n_phases * (int)(sizeof(RayConst) / 4); k += blockDim.x) dst[k] = src[k];
      if (threadIdx.x < kMaxPhases) law.kind[threadIdx.x] = v.kind[threadIdx.x];
      if (sizeof(T) == 4 && threadIdx.x < 6) {
        const double E = v.E[threadIdx.x];
        law.E_hi[threadIdx.x] = (float)E;
        law.E_lo[threadIdx.x] = (float)(E - (double)(float)E);
        law.sub[threadIdx.x] = (float)v.mean[threadIdx.x];
      }
      held = job;
      __syncthreads();
    }
    const int64_t lc = gc - v.vchunk0;
    T acc[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll 1
    for (int o = threadIdx.x; o < v.chunk; o += kMatBlock) {
      const int64_t i = lc * v.chunk + o;
      if (i < v.nvox)
        material_voxel<T, MODE>(i, v.nvox, v.phase, law, (T)v.inv_n3, static_cast<const T*>(v.eps_raw),
                                static_cast<const T*>(v.zn), static_cast<T*>(v.sig), static_cast<T*>(v.z), acc);
    }
    double accd[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) accd[c] = (double)acc[c];
    block_sum6_at(accd, v.mat_part, v.n_vch, lc);
  }
}

// Batched Green-operator update and error partial sums.
template <class T>
__global__ void __launch_bounds__(kGamBlock) ms_gamma_batch_kernel(const JobView* __restrict__ views, int n_jobs,
                                                                   int64_t total_chunks) {
  __shared__ int64_t starts[kMaxBatch];
  for (int j = threadIdx.x; j < n_jobs; j += blockDim.x) starts[j] = views[j].mchunk0;
  __syncthreads();
  for (int64_t gc = blockIdx.x; gc < total_chunks; gc += gridDim.x) {
    const JobView& v = views[owner(starts, n_jobs, gc)];
    const int64_t lc = gc - v.mchunk0;
    const double inv2mu = 1.0 / (2.0 * v.mu0);
    const double coef = (v.lam0 + v.mu0) / (v.mu0 * (v.lam0 + 2.0 * v.mu0));
    double res[1] = {0.0};
    if (sizeof(T) == 4 && v.nmodes % 2 == 0) {
      // FP32 fields: pairs of modes per thread, 16-byte accesses
#pragma unroll 1
      for (int sweep = 0; sweep < kMChunk / (2 * kGamBlock); ++sweep) {
        const int64_t m = lc * kMChunk + sweep * 2 * kGamBlock + 2 * threadIdx.x;
        if (m < v.nmodes)
          gamma_pair_f32(v.N, (float)inv2mu, (float)coef, static_cast<float4*>(v.sig_hat),
                         static_cast<float4*>(v.eps_hat), v.nmodes, (unsigned)m, res[0]);
      }
    } else {
#pragma unroll 1
      for (int sweep = 0; sweep < kMChunk / kGamBlock; ++sweep) {
        const int64_t m = lc * kMChunk + sweep * kGamBlock + threadIdx.x;
        if (m < v.nmodes)
          gamma_mode<T>(v.N, inv2mu, coef, static_cast<typename cplx<T>::type*>(v.sig_hat),
                        static_cast<typename cplx<T>::type*>(v.eps_hat), v.nmodes, m, res[0]);
      }
    }
    block_sum_at<1>(res, v.gam_part, v.n_mch, lc);
  }
}

// Final sums of one problem's partials (six stress components, the error) by
// one block: each thread takes every blockDim-th partial of all seven, with
// their loads in flight together, then the block's fixed shuffle tree.  The
// order depends only on the partial counts and the block size (never on other
// problems in a batch).  The 256^3 sums took 58 us with one warp a sum.
constexpr int kFinBlock = 512;
__device__ void finalize_sums(const double* __restrict__ mat_part, int n_mat, const double* __restrict__ gam_part,
                              int n_gam, double inv_n3, double floor_, Reduced* __restrict__ out,
                              double* __restrict__ mean = nullptr) {
  __shared__ double sum[7];
  double a[7] = {0, 0, 0, 0, 0, 0, 0};
#pragma unroll 4
  for (int b = threadIdx.x; b < n_mat; b += blockDim.x)
#pragma unroll
    for (int c = 0; c < 6; ++c) a[c] += __ldcg(mat_part + (int64_t)c * n_mat + b);
#pragma unroll 4
  for (int b = threadIdx.x; b < n_gam; b += blockDim.x) a[6] += __ldcg(gam_part + b);
  block_sum_at<7>(a, sum, 1, 0);
  if (threadIdx.x == 0) {
    double m[6];
    for (int c = 0; c < 6; ++c) m[c] = sum[c] * inv_n3;
    // sum |xi . c|^2 with xi = 2 pi k and c = sigma^ / N^3
    const double num = sqrt(sum[6]) * kTwoPi * inv_n3;
    const double fro = sqrt(m[0] * m[0] + m[1] * m[1] + m[2] * m[2] + 2.0 * (m[3] * m[3] + m[4] * m[4] + m[5] * m[5]));
    out->e = num / fmax(fro, floor_);
    for (int c = 0; c < 6; ++c) out->mean[c] = m[c];
    if (mean)
      for (int c = 0; c < 6; ++c) mean[c] = m[c];
    out->res = sum[6];
  }
}

// Fixed-order final sums of one problem's partials (single-problem path).
__global__ void ms_finalize_kernel(const double* __restrict__ mat_part, int n_mat, const double* __restrict__ gam_part,
                                   int n_gam, double inv_n3, double floor_, Reduced* __restrict__ out) {
  finalize_sums(mat_part, n_mat, gam_part, n_gam, inv_n3, floor_, out);
}

// One block per job.
__global__ void ms_finalize_batch_kernel(const JobView* __restrict__ views) {
  const JobView& v = views[blockIdx.x];
  finalize_sums(v.mat_part, v.n_vch, v.gam_part, v.n_mch, v.inv_n3, v.mu0 * 1e-6, v.red, v.mean);
}

// Mean mode of the strain spectrum and of the inverse-transform input:
// m = N^3 E (mixed boundary conditions move E during a load step).  One warp.
template <class T>
__global__ void ms_set_mean_kernel(typename cplx<T>::type* __restrict__ eps_hat, typename cplx<T>::type* __restrict__ sig_hat,
                                   int64_t nmodes, double6 m) {
  const int q = threadIdx.x;
  if (q < 6) {
    typename cplx<T>::type v;
    v.x = (T)m.v[q];
    v.y = T(0);
    eps_hat[q * nmodes] = v;
    sig_hat[q * nmodes] = v;
  }
}

// The same for a spectrum whose inverse x pass is done (fft.cuh): the mean mode
// is there a constant along x, which moves by d = N^3 dE; eps_hat's is set to m.
template <class T>
__global__ void ms_move_mean_kernel(typename cplx<T>::type* __restrict__ eps_hat, typename cplx<T>::type* __restrict__ sig_hat,
                                    int N, double6 m, double6 d) {
  const int Nh = N / 2 + 1;
  const int64_t nmodes = (int64_t)N * N * Nh;
  for (int i = threadIdx.x; i < 6 * N; i += blockDim.x) {
    const int q = i / N, x = i % N;
    sig_hat[q * nmodes + (int64_t)x * N * Nh].x += (T)d.v[q];
    if (x == 0) {
      typename cplx<T>::type v;
      v.x = (T)m.v[q];
      v.y = T(0);
      eps_hat[q * nmodes] = v;
    }
  }
}

// Reference medium from tangents (Sec. 3: adjusted per load step to the
// current tangential stiffness): the law with tangent at the predicted strain
// eps_raw / N^3 + dE and z_n; per voxel the isotropic measures
// 3k = J::C = (1/3) sum_{i,j<3} C_ij and 10 mu = tr_Mandel C - 3k; per block
// their min and max -> part[q * gridDim.x + block], q = kmin, kmax, mumin, mumax.
template <int MODE>
__global__ void __launch_bounds__(kMatBlock) ms_reference_kernel(int64_t nvox, const uint8_t* __restrict__ phase,
                                                                 const PhaseTable* __restrict__ tab, double h,
                                                                 const double* __restrict__ eps_raw,
                                                                 const double* __restrict__ zn, double inv_n3,
                                                                 double d0, double d1, double d2, double d3, double d4,
                                                                 double d5, double* __restrict__ part) {
  const double d[6] = {d0, d1, d2, d3, d4, d5};
  double r[4] = {1e300, -1e300, 1e300, -1e300};
  __shared__ RayConst ray[kMaxPhases];
  if (threadIdx.x < kMaxPhases && tab->kind[threadIdx.x] == GSM_PSI_ELASTIC_VP_DEV)
    ray[threadIdx.x] = make_ray(tab->p64[threadIdx.x], h);
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < nvox; base += stride) {
    const int64_t i = base + threadIdx.x;
    const bool in = i < nvox;
    const int ph = in ? (int)phase[i] : 0;
    const bool vp = in && tab->kind[ph] == GSM_PSI_ELASTIC_VP_DEV;
    double e[6], zi[6], s[6], zo[6], t[21];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      e[c] = in ? fma(eps_raw[c * nvox + i], inv_n3, d[c]) : 0.0;
      zi[c] = vp ? zn[c * nvox + i] : 0.0;
    }
    if (vp) voxel_ray<NortonDev>(ray[ph], e, zi, true, MODE == MODE_FP32_FIX, s, zo, t);
    else if (in) voxel_elastic<double>(tab->p64[ph], e, s, t);
    if (in) {
      // packed upper triangle: C11 0, C12 1, C13 2, C22 6, C23 7, C33 11, C44 15, C55 18, C66 20
      const double tk = (t[0] + t[6] + t[11] + 2.0 * (t[1] + t[2] + t[7])) * (1.0 / 3.0);
      const double tr = t[0] + t[6] + t[11] + 2.0 * (t[15] + t[18] + t[20]);
      const double k = tk * (1.0 / 3.0), mu = (tr - tk) * 0.1;
      r[0] = fmin(r[0], k);
      r[1] = fmax(r[1], k);
      r[2] = fmin(r[2], mu);
      r[3] = fmax(r[3], mu);
    }
  }
  __shared__ double sh[4][kMatBlock / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    double v = r[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const double o = __shfl_down_sync(0xffffffffu, v, off);
      v = (q & 1) ? fmax(v, o) : fmin(v, o);
    }
    if (lane == 0) sh[q][w] = v;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    const int q = threadIdx.x;
    double v = sh[q][0];
    for (int k = 1; k < kMatBlock / 32; ++k) v = (q & 1) ? fmax(v, sh[q][k]) : fmin(v, sh[q][k]);
    part[q * gridDim.x + blockIdx.x] = v;
  }
}

// eps_raw += N^3 dE (uniform macro-strain increment at a step start).
template <class T>
__global__ void ms_add_uniform_kernel(int64_t nvox, T* __restrict__ eps_raw, double d0, double d1, double d2,
                                      double d3, double d4, double d5) {
  const double d[6] = {d0, d1, d2, d3, d4, d5};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvox; i += stride)
#pragma unroll
    for (int c = 0; c < 6; ++c) eps_raw[c * nvox + i] = (T)((double)eps_raw[c * nvox + i] + d[c]);
}

// dst = src + off, one offset a component, with conversion (the FP32 strain
// without its mean and back).
template <class S, class D>
__global__ void ms_offset_convert_kernel(int64_t nvox, const S* __restrict__ src, D* __restrict__ dst, double6 off) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvox; i += stride)
#pragma unroll
    for (int c = 0; c < 6; ++c) dst[c * nvox + i] = (D)((double)src[c * nvox + i] + off.v[c]);
}

// eps_hat = R2C(eps_raw) / N^3 with the mean mode set to N^3 E exactly.
template <class T>
__global__ void ms_spectrum_init_kernel(int64_t nmodes, const typename cplx<T>::type* __restrict__ raw_hat,
                                        typename cplx<T>::type* __restrict__ eps_hat, double inv_n3, double n3,
                                        double E0, double E1, double E2, double E3, double E4, double E5) {
  const double E[6] = {E0, E1, E2, E3, E4, E5};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; m < nmodes; m += stride) {
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      typename cplx<T>::type v = raw_hat[q * nmodes + m];
      if (m == 0) {
        v.x = (T)(n3 * E[q]);
        v.y = T(0);
      } else {
        v.x = (T)((double)v.x * inv_n3);
        v.y = (T)((double)v.y * inv_n3);
      }
      eps_hat[q * nmodes + m] = v;
    }
  }
}

// Precision conversion / scaling: dst = src * scale.
template <class S, class D>
__global__ void ms_convert_kernel(int64_t n, const S* __restrict__ src, D* __restrict__ dst, double scale) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    dst[i] = (D)((double)src[i] * scale);
}

}  // namespace
}  // namespace gsm
