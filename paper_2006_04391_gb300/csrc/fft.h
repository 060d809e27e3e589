// The transforms of one grid size and precision as host launchers (fft.cuh holds
// the kernels; fft_f32.cu and fft_f64.cu instantiate them).
#pragma once

#include "ms_kernels.cuh"

namespace gsm {

// Jobs of a launch: indices into the tick's job table.
struct JobList {
  uint8_t at[256];
};

// Launchers.  A batch takes n jobs of `views` (device) listed in `list`: sig ->
// sig_hat, in place on sig_hat, sig_hat -> eps_out.  With views == NULL they
// work on the one job given by pointers.
struct FftOps {
  void (*zy_fwd)(const void* views, const JobList& list, int n, const void* in, void* hat, const void* tw, cudaStream_t s);
  void (*x_fwd)(const void* views, const JobList& list, int n, void* hat, const void* tw, cudaStream_t s);
  void (*x_green)(const void* views, const JobList& list, int n, const void* tw, cudaStream_t s);
  void (*x_inv)(const void* views, const JobList& list, int n, void* hat, const void* tw, cudaStream_t s);
  void (*zy_inv)(const void* views, const JobList& list, int n, void* hat, void* out, const void* tw, cudaStream_t s);
  int green_tiles;  // partial sums the Green pass writes per job
};

// The launchers for grid size N, or NULL (then the library transform is used).
const FftOps* fft_ops_f32(int N);
const FftOps* fft_ops_f64(int N);

}  // namespace gsm
