// Transforms of the FP64 fields for grid sizes N = R1 R2 up to 64 (fft.cuh).
#include "fft.cuh"

namespace gsm {

const FftOps* fft_ops_f64_large(int N);

const FftOps* fft_ops_f64(int N) {
  switch (N) {
    case 8: return Launch<double, 8>::ops();
    case 12: return Launch<double, 12>::ops();
    case 16: return Launch<double, 16>::ops();
    case 20: return Launch<double, 20>::ops();
    case 24: return Launch<double, 24>::ops();
    case 32: return Launch<double, 32>::ops();
    case 36: return Launch<double, 36>::ops();
    case 40: return Launch<double, 40>::ops();
    case 48: return Launch<double, 48>::ops();
    case 60: return Launch<double, 60>::ops();
    case 64: return Launch<double, 64>::ops();
    default: return fft_ops_f64_large(N);
  }
}

}  // namespace gsm
