// Transforms of the FP32 fields for grid sizes N = R1 R2 up to 64 (fft.cuh).
#include "fft.cuh"

namespace gsm {

const FftOps* fft_ops_f32_large(int N);

const FftOps* fft_ops_f32(int N) {
  switch (N) {
    case 8: return Launch<float, 8>::ops();
    case 12: return Launch<float, 12>::ops();
    case 16: return Launch<float, 16>::ops();
    case 20: return Launch<float, 20>::ops();
    case 24: return Launch<float, 24>::ops();
    case 32: return Launch<float, 32>::ops();
    case 36: return Launch<float, 36>::ops();
    case 40: return Launch<float, 40>::ops();
    case 48: return Launch<float, 48>::ops();
    case 60: return Launch<float, 60>::ops();
    case 64: return Launch<float, 64>::ops();
    default: return fft_ops_f32_large(N);
  }
}

}  // namespace gsm
