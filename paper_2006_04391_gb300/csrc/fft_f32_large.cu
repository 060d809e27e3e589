// Transforms of the FP32 fields for grid sizes N = R1 R2 above 64 (fft.cuh).
#include "fft.cuh"

namespace gsm {

const FftOps* fft_ops_f32_large(int N) {
  switch (N) {
    case 72: return Launch<float, 72>::ops();
    case 80: return Launch<float, 80>::ops();
    case 96: return Launch<float, 96>::ops();
    case 100: return Launch<float, 100>::ops();
    case 120: return Launch<float, 120>::ops();
    case 128: return Launch<float, 128>::ops();
    case 144: return Launch<float, 144>::ops();
    case 150: return Launch<float, 150>::ops();
    case 160: return Launch<float, 160>::ops();
    case 180: return Launch<float, 180>::ops();
    case 192: return Launch<float, 192>::ops();
    case 240: return Launch<float, 240>::ops();
    case 256: return Launch<float, 256>::ops();
    default: return nullptr;
  }
}

}  // namespace gsm
