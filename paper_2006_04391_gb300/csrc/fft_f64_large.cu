// Transforms of the FP64 fields for grid sizes N = R1 R2 above 64 (fft.cuh).
#include "fft.cuh"

namespace gsm {

const FftOps* fft_ops_f64_large(int N) {
  switch (N) {
    case 72: return Launch<double, 72>::ops();
    case 80: return Launch<double, 80>::ops();
    case 96: return Launch<double, 96>::ops();
    case 100: return Launch<double, 100>::ops();
    case 120: return Launch<double, 120>::ops();
    case 128: return Launch<double, 128>::ops();
    case 144: return Launch<double, 144>::ops();
    case 150: return Launch<double, 150>::ops();
    case 160: return Launch<double, 160>::ops();
    case 180: return Launch<double, 180>::ops();
    case 192: return Launch<double, 192>::ops();
    case 240: return Launch<double, 240>::ops();
    case 256: return Launch<double, 256>::ops();
    default: return nullptr;
  }
}

}  // namespace gsm
