// Sine variant's rows, FP32 storage.
#include "k_sine.cuh"

namespace fftenkf {
cudaError_t sine_rows_f32(const SineParams& p, bool inverse, int units, cudaStream_t s) {
  return sine_rows_st<kF32>(p, inverse, units, s);
}
}  // namespace fftenkf
