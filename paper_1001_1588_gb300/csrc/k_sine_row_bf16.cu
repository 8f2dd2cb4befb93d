// Sine variant's rows, BF16 storage.
#include "k_sine.cuh"

namespace fftenkf {
cudaError_t sine_rows_bf16(const SineParams& p, bool inverse, int units, cudaStream_t s) {
  return sine_rows_st<kBF16>(p, inverse, units, s);
}
}  // namespace fftenkf
