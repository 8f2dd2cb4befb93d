// Sine variant's columns, instantiated for up to 1 observed block(s).
#include "k_sine.cuh"

namespace fftenkf {
cudaError_t sine_cols_1(const SineParams& p, cudaStream_t s) { return sine_cols_dispatch<1>(p, s); }
}  // namespace fftenkf
