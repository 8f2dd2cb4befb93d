// Sine variant's columns, instantiated for up to 2 observed block(s).
#include "k_sine.cuh"

namespace fftenkf {
cudaError_t sine_cols_2(const SineParams& p, cudaStream_t s) { return sine_cols_dispatch<2>(p, s); }
}  // namespace fftenkf
