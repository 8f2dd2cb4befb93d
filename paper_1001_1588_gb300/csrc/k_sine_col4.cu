// Sine variant's columns, instantiated for up to 4 observed block(s).
#include "k_sine.cuh"

namespace fftenkf {
cudaError_t sine_cols_4(const SineParams& p, cudaStream_t s) { return sine_cols_dispatch<4>(p, s); }
}  // namespace fftenkf
