// Split column pass with drawn perturbations, instantiated for up to 1 observed block(s).
#include "k_split.cuh"

namespace fftenkf {
cudaError_t col_split_drawn_1(const SplitParams& p, int units, cudaStream_t s) {
  return col_split_dispatch<1, true>(p, units, s);
}
}  // namespace fftenkf
