// Split column pass with drawn perturbations, instantiated for up to 4 observed block(s).
#include "k_split.cuh"

namespace fftenkf {
cudaError_t col_split_drawn_4(const SplitParams& p, int units, cudaStream_t s) {
  return col_split_dispatch<4, true>(p, units, s);
}
}  // namespace fftenkf
