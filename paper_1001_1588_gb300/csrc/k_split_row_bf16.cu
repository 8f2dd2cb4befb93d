// Split row passes, BF16 storage.
#include "k_split.cuh"

namespace fftenkf {
cudaError_t row_split_bf16(const SplitParams& p, int units, cudaStream_t s) { return row_split_st<kBF16>(p, units, s); }
cudaError_t row_inv_split_bf16(const SplitParams& p, int units, cudaStream_t s) { return row_inv_split_st<kBF16>(p, units, s); }
}  // namespace fftenkf
