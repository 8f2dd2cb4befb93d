// Split row passes, FP32 storage.
#include "k_split.cuh"

namespace fftenkf {
cudaError_t row_split_f32(const SplitParams& p, int units, cudaStream_t s) { return row_split_st<kF32>(p, units, s); }
cudaError_t row_inv_split_f32(const SplitParams& p, int units, cudaStream_t s) { return row_inv_split_st<kF32>(p, units, s); }
}  // namespace fftenkf
