// Launch shapes and dispatch of the split passes (kernels in k_split.cuh, one translation unit per
// storage type or observed-block count).
#include <map>
#include <mutex>
#include <utility>

#include "k_split.cuh"

namespace fftenkf {

cudaError_t allow_smem(const void* kern, size_t smem) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> allowed;   // largest request so far: never lowered
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t& a = allowed[std::make_pair(dev, kern)];
  if (smem <= a) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) a = smem;
  return e;
}

bool split_rows_supported(int L) { return row_line_supported(L); }

// 8 rows give the transposed store (and the inverse pass's load) 64-byte segments; 4 where 8 line
// buffers would not fit in shared memory.  Every supported ny is a multiple of 8.
int split_row_tile(int L) { return L >= 3072 ? 4 : 8; }

// Groups of one column's CTA: at most split_col_threads threads, and the shared memory of two CTAs per SM
// where that leaves more than one group; then the fewest groups that need as many rounds over the members.
int split_col_groups(int ny, int n_obs, int M, int N, int threads) {
  const bool cross = M > n_obs;
  const int T = ny / plan_V(ny, split_col_sel(ny, cross));
  const int nf = n_obs + 2 * n_obs * (M - n_obs);
  const size_t per = (size_t)nf * ny * sizeof(float) + (size_t)col_line_slots(ny) * sizeof(float2);
  int g = (threads ? threads : split_col_threads(ny, n_obs, cross)) / T;
  if (g < 1) g = 1;
  if (g > 16) g = 16;
  while (g > 2 && g * per > 110 * 1024) --g;
  while (g > 1 && g * per > 226 * 1024) --g;
  if (g * per > 226 * 1024) return 0;
  if (g > N) g = N;
  const int rounds = (N + g - 1) / g;
  return (N + rounds - 1) / rounds;
}

bool split_cols_supported(int ny, int n_obs, int M) {
  switch (ny) {
#define CASE(n) case n: break;
    FFTENKF_SPLIT_COL_SIZES(CASE)
#undef CASE
    default: return false;
  }
  return n_obs >= 1 && n_obs <= kMaxObs && M >= n_obs && split_col_groups(ny, n_obs, M, 1) > 0;
}

cudaError_t launch_row_split(SplitParams p, cudaStream_t s) {
  const int fields = (p.anomalies ? p.M * p.one.N : 0) + (p.innovations ? p.one.N * p.n_obs : 0);
  const int units = p.units ? p.n_units : fields * (p.ny / split_row_tile(p.L));
  return p.storage == kBF16 ? row_split_bf16(p, units, s) : row_split_f32(p, units, s);
}

cudaError_t launch_row_inv_split(SplitParams p, cudaStream_t s) {
  const int units = p.units ? p.n_units : p.M * p.one.N * (p.ny / split_row_tile(p.L));
  return p.storage == kBF16 ? row_inv_split_bf16(p, units, s) : row_inv_split_f32(p, units, s);
}

cudaError_t launch_col_split(SplitParams p, cudaStream_t s) {
  const int units = p.units ? p.n_units : p.L + 1;
  if (!p.groups) p.groups = split_col_groups(p.ny, p.n_obs, p.M, p.one.N);
  const int nf = p.n_obs + 2 * p.n_obs * p.n_un;
  p.acc_bytes = (int)((((size_t)p.groups * nf * p.ny * sizeof(float)) + 127) & ~(size_t)127);
  if (p.drawn) {
    if (p.n_obs <= 1) return col_split_drawn_1(p, units, s);
    return p.n_obs <= 2 ? col_split_drawn_2(p, units, s) : col_split_drawn_4(p, units, s);
  }
  if (p.n_obs <= 1) return col_split_1(p, units, s);
  return p.n_obs <= 2 ? col_split_2(p, units, s) : col_split_4(p, units, s);
}

}  // namespace fftenkf
