// Launch shapes and dispatch of the real sine variant's passes (kernels in k_sine.cuh, one translation
// unit per storage type or observed-block count).
#include "k_sine.cuh"

namespace fftenkf {

// At most 256 threads and the shared memory of two CTAs per SM where that leaves more than one group;
// rows up to 4096 points of the extension.
int sine_col_groups(int ny, int nx, int n_obs, int M, int N) {
  const int P = 2 * (ny - 1);
  if (P % 16 != 0 || (nx - 1) % 8 != 0 || 2 * (nx - 1) > 4096 || P > 4096 || n_obs < 1 || n_obs > kMaxObs) return 0;
  const int T = P / plan_V(P, 0);
  const int nf = n_obs * (1 + M - n_obs);
  const size_t per = (size_t)nf * 2 * (ny - 1) * sizeof(float) + (size_t)col_line_slots(P) * sizeof(float2);
  int g = 256 / T;
  if (g > 16) g = 16;
  while (g > 1 && g * per > 110 * 1024) --g;
  if (g * per > 226 * 1024) return 0;
  if (g > N) g = N;
  const int rounds = (N + g - 1) / g;
  return (N + rounds - 1) / rounds;
}

cudaError_t launch_sine_rows(const SineParams& p, cudaStream_t s) {
  const int fields = (p.anomalies ? p.M * p.N : 0) + (p.innovations ? p.N * p.n_obs : 0);
  const int units = fields * ((p.ny - 1) / (2 * sine_tile_lines(2 * (p.nx - 1))));
  return p.storage == kBF16 ? sine_rows_bf16(p, false, units, s) : sine_rows_f32(p, false, units, s);
}

cudaError_t launch_sine_rows_inv(const SineParams& p, cudaStream_t s) {
  const int units = p.M * p.N * ((p.ny - 1) / (2 * sine_tile_lines(2 * (p.nx - 1))));
  return p.storage == kBF16 ? sine_rows_bf16(p, true, units, s) : sine_rows_f32(p, true, units, s);
}

cudaError_t launch_sine_cols(SineParams p, cudaStream_t s) {
  p.groups = sine_col_groups(p.ny, p.nx, p.n_obs, p.M, p.N);
  if (!p.groups) return cudaErrorInvalidConfiguration;
  const int nf = p.n_obs * (1 + p.M - p.n_obs);
  p.acc_bytes = (int)(((size_t)p.groups * nf * 2 * (p.ny - 1) * sizeof(float) + 127) & ~(size_t)127);
  if (p.n_obs <= 1) return sine_cols_1(p, s);
  return p.n_obs <= 2 ? sine_cols_2(p, s) : sine_cols_4(p, s);
}

}  // namespace fftenkf
