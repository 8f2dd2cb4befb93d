// Launch shapes and dispatch of the real sine variant's passes (kernels in k_sine.cuh, one translation
// unit per storage type or observed-block count).
#include "k_sine.cuh"

namespace fftenkf {

// The groups with the fewest rounds over the members times waves of column pairs over the chip, and of these
// the fewest (1025^2 nodes, 4 blocks, 2 observed, N=20: one group leaves three CTAs of 128 threads on an SM and
// 512 pairs a second wave of 56 CTAs, 2 x 20 rounds; 3 groups take 4 waves of 7 rounds.  257^2, 1 block, N=40:
// 101 us with 8 groups, 63 with 14 and the rows' batched loads).  Rows up to 4096 points of the extension.
int sine_col_groups(int ny, int nx, int n_obs, int M, int N) {
  const int P = 2 * (ny - 1);
  if (P % 16 != 0 || (nx - 1) % 8 != 0 || 2 * (nx - 1) > 4096 || P > 4096 || n_obs < 1 || n_obs > kMaxObs) return 0;
  const int T = P / plan_V(P, 0);
  const int nf = n_obs * (1 + M - n_obs);
  const size_t per = (size_t)nf * P * sizeof(float) + (size_t)col_line_slots(P) * sizeof(float2);
  int best = 0;
  long long best_cost = 0;
  for (int g = 1; g <= 16 && g <= N && g * T <= sine_col_threads(n_obs); ++g) {
    if (g * per > 226 * 1024) break;
    long long per_sm = (long long)(227 * 1024 / (g * per + 1024 + 128));
    const int by_threads = sine_col_threads(n_obs) / ((g * T + 31) / 32 * 32);
    if (per_sm > by_threads) per_sm = by_threads;
    if (per_sm < 1) per_sm = 1;
    const long long slots = sm_count() * per_sm, cost = ((N + g - 1) / g) * (((nx - 1) / 2 + slots - 1) / slots);
    if (best == 0 || cost < best_cost) {
      best = g;
      best_cost = cost;
    }
  }
  return best;
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
