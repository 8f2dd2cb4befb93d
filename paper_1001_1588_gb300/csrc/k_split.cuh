// The analysis passes split into independent CTAs, for grids and ensembles that do not fill the GPU
// with the pipelined passes of k_rows.cuh, k_cols.cuh and k_colf.cuh (one persistent CTA per SM, members
// taken in turn).  Every CTA does one unit and leaves; several CTAs per SM hide each other's latency.
//
//   row_split      one tile of R rows of one transform: the anomaly rows F(u_k - u_0) (k >= 1), the
//                  scaled sum of those differences in the place of k = 0 (as row_anom_kernel), and the
//                  innovation rows F((d - u_k) + e_k), all in one launch
//   col_split      one wavenumber column: members over the CTA's thread groups, each group's sums of
//                  eq. (dii) and eq. (cov-multi-spectral) in shared memory, added over the groups and
//                  turned into the gains of eq. (spectral-multi-enkf) there, then the update with the
//                  members over the groups again
//   row_inv_split  one tile of R rows of one field: inverse rows, added to the forecast
//
// A launch covers one analysis, or the analyses of one shape of a batch (a table of items and a list
// of units).
#pragma once
#include "common.cuh"
#include "dd.cuh"
#include "k_cols.cuh"
#include "k_rows.cuh"
#include "launch.cuh"
#include "perturb.cuh"

namespace fftenkf {

// the item and the unit of this CTA
__device__ __forceinline__ const SplitItem& split_item(const SplitParams& p, int& u) {
  if (!p.units) {
    u = blockIdx.x;
    return p.one;
  }
  const uint2 w = __ldg(p.units + blockIdx.x);
  u = (int)w.y;
  return p.table[w.x];
}

// ----------------------------------------------------------------- forward rows
// unit = tile * n_fields + f; the fields of one tile are consecutive, so their CTAs run together and
// share the pivot and data rows through L2.  f < M: the sum field of block f; then the members 1..N-1
// of every block; then the innovations (k n_obs + i).
template <int L, int V, int ST>
__global__ void __launch_bounds__(256, 2) row_split_kernel(const __grid_constant__ SplitParams p) {
  constexpr int T = L / V;
  constexpr int pitch = row_pitch(L);
  constexpr int es = (ST == kBF16) ? 2 : 4;
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* lines = reinterpret_cast<float2*>(smraw);
  stream_order_wait();
  int u;
  const SplitItem& it = split_item(p, u);
  const int LPC = blockDim.x / T;
  const int g = threadIdx.x / T, t = threadIdx.x - g * T;
  const int N = it.N, R = p.R, nx = p.nx;
  const int n_anom = p.anomalies ? p.M * N : 0;
  const int n_fields = n_anom + (p.innovations ? N * p.n_obs : 0);
  const int tile = u / n_fields;
  int f = u - tile * n_fields;
  const int y0 = tile * R;
  const size_t G = (size_t)p.ny * nx;
  const char* ens = reinterpret_cast<const char*>(it.ens);
  float2* out;
  for (int r = 0; r < R; r += LPC) {
    const size_t row = (size_t)(y0 + r + g) * nx;
    float2 v[V];
    if (f < n_anom) {
      const int j = f < p.M ? f : (f - p.M) / (N - 1);
      const int k = f < p.M ? 0 : 1 + (f - p.M) - j * (N - 1);
      const char* piv = ens + ((size_t)j * N * G + row) * es;   // member 0
      out = it.A + ((size_t)j * N + k) * (size_t)L * p.ny;
      float2 sv[V];
#pragma unroll
      for (int m = 0; m < V; ++m) sv[m] = load2<ST>(piv, 2 * (size_t)(t + T * m));
      if (k > 0) {
        const char* src = piv + (size_t)k * G * es;
#pragma unroll
        for (int m = 0; m < V; ++m) {
          const float2 a = load2<ST>(src, 2 * (size_t)(t + T * m));
          v[m] = make_float2(a.x - sv[m].x, a.y - sv[m].y);
        }
      } else {   // (1/sqrt N) sum_k (u_k - u_0), in member order
#pragma unroll
        for (int m = 0; m < V; ++m) v[m] = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int q = 1; q < N; ++q) {
          const char* src = piv + (size_t)q * G * es;
#pragma unroll
          for (int m = 0; m < V; ++m) {
            const float2 a = load2<ST>(src, 2 * (size_t)(t + T * m));
            v[m] = make_float2(v[m].x + (a.x - sv[m].x), v[m].y + (a.y - sv[m].y));
          }
        }
        const float s = it.inv_sqrt_N;
#pragma unroll
        for (int m = 0; m < V; ++m) v[m] = make_float2(v[m].x * s, v[m].y * s);
      }
    } else {
      const int w = f - n_anom, k = w / p.n_obs, i = w - k * p.n_obs;
      int blk = i;
#pragma unroll
      for (int q = 0; q < kMaxObs; ++q)   // constant indices: the parameter array stays in the constant bank
        if (q == i) blk = p.obs[q];
      const char* src = ens + (((size_t)blk * N + k) * G + row) * es;
      const float* d = it.data + (size_t)i * G + row;
      out = it.W + (size_t)w * (size_t)L * p.ny;
      float2 e2[V];
      if (p.innovations == kInnovation) {   // requested with the others: one wait for all three
        const char* e = reinterpret_cast<const char*>(it.pert) + ((size_t)w * G + row) * es;
#pragma unroll
        for (int m = 0; m < V; ++m) e2[m] = load2<ST>(e, 2 * (size_t)(t + T * m));
      } else {
#pragma unroll
        for (int m = 0; m < V; ++m) e2[m] = make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int m = 0; m < V; ++m) {
        const float2 a = load2<ST>(src, 2 * (size_t)(t + T * m));
        const float2 dd = reinterpret_cast<const float2*>(d)[t + T * m];
        v[m] = make_float2((dd.x - a.x) + e2[m].x, (dd.y - a.y) + e2[m].y);   // d - u first: exact when they are close
      }
    }
    float2* line = lines + (r + g) * pitch;
    fft_line<L, V, false>(v, line, t, p.twL, line_bar<T>(g));
#pragma unroll
    for (int m = 0; m < V; ++m) line[pidx(t + T * m)] = v[m];
  }
  __syncthreads();
  row_twist_store<L>(lines, out, R, p.ny, y0, p.twX);
}

// ----------------------------------------------------------------- inverse rows
// unit = tile * (M N) + field.  The twist reads both columns c, L - c of a pair of rows from global
// memory (R consecutive rows of a column are one 8 R-byte segment) and stages the rows in their line
// buffers, which then serve as exchange buffers.
template <int L, int V, int ST>
__global__ void __launch_bounds__(256, 2) row_inv_split_kernel(const __grid_constant__ SplitParams p) {
  constexpr int T = L / V;
  constexpr int pitch = row_pitch(L);
  constexpr int es = (ST == kBF16) ? 2 : 4;
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* lines = reinterpret_cast<float2*>(smraw);
  stream_order_wait();
  int u;
  const SplitItem& it = split_item(p, u);
  const int LPC = blockDim.x / T;
  const int g = threadIdx.x / T, t = threadIdx.x - g * T;
  const int nf = p.M * it.N, R = p.R, nx = p.nx;
  const int tile = u / nf, f = u - tile * nf;
  const int y0 = tile * R;
  const size_t G = (size_t)p.ny * nx;
  const int RP = R >> 1;
  const int rp = threadIdx.x % RP;
  const float2* in = it.A + (size_t)f * L * p.ny + y0 + 2 * rp;
  float2* l0 = lines + (2 * rp) * pitch;
  float2* l1 = l0 + pitch;
  // from X[c], X[L-c] of a row: z[c] = A + i B conj(W^c), z[L-c] = conj(A - i B conj(W^c)),
  // A = X[c] + conj X[L-c], B = X[c] - conj X[L-c]
  // Both columns of a pair, and of four pairs, are requested before the first is used, as are the three fields
  // of an innovation above (256 mixed analyses 7.97 -> 7.85 ms, one block 1024^2 with the network 124.6 -> 122.6 us).
#pragma unroll 4
  for (int c = threadIdx.x / RP; c <= L / 2; c += blockDim.x / RP) {
    const float4 x = *reinterpret_cast<const float4*>(in + (size_t)c * p.ny);
    const float4 y = *reinterpret_cast<const float4*>(in + (size_t)(c == 0 ? 0 : L - c) * p.ny);
    if (c == 0) {   // packed X[0] + i X[L]
      l0[pidx(0)] = make_float2(x.x + x.y, x.x - x.y);
      l1[pidx(0)] = make_float2(x.z + x.w, x.z - x.w);
      continue;
    }
    const float2 w = __ldg(p.twX + c);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 X = h ? make_float2(x.z, x.w) : make_float2(x.x, x.y);
      const float2 Y = h ? make_float2(y.z, y.w) : make_float2(y.x, y.y);
      const float2 A = make_float2(X.x + Y.x, X.y - Y.y);
      const float2 B = cmulc(make_float2(X.x - Y.x, X.y + Y.y), w);
      float2* line = h ? l1 : l0;
      line[pidx(c)] = make_float2(A.x - B.y, A.y + B.x);
      if (c != L - c) line[pidx(L - c)] = make_float2(A.x + B.y, B.x - A.y);
    }
  }
  __syncthreads();
  for (int r = 0; r < R; r += LPC) {
    float2* line = lines + (r + g) * pitch;
    char* urow = reinterpret_cast<char*>(it.ens) + ((size_t)f * G + (size_t)(y0 + r + g) * nx) * es;
    float2 v[V], a[V];
#pragma unroll
    for (int m = 0; m < V; ++m) a[m] = load2<ST>(urow, 2 * (size_t)(t + T * m));
#pragma unroll
    for (int m = 0; m < V; ++m) v[m] = line[pidx(t + T * m)];
    line_sync<T>(line_bar<T>(g));   // the row is read before the FFT reuses its buffer
    fft_line<L, V, true, false>(v, line, t, p.twL, line_bar<T>(g));
#pragma unroll
    for (int m = 0; m < V; ++m)
      store2<ST>(urow, 2 * (size_t)(t + T * m), make_float2(a[m].x + v[m].x, a[m].y + v[m].y));
  }
}

// ----------------------------------------------------------------- columns
// Sums over the groups -> gains (in the first group's region), or covariance tables when the spectrum
// alone is wanted, or gains of a caller's spectrum; one thread per wavenumber.  The denominator is
// formed in float pairs (dd.cuh) and rounded once, the quotients are FP32, or FP64 where the rounded
// denominator is below FLT_MIN (0 where it is exactly 0); with a caller's spectrum the quotients are
// formed in pairs too.  False if a value is not finite.
template <int NY>
__device__ __forceinline__ bool split_gains(const SplitParams& p, const SplitItem& it, float* acc, int G, int nf, int c) {
  const size_t tab = (size_t)(p.L + 1) * NY;
  const int n_un = p.n_un;
  const float scale = it.scale;
  bool ok = true;
  for (int ky = threadIdx.x; ky < NY; ky += blockDim.x) {
    for (int i = 0; i < p.n_obs; ++i) {
      const double rr = p.chat ? 0.0 : it.rhat[(size_t)i * tab + (size_t)ky * (p.L + 1) + c];
      float2* x0 = reinterpret_cast<float2*>(acc + p.n_obs * NY) + (size_t)i * n_un * NY + ky;
      if (p.spec) {
        const size_t at = (size_t)ky * (p.L + 1) + c;
        const double a = p.spec[(size_t)i * tab + at];
        ok &= finite_double(a);
        SpecQuotient q(a, rr, p.inv_G);
        acc[i * NY + ky] = q.times(a, a, rr);
        for (int u = 0; u < n_un; ++u) {
          const double* s = p.spec + (size_t)p.n_obs * tab + 2 * ((size_t)(i * n_un + u) * tab + at);
          ok &= finite_double(s[0]) && finite_double(s[1]);
          x0[(size_t)u * NY] = make_float2(q.times(s[0], a, rr), q.times(s[1], a, rr));
        }
        continue;
      }
      float val = 0.f;
      for (int g = 0; g < G; ++g) val += acc[(size_t)g * nf * NY + i * NY + ky];
      val *= scale;
      ok &= (bool)isfinite(val);
      float denf;
      const bool tiny = !denominator(val, rr, denf);
      const float inv = __fdividef(p.inv_G, denf);
      const double rd = (tiny && !p.chat) ? quotient_fp64(val, rr, p.inv_G) : 0.0;
      if (p.chat) p.chat[i * tab + (size_t)c * NY + ky] = val;
      else acc[i * NY + ky] = tiny ? (float)((double)val * rd) : val * inv;
      for (int q = 0; q < n_un; ++q) {
        float2 x = make_float2(0.f, 0.f);
        for (int g = 0; g < G; ++g) {
          const float2 a = *reinterpret_cast<const float2*>(reinterpret_cast<const float*>(x0 + (size_t)q * NY) + (size_t)g * nf * NY);
          x = cadd(x, a);
        }
        x = cscale(x, scale);
        ok &= isfinite(x.x) && isfinite(x.y);
        if (p.chat)
          reinterpret_cast<float2*>(p.chat + p.n_obs * tab)[(size_t)(i * n_un + q) * tab + (size_t)c * NY + ky] = x;
        else
          x0[(size_t)q * NY] = tiny ? make_float2((float)((double)x.x * rd), (float)((double)x.y * rd)) : cscale(x, inv);
      }
    }
  }
  return ok;
}

// Perturbations drawn in frequency space (seeded analysis), on the counter layout of the separate
// column update: v += sqrt(ny nx) sqrt(rhat) zhat of one stream; rh: rhat of k_y = 0, stride ys.
template <int NY, int V>
__device__ __forceinline__ void add_drawn(float2 (&v)[V], unsigned long long seed, int stream, int c, int L, int t,
                                          float sqrt_G, const double* rh, int ys) {
  constexpr int T = NY / V;
  if (c != 0 && c != L) {
    const float h = 0.70710678118654752f;
#pragma unroll
    for (int m = 0; m < V / 2; ++m) {
      const uint4 w4 = philox4x32_10(make_uint4((uint32_t)(t + T * m), (uint32_t)c, (uint32_t)stream, 0u),
                                     (uint32_t)seed, (uint32_t)(seed >> 32));
      const float2 zl = box_muller(w4.x, w4.y), zh = box_muller(w4.z, w4.w);
      const float al = h * sqrt_G * sqrtf(to_float(rh[(size_t)(t + T * m) * ys]));
      const float ah = h * sqrt_G * sqrtf(to_float(rh[(size_t)(t + T * (m + V / 2)) * ys]));
      v[m] = make_float2(fmaf(al, zl.x, v[m].x), fmaf(al, zl.y, v[m].y));
      v[m + V / 2] = make_float2(fmaf(ah, zh.x, v[m + V / 2].x), fmaf(ah, zh.y, v[m + V / 2].y));
    }
  } else {
#pragma unroll
    for (int m = 0; m < V; ++m) {
      const float a = sqrt_G * sqrtf(to_float(rh[(size_t)(t + T * m) * ys]));
      const float2 z = white_edge(seed, stream, t + T * m, c, NY);
      v[m] = make_float2(fmaf(a, z.x, v[m].x), fmaf(a, z.y, v[m].y));
    }
  }
}

// smem: sums [G][nf][NY] f32 | exchange lines [G][PL] f2.
// Every group runs the same number of rounds (a group without a member in the last round works on
// zeros), so that lines shorter than a warp can synchronise by whole warps.
template <int NY, int V, int NOBS, bool CROSS, bool DRAWN>
__global__ void __launch_bounds__(split_col_threads(NY, NOBS, CROSS), split_col_threads(NY, NOBS, CROSS) > 320 ? 1 : 2)
    col_split_kernel(const __grid_constant__ SplitParams p) {
  constexpr int T = NY / V;
  constexpr int PL = col_line_slots(NY);
  extern __shared__ __align__(128) unsigned char smraw[];
  stream_order_wait();
  int c;
  const SplitItem& it = split_item(p, c);
  const int G = blockDim.x / T;
  const int g = threadIdx.x / T, t = threadIdx.x - g * T;
  const int N = it.N, M = p.M, n_un = p.n_un;
  const int nf = p.n_obs + 2 * p.n_obs * n_un;
  float* acc0 = reinterpret_cast<float*>(smraw);
  float* acc = acc0 + (size_t)g * nf * NY;
  float2* line = reinterpret_cast<float2*>(smraw + p.acc_bytes) + (size_t)g * PL;
  const int part = (c == 0) ? 1 : ((c == p.L) ? 2 : 0);
  const int col = (c == p.L) ? 0 : c;
  const size_t fstride = (size_t)p.L * NY;
  const int rounds = (N + G - 1) / G;
  const int bid = line_bar<T>(g);

  auto fetch = [&](float2 (&v)[V], const float2* base, bool act) {
    const float2* src = base + (size_t)col * NY + t;
#pragma unroll
    for (int m = 0; m < V; ++m) v[m] = act ? src[T * m] : make_float2(0.f, 0.f);
  };
  auto real_part = [&](float2 (&v)[V]) {   // the packed column's real DC (.x) or Nyquist (.y) column
    if (part) {
#pragma unroll
      for (int m = 0; m < V; ++m) v[m] = make_float2(part == 1 ? v[m].x : v[m].y, 0.f);
    }
  };
  if (!p.spec) {
    // lines in the order (member round, role); the next one is requested before the current one's transform
    float2 nxt[V];
    fetch(nxt, it.A + ((size_t)p.role_block[0] * N + g) * fstride, g < N);
    auto take = [&](float2 (&v)[V], int r, int k) {   // the line of role r, member k, transformed
#pragma unroll
      for (int m = 0; m < V; ++m) v[m] = nxt[m];
      const int r1 = (r + 1 == M) ? 0 : r + 1, k1 = (r + 1 == M) ? k + G : k;
      fetch(nxt, it.A + ((size_t)p.role_block[r1] * N + k1) * fstride, k1 < N);
      real_part(v);
      fft_line<NY, V, false>(v, line, t, p.twY, bid);
    };
    float2 ko[NOBS][V];              // the member's observed spectra
    float au[CROSS ? 1 : NOBS][V];   // without cross sums the auto sums stay in registers
#pragma unroll
    for (int i = 0; i < (CROSS ? 1 : NOBS); ++i)
#pragma unroll
      for (int m = 0; m < V; ++m) au[i][m] = 0.f;
    for (int q = 0, k = g; q < rounds; ++q, k += G) {
      const float sg = (k == 0) ? -1.f : 1.f;   // member 0's place holds the pivot sum
#pragma unroll
      for (int i = 0; i < NOBS; ++i) {
        if (i >= p.n_obs) continue;
        take(ko[i], i, k);
        if constexpr (!CROSS) {
#pragma unroll
          for (int m = 0; m < V; ++m)
            au[i][m] = fmaf(sg * ko[i][m].x, ko[i][m].x, fmaf(sg * ko[i][m].y, ko[i][m].y, au[i][m]));
        } else {
          float* a = acc + i * NY + t;
#pragma unroll
          for (int m = 0; m < V; ++m)
            a[T * m] = fmaf(sg * ko[i][m].x, ko[i][m].x, fmaf(sg * ko[i][m].y, ko[i][m].y, q == 0 ? 0.f : a[T * m]));
        }
      }
      if constexpr (CROSS) {
        for (int u = 0; u < n_un; ++u) {
          float2 v[V];
          take(v, p.n_obs + u, k);
#pragma unroll
          for (int i = 0; i < NOBS; ++i) {
            if (i >= p.n_obs) continue;
            float2* a = reinterpret_cast<float2*>(acc + p.n_obs * NY) + (size_t)(i * n_un + u) * NY + t;
#pragma unroll
            for (int m = 0; m < V; ++m) {   // += sg v conj(ko)
              const float2 w = make_float2(sg * v[m].x, sg * v[m].y);
              float2 o = (q == 0) ? make_float2(0.f, 0.f) : a[T * m];
              o.x = fmaf(w.x, ko[i][m].x, fmaf(w.y, ko[i][m].y, o.x));
              o.y = fmaf(w.y, ko[i][m].x, fmaf(-w.x, ko[i][m].y, o.y));
              a[T * m] = o;
            }
          }
        }
      }
    }
    if constexpr (!CROSS) {
#pragma unroll
      for (int i = 0; i < NOBS; ++i) {
        if (i >= p.n_obs) continue;
#pragma unroll
        for (int m = 0; m < V; ++m) acc[i * NY + t + T * m] = au[i][m];
      }
    }
  }
  __syncthreads();
  if (!split_gains<NY>(p, it, acc0, G, nf, c)) atomicOr(p.status, kStatusNonFinite);
  if (p.chat) return;
  __syncthreads();
  for (int k = g, q = 0; q < rounds; ++q, k += G) {
    const bool act = k < N;
    float2 wv[NOBS][V];
#pragma unroll
    for (int i = 0; i < NOBS; ++i)
      if (i < p.n_obs) fetch(wv[i], it.W + ((size_t)k * p.n_obs + i) * fstride, act);
#pragma unroll
    for (int i = 0; i < NOBS; ++i) {
      if (i < p.n_obs) {
        real_part(wv[i]);
        fft_line<NY, V, false>(wv[i], line, t, p.twY, bid);
        if constexpr (DRAWN)
          if (act) add_drawn<NY, V>(wv[i], p.seed, k * p.n_obs + i, c, p.L, t, p.sqrt_G,
                                    it.rhat + (size_t)i * (p.L + 1) * NY + c, p.L + 1);
      } else {
#pragma unroll
        for (int m = 0; m < V; ++m) wv[i][m] = make_float2(0.f, 0.f);
      }
    }
    for (int r = 0; r < M; ++r) {
      float2 sv[V];
#pragma unroll
      for (int m = 0; m < V; ++m) sv[m] = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < NOBS; ++i) {
        if (i >= p.n_obs) continue;
        if (!CROSS || r < p.n_obs) {
          if (i == r) {
            const float* gp = acc0 + i * NY + t;
#pragma unroll
            for (int m = 0; m < V; ++m) sv[m] = cscale(wv[i][m], gp[T * m]);
          }
        } else {
          const float2* gp = reinterpret_cast<const float2*>(acc0 + p.n_obs * NY) + (size_t)(i * n_un + r - p.n_obs) * NY + t;
#pragma unroll
          for (int m = 0; m < V; ++m) {
            const float2 gv = gp[T * m];
            sv[m].x = fmaf(gv.x, wv[i][m].x, fmaf(-gv.y, wv[i][m].y, sv[m].x));
            sv[m].y = fmaf(gv.x, wv[i][m].y, fmaf(gv.y, wv[i][m].x, sv[m].y));
          }
        }
      }
      fft_line<NY, V, true>(sv, line, t, p.twY, bid);
      if (act) {
        float2* dst = it.A + ((size_t)p.role_block[r] * N + k) * fstride + (size_t)col * NY + t;
        if (part == 0) {
#pragma unroll
          for (int m = 0; m < V; ++m) dst[T * m] = sv[m];
        } else {
          float* d1 = reinterpret_cast<float*>(dst) + (part == 1 ? 0 : 1);
#pragma unroll
          for (int m = 0; m < V; ++m) d1[2 * T * m] = sv[m].x;
        }
      }
    }
  }
}

// ----------------------------------------------------------------- launch
// forward and inverse rows: one line group per row up to 256 threads, the tile in rounds otherwise
template <typename K>
inline cudaError_t launch_rows_split(K kern, int L, int V, SplitParams p, int units, cudaStream_t st) {
  const int T = L / V;
  p.R = split_row_tile(L);
  int lpc = (p.threads ? p.threads : 256) / T;
  if (lpc < 1) lpc = 1;
  if (lpc > p.R) lpc = p.R;
  const size_t smem = (size_t)p.R * row_pitch(L) * sizeof(float2);
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_overlapped(kern, dim3((unsigned)units), T * lpc, smem, st, p);
}

template <int ST>
inline cudaError_t row_split_st(const SplitParams& p, int units, cudaStream_t s) {
  switch (p.L) {
#define CASE(n) case n: return launch_rows_split(row_split_kernel<n, split_row_V(n), ST>, n, split_row_V(n), p, units, s);
    FFTENKF_ROW_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}
template <int ST>
inline cudaError_t row_inv_split_st(const SplitParams& p, int units, cudaStream_t s) {
  switch (p.L) {
#define CASE(n) case n: return launch_rows_split(row_inv_split_kernel<n, split_row_V(n), ST>, n, split_row_V(n), p, units, s);
    FFTENKF_ROW_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t row_split_f32(const SplitParams& p, int units, cudaStream_t s);
cudaError_t row_split_bf16(const SplitParams& p, int units, cudaStream_t s);
cudaError_t row_inv_split_f32(const SplitParams& p, int units, cudaStream_t s);
cudaError_t row_inv_split_bf16(const SplitParams& p, int units, cudaStream_t s);

#define FFTENKF_SPLIT_COL_SIZES(X) \
  X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024) X(1536) X(2048)

template <int NY, int NOBS, bool CROSS, bool DRAWN>
inline cudaError_t col_split_NY(const SplitParams& p, int units, cudaStream_t st) {
  constexpr int V = plan_V(NY, split_col_sel(NY, CROSS)), T = NY / V;
  const size_t smem = (size_t)p.acc_bytes + (size_t)p.groups * col_line_slots(NY) * sizeof(float2);
  auto kern = col_split_kernel<NY, V, NOBS, CROSS, DRAWN>;
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_overlapped(kern, dim3((unsigned)units), T * p.groups, smem, st, p);
}
template <int NOBS, bool DRAWN>
inline cudaError_t col_split_dispatch(const SplitParams& p, int units, cudaStream_t s) {
  switch (p.ny) {
#define CASE(n) \
  case n: return p.n_un ? col_split_NY<n, NOBS, true, DRAWN>(p, units, s) : col_split_NY<n, NOBS, false, DRAWN>(p, units, s);
    FFTENKF_SPLIT_COL_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t col_split_1(const SplitParams& p, int units, cudaStream_t s);
cudaError_t col_split_2(const SplitParams& p, int units, cudaStream_t s);
cudaError_t col_split_4(const SplitParams& p, int units, cudaStream_t s);
cudaError_t col_split_drawn_1(const SplitParams& p, int units, cudaStream_t s);
cudaError_t col_split_drawn_2(const SplitParams& p, int units, cudaStream_t s);
cudaError_t col_split_drawn_4(const SplitParams& p, int units, cudaStream_t s);

}  // namespace fftenkf
