// The real sine variant without the odd extension: DST-I rows and columns of the interior, as split
// passes (one CTA per tile of rows, one per wavenumber column).
//
// The transform of both directions is T(x)_k = 2 sum_j x_j sin(pi j k / n), n = m + 1 (the DFT of the odd
// extension to P = 2 n points is -i T), its own inverse up to the factor P.  Two real lines a, b make one
// complex line z = a + i b, whose odd extension has the P-point DFT T(b) - i T(a): so a P-point line FFT
// transforms two lines, their extension is a matter of indexing, and only real coefficients of the m
// wavenumbers are stored: a quarter of the row spectra of the periodic analysis of the extension, half of
// its transforms, and no extended copies of the inputs.
//
// Layouts: coefficients of a field after the rows [nx-2][ny-1] floats (k_x = 1.., y = 1.. contiguous; the
// entry of y = ny-1 is 0), anomaly field j N + k (k = 0: the scaled sum of the differences to member 0, as in
// the periodic passes), innovation field k n_obs + i.
#pragma once
#include "common.cuh"
#include "dd.cuh"
#include "k_rows.cuh"
#include "launch.cuh"

namespace fftenkf {

// complex lines of a row tile, two rows each: the longest in tiles of 4 rows, so that two CTAs share an SM
// (2049^2 nodes, 4 blocks, N=20, BF16: 11.0 -> 8.4 ms; at 3072 points, 513 x 1537, 2 blocks,
// tiles of 4 would take 916 us instead of 870)
__host__ __device__ constexpr int sine_tile_lines(int P) { return P >= 4096 ? 2 : 4; }

// The line transforms of the sine passes; power-of-two lines up to 1024 points with every twiddle power from the
// table: they are twice as long as the periodic passes' rows of the same grid, and with formed powers FP32 analyses
// were further from the 64-bit result than through the extension (65^2 nodes, N=5, 2 blocks 3.1e-7 and 2.8e-7, mean
// of three draws; 2.5e-7 like this, at the same speed: 1025^2 1543 us both).
template <int P, int V, bool TRAIL = true>
__device__ __forceinline__ void sine_line(float2 (&v)[V], float2* line, int t, const float2* __restrict__ tw, int bid) {
  fft_line<P, V, false, TRAIL, sine_every(P)>(v, line, t, tw, bid);
}

template <int ST>
__device__ __forceinline__ float load1(const void* base, size_t idx) {
  if constexpr (ST == kBF16) return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(base)[idx]);
  else return reinterpret_cast<const float*>(base)[idx];
}

// The odd extension of a line whose first half (positions t + T m, m < V/2, 0 at position 0) is in v: the
// mirrored positions come from other threads of the line through its buffer.
template <int P, int V>
__device__ __forceinline__ void odd_extension(float2 (&v)[V], float2* line, int t, int bid) {
  constexpr int T = P / V, n = P / 2;
#pragma unroll
  for (int m = 0; m < V / 2; ++m) line[pidx(t + T * m)] = v[m];
  line_sync<T>(bid);
#pragma unroll
  for (int m = V / 2; m < V; ++m) {
    const int at = t + T * m;
    const float2 x = at == n ? make_float2(0.f, 0.f) : line[pidx(P - at)];
    v[m] = make_float2(-x.x, -x.y);
  }
  line_sync<T>(bid);
}

// ----------------------------------------------------------------- forward rows
// unit = tile * n_fields + f, as row_split_kernel; rows y = 1 + 2 NL tile .. as NL complex lines
template <int P, int ST>
__global__ void __launch_bounds__(256, 2) sine_rows_kernel(const __grid_constant__ SineParams p) {
  constexpr int V = plan_V(P, 0), T = P / V, pitch = row_pitch(P), NL = sine_tile_lines(P), Q = NL / 2;
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* lines = reinterpret_cast<float2*>(smraw);
  stream_order_wait();
  const int LPC = blockDim.x / T;
  const int g = threadIdx.x / T, t = threadIdx.x - g * T;
  const int N = p.N, ny = p.ny, nx = p.nx;
  const int n_anom = p.anomalies ? p.M * N : 0;
  const int n_fields = n_anom + (p.innovations ? N * p.n_obs : 0);
  const int tile = blockIdx.x / n_fields;
  const int f = blockIdx.x - tile * n_fields;
  const size_t G = (size_t)ny * nx;
  constexpr int es = (ST == kBF16) ? 2 : 4;
  const char* ens = reinterpret_cast<const char*>(p.ens);
  const bool anom = f < n_anom;
  int j = 0, k = 0, i = 0;
  if (anom) {
    j = f < p.M ? f : (f - p.M) / (N - 1);
    k = f < p.M ? 0 : 1 + (f - p.M) - j * (N - 1);
  } else {
    const int w = f - n_anom;
    k = w / p.n_obs;
    i = w - k * p.n_obs;
#pragma unroll
    for (int q = 0; q < kMaxObs; ++q)
      if (q == i) j = p.obs[q];
  }
  const char* u0 = ens + (size_t)j * N * G * es;             // member 0 of the block
  const char* uk = u0 + (size_t)k * G * es;
  const float* d = p.data + (size_t)i * G;
  const char* e = reinterpret_cast<const char*>(p.pert) + ((size_t)k * p.n_obs + i) * G * es;
  for (int l = 0; l < NL; l += LPC) {
    const int y = 1 + 2 * NL * tile + 2 * (l + g);                // rows y and y + 1
    const size_t ra = (size_t)y * nx, rb = ra + nx;
    const bool has_b = y + 1 < ny - 1;                       // the last line's second row is the boundary
    // Every load is unconditional (position 0 and the row after the last are the grid's boundary) and issued
    // before the first use: with the zeros chosen by branches around the loads few were in flight, and 62 % of
    // the stalls were waits for them (analysis of 1025^2 nodes, 4 observed blocks, N=20, BF16: 2.52 -> 1.96 ms).
    float2 v[V], c[V / 2], d2[V / 2];
    const bool sum = anom && k == 0;
#pragma unroll
    for (int m = 0; m < V / 2; ++m) {
      const int x = t + T * m;
      v[m] = make_float2(load1<ST>(uk, ra + x), load1<ST>(uk, rb + x));
      if (anom) c[m] = make_float2(load1<ST>(u0, ra + x), load1<ST>(u0, rb + x));
      else {
        c[m] = make_float2(load1<ST>(e, ra + x), load1<ST>(e, rb + x));
        d2[m] = make_float2(d[ra + x], d[rb + x]);
      }
    }
    if (!anom) {
#pragma unroll
      for (int m = 0; m < V / 2; ++m) v[m] = cadd(csub(d2[m], v[m]), c[m]);   // d - u first
    } else if (!sum) {
#pragma unroll
      for (int m = 0; m < V / 2; ++m) v[m] = csub(v[m], c[m]);
    } else {   // (1/sqrt N) sum_k (u_k - u_0), in member order
#pragma unroll
      for (int m = 0; m < V / 2; ++m) v[m] = make_float2(0.f, 0.f);
#pragma unroll 2
      for (int q = 1; q < N; ++q) {
        const char* uq = u0 + (size_t)q * G * es;
#pragma unroll
        for (int m = 0; m < V / 2; ++m)
          v[m] = cadd(v[m], csub(make_float2(load1<ST>(uq, ra + t + T * m), load1<ST>(uq, rb + t + T * m)), c[m]));
      }
#pragma unroll
      for (int m = 0; m < V / 2; ++m) v[m] = cscale(v[m], p.inv_sqrt_N);
    }
#pragma unroll
    for (int m = 0; m < V / 2; ++m) {
      if (t + T * m == 0) v[m] = make_float2(0.f, 0.f);
      if (!has_b) v[m].y = 0.f;
    }
    float2* line = lines + (l + g) * pitch;
    odd_extension<P, V>(v, line, t, line_bar<T>(g));
    sine_line<P, V>(v, line, t, p.twx, line_bar<T>(g));
    float* fa = reinterpret_cast<float*>(line);   // T(a) = -Im Z, T(b) = Re Z at k = 0..n-1
#pragma unroll
    for (int m = 0; m < V / 2; ++m) {
      fa[t + T * m] = -v[m].y;
      fa[pitch + t + T * m] = v[m].x;
    }
  }
  __syncthreads();
  float* out = (anom ? p.A + ((size_t)j * N + k) * p.fstride : p.W + ((size_t)k * p.n_obs + i) * p.fstride) + 2 * NL * tile;
  const float* fl = reinterpret_cast<const float*>(lines);
  for (int q = threadIdx.x; q < Q * (nx - 2); q += blockDim.x) {
    const int kx = 1 + q / Q, h = q % Q;
    const float* r0 = fl + (size_t)(2 * h) * 2 * pitch + kx;
    *reinterpret_cast<float4*>(out + (size_t)(kx - 1) * (ny - 1) + 4 * h) =
        make_float4(r0[0], r0[pitch], r0[2 * pitch], r0[3 * pitch]);
  }
}

// ----------------------------------------------------------------- inverse rows
// unit = tile * (M N) + field: the increments' coefficients of 2 NL rows, extended, transformed and added
template <int P, int ST>
__global__ void __launch_bounds__(256, 2) sine_rows_inv_kernel(const __grid_constant__ SineParams p) {
  constexpr int V = plan_V(P, 0), T = P / V, n = P / 2, pitch = row_pitch(P), NL = sine_tile_lines(P), Q = NL / 2;
  extern __shared__ __align__(128) unsigned char smraw[];
  float2* lines = reinterpret_cast<float2*>(smraw);
  stream_order_wait();
  const int LPC = blockDim.x / T;
  const int g = threadIdx.x / T, t = threadIdx.x - g * T;
  const int nf = p.M * p.N, ny = p.ny, nx = p.nx;
  const int tile = blockIdx.x / nf, f = blockIdx.x - tile * nf;
  const float* in = p.A + (size_t)f * p.fstride + 2 * NL * tile;
#pragma unroll 4
  for (int q = threadIdx.x; q < Q * (nx - 2); q += blockDim.x) {
    const int kx = 1 + q / Q, h = q % Q;
    const float4 s = *reinterpret_cast<const float4*>(in + (size_t)(kx - 1) * (ny - 1) + 4 * h);
    float2* l0 = lines + (2 * h) * pitch;
    float2* l1 = l0 + pitch;
    l0[pidx(kx)] = make_float2(s.x, s.y);
    l0[pidx(P - kx)] = make_float2(-s.x, -s.y);
    l1[pidx(kx)] = make_float2(s.z, s.w);
    l1[pidx(P - kx)] = make_float2(-s.z, -s.w);
  }
  for (int q = threadIdx.x; q < 2 * NL; q += blockDim.x) lines[(q >> 1) * pitch + pidx((q & 1) * n)] = make_float2(0.f, 0.f);
  __syncthreads();
  constexpr int es = (ST == kBF16) ? 2 : 4;
  char* u = reinterpret_cast<char*>(p.ens) + (size_t)f * ny * nx * es;
  for (int l = 0; l < NL; l += LPC) {
    const int y = 1 + 2 * NL * tile + 2 * (l + g);
    const size_t ra = (size_t)y * nx, rb = ra + nx;
    const bool has_b = y + 1 < ny - 1;
    float2* line = lines + (l + g) * pitch;
    float2 v[V], a[V / 2];
#pragma unroll
    for (int m = 0; m < V / 2; ++m) {
      const int x = t + T * m;
      a[m] = make_float2(load1<ST>(u, ra + x), load1<ST>(u, rb + x));
    }
#pragma unroll
    for (int m = 0; m < V; ++m) v[m] = line[pidx(t + T * m)];
    line_sync<T>(line_bar<T>(g));
    sine_line<P, V, false>(v, line, t, p.twx, line_bar<T>(g));
#pragma unroll
    for (int m = 0; m < V / 2; ++m) {
      const int x = t + T * m;
      if (x == 0) continue;
      const float va = a[m].x - v[m].y, vb = a[m].y + v[m].x;
      if constexpr (ST == kBF16) {
        __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(u);
        o[ra + x] = __float2bfloat16_rn(va);
        if (has_b) o[rb + x] = __float2bfloat16_rn(vb);
      } else {
        float* o = reinterpret_cast<float*>(u);
        o[ra + x] = va;
        if (has_b) o[rb + x] = vb;
      }
    }
  }
}

// ----------------------------------------------------------------- columns
// unit: the wavenumber columns k_x = 1 + 2 blockIdx.x and the next, as the two real lines of one complex
// line (of one field: a column's coefficients carry the row transform's rounding of their neighbours
// already, so the pair adds none that a block or member of another scale would bring).  As
// col_split_kernel: members over the CTA's groups, sums in shared memory, gains, update; all tables real.
// smem: sums [groups][nf][2][n] f32, n = ny - 1 | exchange lines [groups][PL] f2
template <int P, int NOBS>
__global__ void __launch_bounds__(sine_col_threads(NOBS), 1) sine_cols_kernel(const __grid_constant__ SineParams p) {
  constexpr int V = plan_V(P, 0), T = P / V, n = P / 2, H = V / 2, PL = col_line_slots(P);
  extern __shared__ __align__(128) unsigned char smraw[];
  stream_order_wait();
  const int G = blockDim.x / T;
  const int g = threadIdx.x / T, t = threadIdx.x - g * T;
  const int N = p.N, M = p.M, n_un = M - p.n_obs;
  const int nf = p.n_obs * (1 + n_un);
  float* acc0 = reinterpret_cast<float*>(smraw);
  float* acc = acc0 + (size_t)g * nf * P;
  float2* line = reinterpret_cast<float2*>(smraw + p.acc_bytes) + (size_t)g * PL;
  const int bid = line_bar<T>(g);
  const int rounds = (N + G - 1) / G;
  const size_t col = (size_t)2 * blockIdx.x * n;          // of a field
  const bool two = 2 * (int)blockIdx.x + 1 < p.nx - 2;    // the last column has no partner
  // transform both columns of a field (nullptr: zeros): c[m], c[H + m] = coefficient t + T m of the first
  // and of the second
  auto coefficients = [&](float (&c)[V], const float* f) {
    float2 v[V];
#pragma unroll
    for (int m = 0; m < H; ++m) {
      const int y = t + T * m;
      const bool in = f && y != 0;
      v[m] = make_float2(in ? f[col + y - 1] : 0.f, in && two ? f[col + n + y - 1] : 0.f);
    }
    odd_extension<P, V>(v, line, t, bid);
    sine_line<P, V>(v, line, t, p.twy, bid);
#pragma unroll
    for (int m = 0; m < H; ++m) {
      c[m] = -v[m].y;
      c[H + m] = v[m].x;
    }
  };
  for (int q = 0, k = g; q < rounds; ++q, k += G) {
    const float sg = (k == 0) ? -1.f : 1.f;   // member 0's place holds the pivot sum
    float ko[NOBS][V];
#pragma unroll
    for (int i = 0; i < NOBS; ++i) {
      if (i < p.n_obs) {
        coefficients(ko[i], k < N ? p.A + ((size_t)p.role_block[i] * N + k) * p.fstride : nullptr);
        float* s = acc + (size_t)i * P + t;
#pragma unroll
        for (int m = 0; m < V; ++m) s[T * m] = fmaf(sg * ko[i][m], ko[i][m], q == 0 ? 0.f : s[T * m]);
      } else {
#pragma unroll
        for (int m = 0; m < V; ++m) ko[i][m] = 0.f;
      }
    }
    for (int u = 0; u < n_un; ++u) {
      float c[V];
      coefficients(c, k < N ? p.A + ((size_t)p.role_block[p.n_obs + u] * N + k) * p.fstride : nullptr);
#pragma unroll
      for (int i = 0; i < NOBS; ++i) {
        if (i >= p.n_obs) continue;
        float* s = acc + (size_t)(p.n_obs + i * n_un + u) * P + t;
#pragma unroll
        for (int m = 0; m < V; ++m) s[T * m] = fmaf(sg * c[m], ko[i][m], q == 0 ? 0.f : s[T * m]);
      }
    }
  }
  __syncthreads();
  bool ok = true;
  const size_t tab = (size_t)(p.ny - 2) * (p.nx - 2);
  for (int at = threadIdx.x; at < P; at += blockDim.x) {   // the first column's wavenumbers, then the second's
    const int ky = at < n ? at : at - n;
    if (ky == 0 || (at >= n && !two)) continue;
    const size_t out = (size_t)(ky - 1) * (p.nx - 2) + 2 * blockIdx.x + (at >= n);
    auto total = [&](int f) {
      float s = 0.f;
      for (int q = 0; q < G; ++q) s += acc0[((size_t)q * nf + f) * P + at];
      return s * p.scale;
    };
    for (int i = 0; i < p.n_obs; ++i) {
      const float val = total(i);
      ok &= (bool)isfinite(val);
      if (p.spectrum_out) {
        p.spectrum_out[i * tab + out] = to_double(val);
        for (int u = 0; u < n_un; ++u) {
          const float x = total(p.n_obs + i * n_un + u);
          ok &= (bool)isfinite(x);
          p.spectrum_out[(p.n_obs + i * n_un + u) * tab + out] = to_double(x);
        }
        continue;
      }
      const double r = p.rhat[i * tab + out];
      float den;
      const bool tiny = !denominator(val, r, den);
      const float inv = __fdividef(p.inv_G, den);
      const double rd = tiny ? quotient_fp64(val, r, p.inv_G) : 0.0;
      acc0[(size_t)i * P + at] = tiny ? (float)((double)val * rd) : val * inv;
      for (int u = 0; u < n_un; ++u) {
        const int f = p.n_obs + i * n_un + u;
        const float x = total(f);
        ok &= (bool)isfinite(x);
        acc0[(size_t)f * P + at] = tiny ? (float)((double)x * rd) : x * inv;
      }
    }
  }
  if (!ok) atomicOr(p.status, kStatusNonFinite);
  if (p.spectrum_out) return;
  __syncthreads();
  for (int q = 0, k = g; q < rounds; ++q, k += G) {
    const bool act = k < N;
    float w[NOBS][V];
#pragma unroll
    for (int i = 0; i < NOBS; ++i) {
      if (i < p.n_obs) {
        coefficients(w[i], act ? p.W + ((size_t)k * p.n_obs + i) * p.fstride : nullptr);
      } else {
#pragma unroll
        for (int m = 0; m < V; ++m) w[i][m] = 0.f;
      }
    }
    for (int r = 0; r < M; ++r) {
      float s[V];
#pragma unroll
      for (int m = 0; m < V; ++m) s[m] = 0.f;
#pragma unroll
      for (int i = 0; i < NOBS; ++i) {
        if (i >= p.n_obs || (r < p.n_obs && i != r)) continue;
        const float* gain = acc0 + (size_t)(r < p.n_obs ? r : p.n_obs + i * n_un + r - p.n_obs) * P + t;
#pragma unroll
        for (int m = 0; m < V; ++m) s[m] = fmaf(gain[T * m], w[i][m], s[m]);
      }
      float2 v[V];
#pragma unroll
      for (int m = 0; m < H; ++m) {
        const bool in = t + T * m != 0;   // no wavenumber 0
        v[m] = make_float2(in ? s[m] : 0.f, in && two ? s[H + m] : 0.f);
      }
      odd_extension<P, V>(v, line, t, bid);
      sine_line<P, V>(v, line, t, p.twy, bid);
      if (!act) continue;
      float* o = p.A + ((size_t)p.role_block[r] * N + k) * p.fstride + col;
#pragma unroll
      for (int m = 0; m < H; ++m) {
        const int y = t + T * m;
        if (y == 0) continue;
        o[y - 1] = -v[m].y;
        if (two) o[n + y - 1] = v[m].x;
      }
    }
  }
}

// ----------------------------------------------------------------- launch
// lengths of the extension; the rows' tiles of 8 need ny - 1 to be a multiple of 8
#define FFTENKF_SINE_SIZES(X) \
  X(16) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(384) X(512) X(768) X(1024) X(1536) X(2048) X(3072) X(4096)

template <typename K>
inline cudaError_t launch_sine_rows(K kern, int P, const SineParams& p, int units, cudaStream_t s) {
  const int T = P / plan_V(P, 0);
  int lpc = 256 / T;
  if (lpc < 1) return cudaErrorInvalidConfiguration;
  lpc = lpc >= sine_tile_lines(P) ? sine_tile_lines(P) : lpc >= 2 ? 2 : 1;
  const size_t smem = (size_t)sine_tile_lines(P) * row_pitch(P) * sizeof(float2);
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_overlapped(kern, dim3((unsigned)units), T * lpc, smem, s, p);
}
template <int ST>
inline cudaError_t sine_rows_st(const SineParams& p, bool inverse, int units, cudaStream_t s) {
  switch (2 * (p.nx - 1)) {
#define CASE(n) \
  case n: return inverse ? launch_sine_rows(sine_rows_inv_kernel<n, ST>, n, p, units, s) : launch_sine_rows(sine_rows_kernel<n, ST>, n, p, units, s);
    FFTENKF_SINE_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}
template <int P, int NOBS>
inline cudaError_t sine_cols_P(const SineParams& p, cudaStream_t s) {
  const size_t smem = (size_t)p.acc_bytes + (size_t)p.groups * col_line_slots(P) * sizeof(float2);
  const int threads = P / plan_V(P, 0) * p.groups;
  auto kern = sine_cols_kernel<P, NOBS>;
  cudaError_t e = allow_smem(reinterpret_cast<const void*>(kern), smem);
  if (e != cudaSuccess) return e;
  return launch_overlapped(kern, dim3((unsigned)((p.nx - 1) / 2)), threads, smem, s, p);
}
template <int NOBS>
inline cudaError_t sine_cols_dispatch(const SineParams& p, cudaStream_t s) {
  switch (2 * (p.ny - 1)) {
#define CASE(n) case n: return sine_cols_P<n, NOBS>(p, s);
    FFTENKF_SINE_SIZES(CASE)
#undef CASE
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t sine_rows_f32(const SineParams& p, bool inverse, int units, cudaStream_t s);
cudaError_t sine_rows_bf16(const SineParams& p, bool inverse, int units, cudaStream_t s);
cudaError_t sine_cols_1(const SineParams& p, cudaStream_t s);
cudaError_t sine_cols_2(const SineParams& p, cudaStream_t s);
cudaError_t sine_cols_4(const SineParams& p, cudaStream_t s);

}  // namespace fftenkf
