// Gain tables of eq. (spectral-enkf) / eq. (spectral-multi-enkf) from a caller's
// spectrum, in float pairs per wavenumber (dd.cuh), and the transpose of the covariance tables to the
// boundary's [k_y][k_x] layout.
//
//   G^(oo) = chat^(oo) / (chat^(oo) + rhat_o),  G^(jo) = chat^(jo) / (chat^(oo) + rhat_o)
//
// with G = 0 where the denominator is 0.  The tables are stored as float in
// the column passes' [k_x][k_y] layout with 1/(ny nx) folded in (the column
// and row passes use unnormalised transforms).  rhat and a caller-supplied
// spectrum arrive in [k_y][k_x] layout and are transposed through shared
// memory in 32 x 32 tiles so that every global access is coalesced.
#include <cstring>

#include "common.cuh"
#include "dd.cuh"

namespace fftenkf {

constexpr int TB = 32;

// load a [ny][L+1] double tile (rows ky0.., cols c0..) into s[ky][c]
__device__ __forceinline__ void load_tile(double (*s)[TB + 1], const double* __restrict__ src, int ny, int L1,
                                          int ky0, int c0, int stride_elems, int comp) {
  for (int yy = threadIdx.y; yy < TB; yy += blockDim.y) {
    const int ky = ky0 + yy, c = c0 + threadIdx.x;
    s[yy][threadIdx.x] = (ky < ny && c < L1) ? src[((size_t)ky * L1 + c) * stride_elems + comp] : 0.0;
  }
}

__global__ void __launch_bounds__(256) gain_kernel(const GainParams p) {
  __shared__ double rs[TB][TB + 1];
  __shared__ double ca[TB][TB + 1];
  __shared__ double cre[TB][TB + 1];
  __shared__ double cim[TB][TB + 1];
  const int L1 = p.L + 1;
  const int c0 = blockIdx.x * TB, ky0 = blockIdx.y * TB, i = blockIdx.z;
  const size_t K = (size_t)p.ny * L1;   // doubles per real table (natural layout)
  const size_t tab = (size_t)L1 * p.ny;  // elements per transposed table
  load_tile(rs, p.rhat + i * K, p.ny, L1, ky0, c0, 1, 0);
  load_tile(ca, p.spec + i * K, p.ny, L1, ky0, c0, 1, 0);
  __syncthreads();
  // thread (x -> ky offset, y -> column offset): coalesced along k_y on output
  const int ky = ky0 + threadIdx.x;
  bool bad = false;
  auto quotient = [&](int q) {   // of this thread's q-th wavenumber (entries off the grid are 0)
    const int cl = threadIdx.y + 8 * q;
    return SpecQuotient(ca[threadIdx.x][cl], rs[threadIdx.x][cl], p.scale);
  };
  SpecQuotient inv[TB / 8] = {quotient(0), quotient(1), quotient(2), quotient(3)};
#pragma unroll
  for (int q = 0; q < TB / 8; ++q) {
    const int cl = threadIdx.y + 8 * q;
    const int c = c0 + cl;
    if (c < L1 && ky < p.ny) {
      const double a = ca[threadIdx.x][cl];
      bad |= !finite_double(a);
      p.goo[i * tab + (size_t)c * p.ny + ky] = inv[q].times(a, a, rs[threadIdx.x][cl]);
    }
  }
  const double* xspec = p.spec + (size_t)p.n_obs * K;
  for (int u = 0; u < p.n_un; ++u) {
    const int qt = i * p.n_un + u;
    __syncthreads();
    load_tile(cre, xspec + (size_t)qt * 2 * K, p.ny, L1, ky0, c0, 2, 0);
    load_tile(cim, xspec + (size_t)qt * 2 * K, p.ny, L1, ky0, c0, 2, 1);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < TB / 8; ++q) {
      const int cl = threadIdx.y + 8 * q;
      const int c = c0 + cl;
      if (c < L1 && ky < p.ny) {
        const double re = cre[threadIdx.x][cl], im = cim[threadIdx.x][cl];
        bad |= !(finite_double(re) && finite_double(im));
        const double a = ca[threadIdx.x][cl], r = rs[threadIdx.x][cl];
        p.gjo[qt * tab + (size_t)c * p.ny + ky] = make_float2(inv[q].times(re, a, r), inv[q].times(im, a, r));
      }
    }
  }
  if (bad) atomicOr(p.status, kStatusNonFinite);
}

cudaError_t launch_gain(const GainParams& p, cudaStream_t s) {
  dim3 grid((p.L + 1 + TB - 1) / TB, (p.ny + TB - 1) / TB, p.n_obs);
  gain_kernel<<<grid, dim3(TB, 8), 0, s>>>(p);
  return cudaGetLastError();
}

// chat_t (float, [table][L+1][ny]) -> out (double, natural [table][ny][L+1], crosses (re,im))
__global__ void __launch_bounds__(256) chat_out_kernel(const float* __restrict__ chat_t, double* __restrict__ out,
                                                       int ny, int L, const ChatOutMap map) {
  __shared__ float2 tile[TB][TB + 1];
  const int L1 = L + 1;
  const int c0 = blockIdx.x * TB, ky0 = blockIdx.y * TB, q = blockIdx.z;
  const bool is_auto = q < map.n_auto;
  const size_t tab = (size_t)L1 * ny;
  const size_t K = (size_t)ny * L1;
  int src = 0, cj = 0;
  if (!is_auto) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)   // constant indices keep the map in the parameter bank
      if (i == q - map.n_auto) {
        src = map.src[i];
        cj = map.conj[i];
      }
  }
  for (int cc = threadIdx.y; cc < TB; cc += blockDim.y) {
    const int c = c0 + cc, ky = ky0 + threadIdx.x;
    float2 v = make_float2(0.f, 0.f);
    if (c < L1 && ky < ny) {
      if (is_auto) {
        v.x = chat_t[q * tab + (size_t)c * ny + ky];
      } else {
        v = reinterpret_cast<const float2*>(chat_t + map.n_auto * tab)[src * tab + (size_t)c * ny + ky];
        if (cj) v.y = -v.y;
      }
    }
    tile[cc][threadIdx.x] = v;
  }
  __syncthreads();
  for (int yy = threadIdx.y; yy < TB; yy += blockDim.y) {
    const int ky = ky0 + yy, c = c0 + threadIdx.x;
    if (ky < ny && c < L1) {
      const float2 v = tile[threadIdx.x][yy];
      if (is_auto) {
        out[q * K + (size_t)ky * L1 + c] = to_double(v.x);
      } else {
        double* o = out + map.n_auto * K + (size_t)(q - map.n_auto) * 2 * K + ((size_t)ky * L1 + c) * 2;
        o[0] = to_double(v.x);
        o[1] = to_double(v.y);
      }
    }
  }
}

// Output tables: the auto table of every observed block, then for every observed o (ascending)
// the cross tables chat^(jo) of every block j != o (ascending; unobserved j only unless coupled).
// Column-pass tables: autos, then (coupled) the observed pair chat^(o1 o0), then chat^(u o_i) at
// n_pair + i n_un + u.
ChatOutMap chat_out_map(int n_obs, int n_un, int coupled, const int* obs, const int* un, int M) {
  ChatOutMap m;
  memset(&m, 0, sizeof(m));
  m.n_auto = n_obs;
  const int n_pair = coupled ? n_obs * (n_obs - 1) / 2 : 0;
  for (int i = 0; i < n_obs; ++i) {
    for (int j = 0; j < M; ++j) {
      if (j == obs[i]) continue;
      int u = -1, oi = -1;
      for (int a = 0; a < n_un; ++a)
        if (un[a] == j) u = a;
      for (int a = 0; a < n_obs; ++a)
        if (obs[a] == j) oi = a;
      if (u >= 0) {
        m.src[m.n_cplx] = n_pair + i * n_un + u;
        m.conj[m.n_cplx] = 0;
        ++m.n_cplx;
      } else if (coupled && oi >= 0) {   // n_obs = 2: chat^(o1 o0) stored, chat^(o0 o1) its conjugate
        m.src[m.n_cplx] = 0;
        m.conj[m.n_cplx] = (oi == 0) ? 1 : 0;
        ++m.n_cplx;
      }
    }
  }
  return m;
}

cudaError_t launch_chat_out(const float* chat_t, double* out, int ny, int L, const ChatOutMap& map, cudaStream_t s) {
  dim3 grid((L + 1 + TB - 1) / TB, (ny + TB - 1) / TB, map.n_auto + map.n_cplx);
  chat_out_kernel<<<grid, dim3(TB, 8), 0, s>>>(chat_t, out, ny, L, map);
  return cudaGetLastError();
}

// rhat [n][ny][L1] -> rhat_t [n][L1][ny]; with amp non-null also amp [n][L1][ny] = sqrt_G sqrt(rhat) in
// FP32, the amplitude of the perturbations drawn in frequency space
__global__ void __launch_bounds__(256) rhat_transpose_kernel(const double* __restrict__ in, double* __restrict__ out,
                                                             int ny, int L1, float* __restrict__ amp, float sqrt_G) {
  __shared__ double tile[TB][TB + 1];
  const int c0 = blockIdx.x * TB, ky0 = blockIdx.y * TB;
  const size_t K = (size_t)ny * L1;
  const double* src = in + blockIdx.z * K;
  double* dst = out + blockIdx.z * K;
  for (int yy = threadIdx.y; yy < TB; yy += blockDim.y) {
    const int ky = ky0 + yy, c = c0 + threadIdx.x;
    tile[yy][threadIdx.x] = (ky < ny && c < L1) ? src[(size_t)ky * L1 + c] : 0.0;
  }
  __syncthreads();
  for (int cc = threadIdx.y; cc < TB; cc += blockDim.y) {
    const int c = c0 + cc, ky = ky0 + threadIdx.x;
    if (c < L1 && ky < ny) {
      const double r = tile[threadIdx.x][cc];
      dst[(size_t)c * ny + ky] = r;
      if (amp) amp[blockIdx.z * K + (size_t)c * ny + ky] = sqrt_G * sqrtf(to_float(r));
    }
  }
}

cudaError_t launch_rhat_transpose(const double* rhat, double* rhat_t, int n, int ny, int L, cudaStream_t s,
                                  float* amp, float sqrt_G) {
  dim3 grid((L + 1 + TB - 1) / TB, (ny + TB - 1) / TB, n);
  rhat_transpose_kernel<<<grid, dim3(TB, 8), 0, s>>>(rhat, rhat_t, ny, L + 1, amp, sqrt_G);
  return cudaGetLastError();
}

// One thread per wavenumber (column-major index at = k_x ny + k_y).  The bracket A = chat_OO +
// diag(rhat) is inverted (bracket, dd.cuh; in FP64 the kernel took 465 us at 4096^2 with three blocks),
// scaled by 1/(ny nx) and rounded to float, and K_r = chat_{r,O} A^-1 is formed in FP32.
__global__ void __launch_bounds__(256) coupled_gain_kernel(const CoupledGainParams p) {
  const size_t tab = (size_t)(p.L + 1) * p.ny;
  const float2* cx = reinterpret_cast<const float2*>(p.chat_t + p.n_obs * tab);
  bool bad = false;
  for (size_t at = blockIdx.x * (size_t)blockDim.x + threadIdx.x; at < tab; at += (size_t)gridDim.x * blockDim.x) {
    const float a0 = p.chat_t[at];
    const float a1 = (p.n_obs == 2) ? p.chat_t[tab + at] : 0.f;
    const float2 b10 = (p.n_obs == 2) ? cx[at] : make_float2(0.f, 0.f);   // chat^(o1 o0)
    float s00 = 0.f, s11 = 0.f;
    float2 s01 = make_float2(0.f, 0.f);
    if (p.n_obs == 1) {
      s00 = quotient(a0, p.rhat_t[at], p.inv_G);
    } else {
      const Bracket k = bracket(a0, a1, b10, p.rhat_t[at], p.rhat_t[tab + at], p.inv_G);
      s00 = k.s00;
      s11 = k.s11;
      s01 = k.s01;
    }
    const float2 s10 = make_float2(s01.x, -s01.y);
    bad |= !(isfinite(s00) && isfinite(s11) && isfinite(s01.x) && isfinite(s01.y));
    // rows chat_{r,O}: observed o0 (a0, conj b10); observed o1 (b10, a1); unobserved u (x_0u, x_1u)
    for (int r = 0; r < p.n_obs + p.n_un; ++r) {
      float2 c0, c1 = make_float2(0.f, 0.f);
      if (r == 0) {
        c0 = make_float2(a0, 0.f);
        c1 = make_float2(b10.x, -b10.y);
      } else if (r == 1 && p.n_obs == 2) {
        c0 = b10;
        c1 = make_float2(a1, 0.f);
      } else {
        const int u = r - p.n_obs;
        c0 = cx[(size_t)(p.n_pair + u) * tab + at];
        if (p.n_obs == 2) c1 = cx[(size_t)(p.n_pair + p.n_un + u) * tab + at];
      }
      // K_{r,0} = c0 A^-1[0][0] + c1 A^-1[1][0], K_{r,1} = c0 A^-1[0][1] + c1 A^-1[1][1]
      const float2 k0 = cadd(cscale(c0, s00), cmul(c1, s10));
      p.gall[(size_t)r * p.n_obs * tab + at] = (p.n_obs == 2) ? k0 : cscale(c0, s00);
      if (p.n_obs == 2) p.gall[((size_t)r * 2 + 1) * tab + at] = cadd(cmul(c0, s01), cscale(c1, s11));
    }
  }
  if (bad) atomicOr(p.status, kStatusNonFinite);
}

cudaError_t launch_coupled_gain(const CoupledGainParams& p, cudaStream_t s) {
  const size_t tab = (size_t)(p.L + 1) * p.ny;
  long long blocks = (long long)((tab + 255) / 256);
  if (blocks > 8LL * sm_count()) blocks = 8LL * sm_count();
  coupled_gain_kernel<<<(unsigned)blocks, 256, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace fftenkf
