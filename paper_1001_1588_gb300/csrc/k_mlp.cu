// Learned spectral-variance denoiser: radial binning of log chat, a small MLP
// (256 -> 64 -> 64 -> 64 -> 128, exact GELU, BF16 weights, FP32 accumulation)
// with its backward pass and Adam update, and unbinning back to a
// per-wavenumber spectrum.  Parameters are one flat FP32 vector
// [W1 (64x256, out-major), b1, W2, b2, W3, b3, W4 (128x64), b4]; the forward
// and backward passes use their BF16 rounding (gradients are those of the
// BF16 network and are applied to the FP32 master copy).
#include <cuda_bf16.h>

#include <algorithm>

#include "common.cuh"
#include "dd.cuh"
#include "launch.cuh"

namespace fftenkf {

constexpr int kBins = 128;
constexpr int kIn = 256, kH = 64, kOut = 128;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH * kH, kOffW4 = kOffB3 + kH, kOffB4 = kOffW4 + kOut * kH,
              kParams = kOffB4 + kOut;

// ----------------------------------------------------------------- binning
// chat: [B][ny][L+1] f64 (one real table per sample); feat: [B][256] f32; mean: [B] f32.
// The bins are fixed per grid (FP64 decision, made on the host): bin_order lists the K1
// half-spectrum entries grouped by bin (ascending), bin_start[129] their offsets.  Each bin is
// cut into segments of at most kSegLen entries (seg_off[nseg+1], bin_seg[129] the segments of
// every bin), so that one spectrum spreads over many CTAs:
//   1. mlp_max_kernel: the maxima of chunks of every spectrum (floats >= 0);
//   2. mlp_binsum_kernel: one CTA per (segment, sample) takes cmax over the chunks and sums
//      log(max(c / cmax, 1e-30));
//   3. per bin the segment sums in segment order, mean log + log cmax, the features: mlp_binfin_kernel,
//      or the head of the network (mlp_head_kernel) for one spectrum.
// log(max(c, 1e-30 cmax)) is evaluated as log(max(c/cmax, 1e-30)) + log(cmax) so that the floor
// never underflows; one conversion to float per entry.  No floating-point atomics: the result
// does not depend on the schedule.
constexpr int kSegLen = 2048;

__device__ __forceinline__ float block_sum256(float v, float* red8) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red8[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x == 0)
#pragma unroll
    for (int w = 0; w < 8; ++w) t += red8[w];
  return t;   // valid in thread 0
}

struct MlpBinParams {
  const double* chat;   // [B][K1]
  MlpBins bins;
  float* feat;          // [B][256]
  float* mean;          // [B]
};

// grid (chunks, B): cmax[smp][chunk], the largest entry of the chunk or 0 (NaN entries are ignored)
__global__ void __launch_bounds__(256) mlp_max_kernel(const MlpBinParams p) {
  __shared__ float red8[8];
  const double* c = p.chat + (size_t)blockIdx.y * p.bins.K1;
  stream_order_wait();
  next_may_start();
  float mx = 0.f;
#pragma unroll 4
  for (int i = blockIdx.x * 256 + threadIdx.x; i < p.bins.K1; i += gridDim.x * 256) mx = fmaxf(mx, to_float(c[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) red8[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = fmaxf(m, red8[w]);
    p.bins.cmax[(size_t)blockIdx.y * p.bins.chunks + blockIdx.x] = m;
  }
}

// cmax of one sample over its chunks by the first warp (1 where no entry is positive), to every thread
// of the CTA through *sh
__device__ __forceinline__ float cmax_of(const MlpBins& t, int smp, float* sh) {
  if (threadIdx.x < 32) {
    float m = 0.f;
    for (int i = threadIdx.x; i < t.chunks; i += 32) m = fmaxf(m, t.cmax[(size_t)smp * t.chunks + i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) *sh = m > 0.f ? m : 1.f;
  }
  __syncthreads();
  return *sh;
}

// grid (nseg, B): part[smp][seg] = sum over the segment of log(max(c / cmax, 1e-30))
__global__ void __launch_bounds__(256) mlp_binsum_kernel(const MlpBinParams p) {
  __shared__ float red8[8];
  __shared__ float cm;
  const uint32_t i0 = __ldg(p.bins.seg_off + blockIdx.x), i1 = __ldg(p.bins.seg_off + blockIdx.x + 1);
  constexpr int E = kSegLen / 256;
  uint32_t at[E];   // the entries of this thread, requested before the spectrum may be read
#pragma unroll
  for (int e = 0; e < E; ++e) at[e] = i0 + threadIdx.x + 256 * e < i1 ? __ldg(p.bins.order + i0 + threadIdx.x + 256 * e) : ~0u;
  stream_order_wait();
  next_may_start();
  const double* c = p.chat + (size_t)blockIdx.y * p.bins.K1;
  float v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) v[e] = at[e] != ~0u ? to_float(c[at[e]]) : 0.f;
  const float inv = 1.f / cmax_of(p.bins, blockIdx.y, &cm);
  float acc = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e)
    if (at[e] != ~0u) acc += logf(fmaxf(v[e] * inv, 1e-30f));
  const float t = block_sum256(acc, red8);
  if (threadIdx.x == 0) p.bins.part[(size_t)blockIdx.y * p.bins.nseg + blockIdx.x] = t;
}

// Per-bin means of one sample from its segment sums (in segment order), by the first 128 threads of the
// CTA: features [binned - mu | centre_log] to feat, returns their mean mu to every thread.
__device__ __forceinline__ float bin_features(const MlpBins& t, int smp, float* feat, float* red4, float* sh) {
  const float lmax = logf(cmax_of(t, smp, sh));
  const int b = threadIdx.x;
  float v = 0.f;
  if (b < kBins) {
    const float* ps = t.part + (size_t)smp * t.nseg;
    float acc = 0.f;
    for (uint32_t sg = t.bin_seg[b]; sg < t.bin_seg[b + 1]; ++sg) acc += ps[sg];
    const uint32_t n = t.start[b + 1] - t.start[b];
    v = n ? acc / (float)n + lmax : 0.f;
    float s = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((b & 31) == 0) red4[b >> 5] = s;
  }
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < kBins / 32; ++w) tot += red4[w];
  const float mu = tot / kBins;
  if (b < kBins) {
    feat[b] = v - mu;
    feat[kBins + b] = t.centre_log[b];
  }
  __syncthreads();
  return mu;
}

// grid B
__global__ void __launch_bounds__(kBins) mlp_binfin_kernel(const MlpBinParams p) {
  __shared__ float red4[kBins / 32];
  __shared__ float cm;
  stream_order_wait();
  next_may_start();
  const int smp = blockIdx.x;
  const float mu = bin_features(p.bins, smp, p.feat + (size_t)smp * kIn, red4, &cm);
  if (threadIdx.x == 0) p.mean[smp] = mu;
}

// out_log: [128] learned binned log spectrum (mean already added); chat_out: [ny][L+1] f64, chat_in itself
// where the network output is not finite (*flag)
struct MlpUnbinParams {
  const float* out_log;
  const int* flag;
  const double* chat_in;
  double* chat_out;
  int ny, L;
  float w;
};
__global__ void __launch_bounds__(256) mlp_unbin_kernel(const MlpUnbinParams p) {
  const int K1 = p.ny * (p.L + 1);
  stream_order_wait();
  next_may_start();
  const bool plain = *p.flag != 0;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < K1; i += gridDim.x * 256) {
    if (plain) {
      p.chat_out[i] = p.chat_in[i];
      continue;
    }
    const int ky = i / (p.L + 1), kx = i - ky * (p.L + 1);
    const int kyv = (ky <= p.ny / 2) ? ky : ky - p.ny;
    const float kabs = sqrtf((float)(kyv * kyv + kx * kx));
    const float pos = kabs / p.w - 0.5f;   // position in units of bins relative to centre 0
    float v;
    if (pos <= 0.f) {
      v = p.out_log[0];
    } else if (pos >= kBins - 1) {
      v = p.out_log[kBins - 1];
    } else {
      const int b = (int)pos;
      const float fr = pos - b;
      v = p.out_log[b] + fr * (p.out_log[b + 1] - p.out_log[b]);
    }
    p.chat_out[i] = to_double(expf(v));
  }
}

// ----------------------------------------------------------------- MLP
__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}
__device__ __forceinline__ float bf16_round(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// four consecutive floats; vec: p is 16-byte aligned (the caller's arrays need only be 4-byte aligned)
__device__ __forceinline__ float4 load4(const float* p, bool vec) {
  if (vec) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}
__device__ __forceinline__ void add4(float* p, float4 v, bool vec) {
  if (vec) {
    atomicAdd(reinterpret_cast<float4*>(p), v);
  } else {
    atomicAdd(p, v.x);
    atomicAdd(p + 1, v.y);
    atomicAdd(p + 2, v.z);
    atomicAdd(p + 3, v.w);
  }
}

// Sums of S values over the 32 lanes (S = 1, 4 or 8): the halves of the values are exchanged along
// with the halves of the lanes, so that S sums take S - 1 + log2(32 / S) shuffles instead of 5 S.  Returns the
// sum of value lane_sample<S>(lane).
template <int S>
__device__ __forceinline__ float warp_sums(float (&a)[S], int lane) {
  int o = 16;
#pragma unroll
  for (int n = S; n > 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < n / 2; ++j) {
      const float mine = up ? a[j + n / 2] : a[j], other = up ? a[j] : a[j + n / 2];
      a[j] = mine + __shfl_xor_sync(0xffffffffu, other, o);
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
  return a[0];
}
template <int S>
__device__ __forceinline__ int lane_sample(int lane) { return lane / (32 / S); }

// Activations of S samples: inputs, pre-activations and activations of the hidden layers, outputs.
template <int S>
struct alignas(16) MlpActs {
  float x[S][kIn];
  float z[3][S][kH];
  float h[3][S][kH];
  float out[S][kOut];
};

// One dense layer of the CTA's samples, z[s][o] = b[o] + sum_i W[o][i] in[s][i]: a warp per output,
// the inputs over its lanes (every weight row is read once, coalesced, straight from L2 and the inputs
// stay in registers), so neither weights nor inputs go through shared memory per product.
template <int S, int NW, int IN, int OUT, bool HIDDEN>
__device__ __forceinline__ void mlp_layer(const float* W, const float* b, bool vec,
                                          const float* in, float* z, float* h, int warp, int lane) {
  constexpr int Q = IN / 128;   // float4 per lane (0: a pair of floats)
  constexpr int E = Q ? 4 * Q : 2;
  float xr[S][E];
#pragma unroll
  for (int s = 0; s < S; ++s)
#pragma unroll
    for (int e = 0; e < E; ++e) xr[s][e] = in[s * IN + (Q ? 128 * (e / 4) + 4 * lane + e % 4 : 2 * lane + e)];
#pragma unroll (S == 1 ? OUT / NW : 2)
  for (int o = warp; o < OUT; o += NW) {
    float w[E];
    if constexpr (Q > 0) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const float4 v = load4(W + o * IN + 128 * q + 4 * lane, vec);
        w[4 * q] = v.x; w[4 * q + 1] = v.y; w[4 * q + 2] = v.z; w[4 * q + 3] = v.w;
      }
    } else {
      w[0] = W[o * IN + 2 * lane];
      w[1] = W[o * IN + 2 * lane + 1];
    }
    float acc[S];
#pragma unroll
    for (int s = 0; s < S; ++s) acc[s] = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const float we = bf16_round(w[e]);
#pragma unroll
      for (int s = 0; s < S; ++s) acc[s] = fmaf(we, xr[s][e], acc[s]);
    }
    const float v = warp_sums<S>(acc, lane) + b[o];
    if (lane % (32 / S) == 0) {
      const int s = lane_sample<S>(lane);
      z[s * OUT + o] = v;
      if constexpr (HIDDEN) h[s * OUT + o] = gelu(v);
    }
  }
  __syncthreads();
}

template <int S, int NW>
__device__ __forceinline__ void mlp_forward(MlpActs<S>& a, const float* p, bool vec, int warp, int lane) {
  mlp_layer<S, NW, kIn, kH, true>(p + kOffW1, p + kOffB1, vec, &a.x[0][0], &a.z[0][0][0], &a.h[0][0][0], warp, lane);
  mlp_layer<S, NW, kH, kH, true>(p + kOffW2, p + kOffB2, vec, &a.h[0][0][0], &a.z[1][0][0], &a.h[1][0][0], warp, lane);
  mlp_layer<S, NW, kH, kH, true>(p + kOffW3, p + kOffB3, vec, &a.h[1][0][0], &a.z[2][0][0], &a.h[2][0][0], warp, lane);
  mlp_layer<S, NW, kH, kOut, false>(p + kOffW4, p + kOffB4, vec, &a.h[2][0][0], &a.out[0][0], nullptr, warp, lane);
}

template <int S>
__device__ __forceinline__ void load_samples(MlpActs<S>& a, const float* X, int s0, int nsamp, int threads) {
  for (int i = threadIdx.x; i < S * kIn; i += threads) a.x[i / kIn][i % kIn] = i / kIn < nsamp ? X[(size_t)s0 * kIn + i] : 0.f;
  __syncthreads();
}

struct MlpFwdParams {
  const float* params;
  const float* X;       // [B][256]
  float* out;           // [B][128]
  int B;
};
template <int S, int NW>
__global__ void __launch_bounds__(32 * NW) mlp_fwd_kernel(const MlpFwdParams p) {
  __shared__ MlpActs<S> a;
  const int s0 = blockIdx.x * S, nsamp = min(S, p.B - s0);
  const bool vec = (reinterpret_cast<uintptr_t>(p.params) & 15) == 0;
  stream_order_wait();
  next_may_start();
  load_samples<S>(a, p.X, s0, nsamp, 32 * NW);
  mlp_forward<S, NW>(a, p.params, vec, threadIdx.x >> 5, threadIdx.x & 31);
  for (int i = threadIdx.x; i < nsamp * kOut; i += 32 * NW) p.out[(size_t)s0 * kOut + i] = a.out[i / kOut][i % kOut];
}

struct MlpGradParams {
  const float* params;
  const float* X;        // [B][256]
  const float* target;   // [B][128]
  float* grads;
  float* loss;
  int B;
};
__global__ void __launch_bounds__(256) mlp_zero_kernel(const MlpGradParams p) {
  stream_order_wait();
  next_may_start();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < kParams) p.grads[i] = 0.f;
  if (i == 0) *p.loss = 0.f;
}

// Weight and bias gradients of one layer, summed over the CTA's samples and added to grads (four
// consecutive weights of one output per atomic): d [OUT][S] the deltas, a [S][IN] the input activations.
template <int S, int IN, int OUT>
__device__ __forceinline__ void mlp_weight_grads(float* g, float* gb, bool vec, const float* d, const float* a, int tid) {
  constexpr int QI = IN / 4, OG = 256 / QI;   // quads of inputs, groups of outputs
  const int q = tid % QI, og = tid / QI;
  float4 ar[S];
#pragma unroll
  for (int s = 0; s < S; ++s) ar[s] = *reinterpret_cast<const float4*>(a + s * IN + 4 * q);
#pragma unroll 4
  for (int o = og; o < OUT; o += OG) {
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const float ds = d[o * S + s];
      w.x = fmaf(ds, ar[s].x, w.x);
      w.y = fmaf(ds, ar[s].y, w.y);
      w.z = fmaf(ds, ar[s].z, w.z);
      w.w = fmaf(ds, ar[s].w, w.w);
    }
    add4(g + o * IN + 4 * q, w, vec);
  }
  if (tid < OUT) {
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < S; ++k) s += d[tid * S + k];
    atomicAdd(gb + tid, s);
  }
}

// Deltas of the layer below, dn[i][s] = gelu'(z[s][i]) sum_o W[o][i] d[o][s] (64 inputs): a thread per
// input and quarter of the outputs, the quarters added through part [4][64][S].
template <int S, int OUT>
__device__ __forceinline__ void mlp_delta(const float* W, const float* d, const float* z, float* part,
                                          float* dn, int tid) {
  const int i = tid & 63, og = tid >> 6;
  float acc[S];
#pragma unroll
  for (int s = 0; s < S; ++s) acc[s] = 0.f;
#pragma unroll 8
  for (int o = og * (OUT / 4); o < (og + 1) * (OUT / 4); ++o) {
    const float w = bf16_round(W[o * kH + i]);
#pragma unroll
    for (int s = 0; s < S; ++s) acc[s] = fmaf(w, d[o * S + s], acc[s]);
  }
#pragma unroll
  for (int s = 0; s < S; ++s) part[(og * kH + i) * S + s] = acc[s];
  __syncthreads();
  for (int k = tid; k < kH * S; k += 256) {
    const int ii = k / S, s = k - ii * S;
    dn[k] = (part[k] + part[kH * S + k] + part[2 * kH * S + k] + part[3 * kH * S + k]) * gelu_grad(z[s * kH + ii]);
  }
  __syncthreads();
}

// Back-propagation of the CTA's samples from the output deltas in d0
template <int S>
__device__ __forceinline__ void mlp_gradients(const MlpGradParams& p, const MlpActs<S>& a, float* d0, float* d1, float* part,
                                              bool gvec, int tid) {
  mlp_weight_grads<S, kH, kOut>(p.grads + kOffW4, p.grads + kOffB4, gvec, d0, &a.h[2][0][0], tid);
  mlp_delta<S, kOut>(p.params + kOffW4, d0, &a.z[2][0][0], part, d1, tid);
  mlp_weight_grads<S, kH, kH>(p.grads + kOffW3, p.grads + kOffB3, gvec, d1, &a.h[1][0][0], tid);
  mlp_delta<S, kH>(p.params + kOffW3, d1, &a.z[1][0][0], part, d0, tid);
  mlp_weight_grads<S, kH, kH>(p.grads + kOffW2, p.grads + kOffB2, gvec, d0, &a.h[0][0][0], tid);
  mlp_delta<S, kH>(p.params + kOffW2, d0, &a.z[0][0][0], part, d1, tid);
  mlp_weight_grads<S, kIn, kH>(p.grads + kOffW1, p.grads + kOffB1, gvec, d1, &a.x[0][0], tid);
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// *x of the cluster's first CTA = v
__device__ __forceinline__ void store_to_first(float* x, float v) {
  uint32_t at;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(x)));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(at), "f"(v) : "memory");
}

// Gradient of mean((out - target)^2) over all B x 128 outputs: forward pass of S samples per CTA, then
// back-propagation; grads and loss zeroed before.  At this size the work is a chain of short phases, so
// what counts is latency and conflict-free operand access: batch 256 took 60 us with the weights staged in shared
// memory (32-way bank conflicts of the row-major weights), 8 samples per CTA and scalar atomics; a gradient
// and Adam step of that batch went from 71.9 to 29.2 us (26.9 without the pairs below).
//
// The losses of the CTAs are added in FP32 in free order, with an error that grows with their number.  CTAs of four
// samples come in clusters of two, which add their losses first (through the pair's distributed shared memory), so
// that as many terms are added as with eight samples per CTA.  (Relative error against 64 bits, root mean square over
// 24 batches: of 600 samples 2.1e-7 without, 1.5e-7 like this, 1.2e-7 the first kernel above; of 256 1.0e-7, 0.6e-7 and
// 0.8e-7.  The gradients of 256 are 1.7e-7 off, 1.5e-7 with eight samples per CTA, 2.8e-7 with the first kernel.)
template <int S>
__global__ void __launch_bounds__(256) mlp_bwd_kernel(const MlpGradParams p) {
  constexpr bool PAIR = S == 4;   // launched in clusters of two
  __shared__ MlpActs<S> a;
  __shared__ alignas(16) float d0[kOut * S];
  __shared__ alignas(16) float d1[kH * S];
  __shared__ float part[4 * kH * S];
  __shared__ float red8[8];
  __shared__ float partner;   // the second CTA's loss, in the first
  const int s0 = blockIdx.x * S, nsamp = min(S, p.B - s0), tid = threadIdx.x;   // nsamp <= 0: completes a pair
  const bool vec = (reinterpret_cast<uintptr_t>(p.params) & 15) == 0;
  const bool gvec = (reinterpret_cast<uintptr_t>(p.grads) & 15) == 0;
  stream_order_wait();
  next_may_start();
  if constexpr (PAIR) cluster_arrive();
  load_samples<S>(a, p.X, s0, nsamp, 256);
  mlp_forward<S, 8>(a, p.params, vec, tid >> 5, tid & 31);
  const float scale = 2.f / ((float)p.B * kOut);
  float l = 0.f;
  for (int k = tid; k < S * kOut; k += 256) {
    const int s = k / kOut, o = k - s * kOut;
    const float diff = s < nsamp ? a.out[s][o] - p.target[(size_t)(s0 + s) * kOut + o] : 0.f;
    l += diff * diff;
    d0[o * S + s] = scale * diff;
  }
  const float t = block_sum256(l, red8);   // holds a barrier: d0 is complete after it
  if constexpr (PAIR) {
    cluster_wait();   // both CTAs have started
    if (tid == 0 && cluster_rank() == 1) store_to_first(&partner, t);
    cluster_arrive();
  } else {
    if (tid == 0) atomicAdd(p.loss, t / ((float)p.B * kOut));
  }
  if (nsamp > 0) mlp_gradients<S>(p, a, d0, d1, part, gvec, tid);
  if constexpr (PAIR) {
    cluster_wait();   // the partner's loss has arrived
    if (tid == 0 && cluster_rank() == 0) atomicAdd(p.loss, (t + partner) / ((float)p.B * kOut));
  }
}

struct MlpAdamParams {
  float *params, *m, *v;
  const float* g;
  float lr, b1, b2, eps, c1, c2;
};
__global__ void __launch_bounds__(256) mlp_adam_kernel(const MlpAdamParams p) {
  stream_order_wait();
  next_may_start();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= kParams) return;
  const float gi = p.g[i];
  const float mi = p.b1 * p.m[i] + (1.f - p.b1) * gi;
  const float vi = p.b2 * p.v[i] + (1.f - p.b2) * gi * gi;
  p.m[i] = mi;
  p.v[i] = vi;
  p.params[i] -= p.lr * (mi / p.c1) / (sqrtf(vi / p.c2) + p.eps);
}

// The learned spectrum's middle: bin means of one spectrum, the network, out + mean; flag = 1 if any
// value is not finite.  One CTA of 32 warps (a warp per output): the chain bin means -> four layers is
// latency; as three kernels it took 24.8 + 3.0 + 1.8 us.  With it, the maxima without a memset, and the
// fallback inside the unbinning, the learned analysis of 1024^2, N=5 went from 185 to 135 us.
struct MlpHeadParams {
  MlpBins bins;
  const float* params;
  float* out_log;       // [128]
  int* flag;
};
__global__ void __launch_bounds__(1024) mlp_head_kernel(const MlpHeadParams p) {
  __shared__ MlpActs<1> a;
  __shared__ float red4[kBins / 32];
  __shared__ float cm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool vec = (reinterpret_cast<uintptr_t>(p.params) & 15) == 0;
  stream_order_wait();
  next_may_start();
  const float mu = bin_features(p.bins, 0, &a.x[0][0], red4, &cm);
  mlp_forward<1, 32>(a, p.params, vec, warp, lane);
  bool bad = false;
  if (tid < kOut) {
    const float v = a.out[0][tid] + mu;
    p.out_log[tid] = v;
    bad = !isfinite(v);
  }
  const int any = __syncthreads_or(bad);
  if (tid == 0) *p.flag = any;
}

// ----------------------------------------------------------------- launchers
int mlp_param_count() { return kParams; }

int mlp_seg_len() { return kSegLen; }
// chunks of the maximum of one spectrum of K1 entries (at most mlp_max_chunks())
int mlp_max_chunks() { return 1024; }
int mlp_chunks(int K1) { return std::max(1, std::min((K1 + 1023) / 1024, mlp_max_chunks())); }

static cudaError_t launch_bin_sums(const MlpBinParams& p, int nb, cudaStream_t s) {
  cudaError_t e = launch_overlapped(mlp_max_kernel, dim3(p.bins.chunks, nb), 256, 0, s, p);
  if (e == cudaSuccess) e = launch_overlapped(mlp_binsum_kernel, dim3(p.bins.nseg, nb), 256, 0, s, p);
  return e;
}

// Features of B spectra in slices of at most max_batch samples (the scratch: cmax [max_batch][chunks],
// part [max_batch][nseg]).
cudaError_t launch_mlp_bin(const double* chat, const MlpBins& t, int B, float* feat, float* mean, cudaStream_t s) {
  for (int b0 = 0; b0 < B; b0 += t.max_batch) {
    const int nb = std::min(t.max_batch, B - b0);
    MlpBinParams p{chat + (size_t)b0 * t.K1, t, feat + (size_t)b0 * kIn, mean + b0};
    cudaError_t e = launch_bin_sums(p, nb, s);
    if (e == cudaSuccess) e = launch_overlapped(mlp_binfin_kernel, dim3(nb), kBins, 0, s, p);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// chat_in -> bins -> network -> chat_out (chat_in where the network output is not finite; *flag says so)
cudaError_t launch_mlp_denoise(const double* chat_in, const MlpBins& t, const float* params, float* out_log, int* flag,
                               double* chat_out, int ny, int L, float w, cudaStream_t s) {
  MlpBinParams p{chat_in, t, nullptr, nullptr};
  cudaError_t e = launch_bin_sums(p, 1, s);
  if (e == cudaSuccess) e = launch_overlapped(mlp_head_kernel, dim3(1), 1024, 0, s, MlpHeadParams{t, params, out_log, flag});
  if (e != cudaSuccess) return e;
  int grid = (t.K1 + 255) / 256;
  if (grid > 4096) grid = 4096;
  return launch_overlapped(mlp_unbin_kernel, dim3(grid), 256, 0, s, MlpUnbinParams{out_log, flag, chat_in, chat_out, ny, L, w});
}

cudaError_t launch_mlp_forward(const float* params, const float* X, int B, float* out, cudaStream_t s) {
  const MlpFwdParams p{params, X, out, B};
  // a sample per CTA of 32 warps up to two such CTAs per SM (batch 304: 8.0 us, 20.7 with eight samples per CTA)
  if (B <= 304) return launch_overlapped(mlp_fwd_kernel<1, 32>, dim3(B), 1024, 0, s, p);
  return launch_overlapped(mlp_fwd_kernel<8, 8>, dim3((B + 7) / 8), 256, 0, s, p);
}

// 4 samples per CTA, in pairs, up to one CTA per SM of a 152-SM GPU (with Adam, batch 256: 29.2 us, 31.4 with 8), then
// 8 (half the atomics)
cudaError_t launch_mlp_gradient(const float* params, const float* X, const float* target, int B, float* grads,
                                float* loss, cudaStream_t s) {
  const MlpGradParams p{params, X, target, grads, loss, B};
  cudaError_t e = launch_overlapped(mlp_zero_kernel, dim3((kParams + 255) / 256), 256, 0, s, p);
  if (e != cudaSuccess) return e;
  if (B <= 608) return launch_overlapped(mlp_bwd_kernel<4>, dim3(2 * ((B + 7) / 8)), 256, 0, s, p, 2);
  return launch_overlapped(mlp_bwd_kernel<8>, dim3((B + 7) / 8), 256, 0, s, p);
}

cudaError_t launch_mlp_adam(float* params, float* m, float* v, const float* g, int step, float lr, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  const MlpAdamParams p{params, m, v, g, lr, b1, b2, 1e-8f, c1, c2};
  return launch_overlapped(mlp_adam_kernel, dim3((kParams + 255) / 256), 256, 0, s, p);
}

}  // namespace fftenkf
