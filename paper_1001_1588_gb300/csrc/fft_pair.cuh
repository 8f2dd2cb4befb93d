// Line FFTs of two lines at once in paired FP32 arithmetic.
//
// Blackwell issues add/sub/mul/fma on two packed FP32 values (f32x2) at the
// issue cost of one scalar instruction.  A thread that transforms two lines a
// and b with the same plan holds each element as a "pair" {re = (a.re, b.re),
// im = (a.im, b.im)}: every butterfly add and multiply then becomes one
// paired instruction for both lines, multiplication by +-i is a renaming of
// re and im, and an exchange through shared memory moves both lines' element
// as one 16-byte access.  The schedule (canonical distribution: thread t owns
// elements t + T m, radix plan, Stockham stages, stage-major twiddle tables)
// and the twiddle tables are those of fft_core.cuh.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_core.cuh"

namespace fftenkf {

// ------------------------------------------------------------------ paired scalars
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) {
  unsigned long long A, B, D;
  __builtin_memcpy(&A, &a, 8);
  __builtin_memcpy(&B, &b, 8);
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(D) : "l"(A), "l"(B));
  float2 d;
  __builtin_memcpy(&d, &D, 8);
  return d;
}
__device__ __forceinline__ float2 p_bc(float s) { return make_float2(s, s); }

// one element of two lines
struct cp {
  float2 re, im;
};
__device__ __forceinline__ cp cp_add(cp a, cp b) { return {p_add(a.re, b.re), p_add(a.im, b.im)}; }
__device__ __forceinline__ cp cp_sub(cp a, cp b) { return {p_sub(a.re, b.re), p_sub(a.im, b.im)}; }
// a + s d and a - s d with s = -i (forward) or +i (INV)
template <bool INV>
__device__ __forceinline__ cp cp_add_rot(cp a, cp d) {
  return INV ? cp{p_sub(a.re, d.im), p_add(a.im, d.re)} : cp{p_add(a.re, d.im), p_sub(a.im, d.re)};
}
template <bool INV>
__device__ __forceinline__ cp cp_sub_rot(cp a, cp d) {
  return INV ? cp{p_add(a.re, d.im), p_sub(a.im, d.re)} : cp{p_sub(a.re, d.im), p_add(a.im, d.re)};
}
// 16-byte shared-memory form {a.re, b.re, a.im, b.im}
__device__ __forceinline__ float4 cp_pack(cp a) { return make_float4(a.re.x, a.re.y, a.im.x, a.im.y); }
__device__ __forceinline__ cp cp_unpack(float4 v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
// the pair of two separate complex values
__device__ __forceinline__ cp cp_of(float2 a, float2 b) { return {make_float2(a.x, b.x), make_float2(a.y, b.y)}; }
__device__ __forceinline__ float2 cp_a(cp v) { return make_float2(v.re.x, v.im.x); }
__device__ __forceinline__ float2 cp_b(cp v) { return make_float2(v.re.y, v.im.y); }

// ------------------------------------------------------------------ small DFTs
template <int R, bool INV> struct PDft;

template <bool INV> struct PDft<2, INV> {
  static __device__ __forceinline__ void run(cp* a) {
    const cp t = a[0];
    a[0] = cp_add(t, a[1]);
    a[1] = cp_sub(t, a[1]);
  }
};

template <bool INV> struct PDft<3, INV> {
  static __device__ __forceinline__ void run(cp* a) {
    const float2 h = p_bc(0.86602540378443864676f);   // sin(2 pi / 3)
    const float2 half = p_bc(0.5f);
    const cp s = cp_add(a[1], a[2]);
    const cp df = cp_sub(a[1], a[2]);
    const cp d = {p_mul(df.re, h), p_mul(df.im, h)};
    const cp m = {p_sub(a[0].re, p_mul(half, s.re)), p_sub(a[0].im, p_mul(half, s.im))};
    a[0] = cp_add(a[0], s);
    a[1] = cp_add_rot<INV>(m, d);
    a[2] = cp_sub_rot<INV>(m, d);
  }
};

template <bool INV> struct PDft<4, INV> {
  static __device__ __forceinline__ void run(cp* a) {
    const cp t0 = cp_add(a[0], a[2]), t1 = cp_sub(a[0], a[2]);
    const cp t2 = cp_add(a[1], a[3]), d = cp_sub(a[1], a[3]);
    a[0] = cp_add(t0, t2);
    a[2] = cp_sub(t0, t2);
    a[1] = cp_add_rot<INV>(t1, d);
    a[3] = cp_sub_rot<INV>(t1, d);
  }
};

struct PairOps {
  using C = cp;
  using S = float2;
  static __device__ __forceinline__ S re(const C& c) { return c.re; }
  static __device__ __forceinline__ S im(const C& c) { return c.im; }
  static __device__ __forceinline__ C mk(S r, S i) { return {r, i}; }
  static __device__ __forceinline__ S add(S a, S b) { return p_add(a, b); }
  static __device__ __forceinline__ S sub(S a, S b) { return p_sub(a, b); }
  static __device__ __forceinline__ S fma(float k, S a, S b) { return p_fma(p_bc(k), a, b); }
};
template <bool INV> struct PDft<8, INV> {
  static __device__ __forceinline__ void run(cp* a) { dft8<PairOps, INV>(a); }
};
template <bool INV> struct PDft<16, INV> {
  static __device__ __forceinline__ void run(cp* a) { dft16<PairOps, INV>(a); }
};

// ------------------------------------------------------------------ exchange layout
// 16-byte slots; one spare slot per 2^sh keeps the stride-R writes of the first
// stage (the only strided ones) on distinct bank quads: sh = 4 when the first
// radix is 16, else 3.
__host__ __device__ constexpr int pair_pad_shift(int N, int V) { return radix_at(N, V, 0) == 16 ? 4 : 3; }
__host__ __device__ constexpr int pair_padded_len(int N, int V) { return N + (N >> pair_pad_shift(N, V)); }
template <int SH>
__device__ __forceinline__ int ppidx(int i) { return i + (i >> SH); }

// ------------------------------------------------------------------ stages
// a w for one twiddle factor of both lines (4096^2, N=20: fused column pass 4.38 ms; with the twiddle powers
// formed as pairs too 4.56, with single multiplies 4.41)
__device__ __forceinline__ cp cp_mulw(cp a, float2 w) {
  return {p_fma(a.im, p_bc(-w.y), p_mul(a.re, p_bc(w.x))), p_fma(a.im, p_bc(w.x), p_mul(a.re, p_bc(w.y)))};
}

// As Stage in fft_core.cuh, for two lines.
template <int N, int V, int S, int NS, bool INV, bool TRAIL>
struct PStage {
  static __device__ __forceinline__ void run(cp (&v)[V], float4* sm, int t, const float2* __restrict__ tw, int bid) {
    constexpr int R = radix_at(N, V, S);
    constexpr int T = N / V;
    constexpr int B = V / R;
    constexpr int SH = pair_pad_shift(N, V);
    constexpr bool LAST = (S == num_stages(N, V) - 1);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      cp a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = v[b + r * B];
      const int j = t + T * b;
      if (NS > 1) {
        float2 w[R];
        twiddle_powers<R, INV, tw_every(N, V)>(w, tw + twiddle_offset(N, V, S, tw_every(N, V)) + (j % NS), NS);
#pragma unroll
        for (int r = 1; r < R; ++r) a[r] = cp_mulw(a[r], w[r]);
      }
      PDft<R, INV>::run(a);
      if (LAST) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[b + r * B] = a[r];
      } else {
        const int p = (j / NS) * NS * R + (j % NS);
#pragma unroll
        for (int r = 0; r < R; ++r) sm[ppidx<SH>(p + r * NS)] = cp_pack(a[r]);
      }
    }
    if constexpr (!LAST) {
      line_sync<T>(bid);
#pragma unroll
      for (int m = 0; m < V; ++m) v[m] = cp_unpack(sm[ppidx<SH>(t + T * m)]);
      if constexpr (TRAIL || S + 2 < num_stages(N, V)) line_sync<T>(bid);
      PStage<N, V, S + 1, NS * R, INV, TRAIL>::run(v, sm, t, tw, bid);
    }
  }
};

// As PStage, with the exchanges alternating between two buffers (even exchanges in sa, odd
// ones in sb), so that no barrier separates one exchange's reads from the next one's writes:
// a thread writes sb only after the barrier of the previous exchange, which every thread
// reaches after its last read of sb, and likewise for sa.  With an odd number of exchanges the
// last one is followed by a barrier, so that the next transform may start again in sa.
template <int N, int V, int S, int NS, bool INV>
struct PStage2 {
  static __device__ __forceinline__ void run(cp (&v)[V], float4* sa, float4* sb, int t, const float2* __restrict__ tw,
                                             int bid) {
    constexpr int R = radix_at(N, V, S);
    constexpr int T = N / V;
    constexpr int B = V / R;
    constexpr int SH = pair_pad_shift(N, V);
    constexpr bool LAST = (S == num_stages(N, V) - 1);
    float4* sm = (S % 2 == 0) ? sa : sb;
#pragma unroll
    for (int b = 0; b < B; ++b) {
      cp a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = v[b + r * B];
      const int j = t + T * b;
      if (NS > 1) {
        float2 w[R];
        twiddle_powers<R, INV, tw_every(N, V)>(w, tw + twiddle_offset(N, V, S, tw_every(N, V)) + (j % NS), NS);
#pragma unroll
        for (int r = 1; r < R; ++r) a[r] = cp_mulw(a[r], w[r]);
      }
      PDft<R, INV>::run(a);
      if (LAST) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[b + r * B] = a[r];
      } else {
        const int p = (j / NS) * NS * R + (j % NS);
#pragma unroll
        for (int r = 0; r < R; ++r) sm[ppidx<SH>(p + r * NS)] = cp_pack(a[r]);
      }
    }
    if constexpr (!LAST) {
      line_sync<T>(bid);
#pragma unroll
      for (int m = 0; m < V; ++m) v[m] = cp_unpack(sm[ppidx<SH>(t + T * m)]);
      if constexpr (S + 2 == num_stages(N, V) && (num_stages(N, V) - 1) % 2 == 1) line_sync<T>(bid);
      PStage2<N, V, S + 1, NS * R, INV>::run(v, sa, sb, t, tw, bid);
    }
  }
};

// Unnormalised DFT of two lines at once, sign -1 (forward) or +1 (INV); the
// calling conventions (bid, TRAIL, canonical distribution) are those of
// fft_line.  sm: the pair's buffer of pair_padded_len(N, V) 16-byte slots.
template <int N, int V, bool INV, bool TRAIL = true>
__device__ __forceinline__ void fft_pair(cp (&v)[V], float4* sm, int t, const float2* __restrict__ tw, int bid = 0) {
  static_assert(N % V == 0, "V must divide N");
  static_assert(num_stages(N, V) > 0, "no radix plan");
  PStage<N, V, 0, 1, INV, TRAIL>::run(v, sm, t, tw, bid);
}

// Two-buffer form (PStage2): each exchange takes one barrier.  Every thread of the line (bid)
// calls it; sa and sb hold pair_padded_len(N, V) slots each; on return both may be written
// again by the next transform's exchanges (which start in sa), but not by anything else
// before a barrier of the line.
template <int N, int V, bool INV>
__device__ __forceinline__ void fft_pair2(cp (&v)[V], float4* sa, float4* sb, int t, const float2* __restrict__ tw,
                                          int bid = 0) {
  static_assert(N % V == 0, "V must divide N");
  static_assert(num_stages(N, V) > 0, "no radix plan");
  PStage2<N, V, 0, 1, INV>::run(v, sa, sb, t, tw, bid);
}

}  // namespace fftenkf
