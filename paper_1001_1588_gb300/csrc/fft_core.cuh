// Register/shared-memory FFT of one line, the building block of every pass.
//
// A line of N complex values (N = 2^a or 3*2^a) is transformed by T = N/V
// threads.  Data is held in the "canonical" distribution: thread t owns
// elements t + T*m in register slot m (m < V), both on input and on output,
// so a line is loaded from and stored to global memory with unit-stride,
// fully coalesced warp accesses, and a forward transform's output can feed an
// inverse transform without any exchange.  Between radix stages the values go
// through a padded shared-memory line buffer (Stockham self-sorting order), so
// no bit reversal is needed.  Radices are 24, 16, 12, 8, 6, 4, 3 and 2; the plan is fixed
// at compile time from (N, V).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fftenkf {

// ------------------------------------------------------------------ complex
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {  // a * conj(b)
  return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// multiply by -i (forward sign) or +i (inverse sign)
template <bool INV>
__device__ __forceinline__ float2 rot90(float2 a) {
  return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// ------------------------------------------------------------------ plan
// Radix of the next stage of a line with `rem` left, V values per thread.  3 * 2^a lines take the factor
// 3 together with a power of two (radices 6, 12 and 24), so that it costs no exchange of its own: 24
// first, where it leaves stages of 8 and at most one of 4, otherwise last as 6 (384 = 8 8 6; V = 12:
// 12 first or 6 last, as the power of two is even or odd).
__host__ __device__ constexpr int pick_radix(int rem, int V) {
  return (V == 24 && (rem == 24 || rem == 96 || rem == 192 || rem == 768 || rem == 1536)) ? 24
       : (V == 24 && rem == 6)          ? 6
       : (V == 12 && (rem == 12 || rem == 48 || rem == 192 || rem == 768 || rem == 3072)) ? 12
       : (V == 12 && rem == 6)          ? 6
       : (rem % 16 == 0 && V % 16 == 0) ? 16
       : (rem % 8 == 0 && V % 8 == 0)   ? 8
       : (rem % 4 == 0 && V % 4 == 0)   ? 4
       : (rem % 2 == 0 && V % 2 == 0)   ? 2
       : (rem % 3 == 0 && V % 3 == 0)   ? 3
                                        : 0;
}
__host__ __device__ constexpr int radix_at(int N, int V, int s) {
  int rem = N;
  for (int i = 0; i < s; ++i) rem /= pick_radix(rem, V);
  return rem == 1 ? 1 : pick_radix(rem, V);
}
__host__ __device__ constexpr int num_stages(int N, int V) {
  int rem = N, s = 0;
  while (rem > 1) {
    int r = pick_radix(rem, V);
    if (r == 0) return -1;
    rem /= r;
    ++s;
  }
  return s;
}
// default values per thread: 16 for powers of two, 24 (or N) for 3*2^a
__host__ __device__ constexpr int default_V(int N) {
  return (N % 3 == 0) ? (N >= 24 ? 24 : N) : (N >= 16 ? 16 : N);
}
// values per thread of schedule `sel`: 0 = wide (radix 16 / 8-3), 1 = narrow (radix 8 / 4-3):
// twice the threads per line, one more exchange
__host__ __device__ constexpr int plan_V(int N, int sel) {
  return sel == 0 ? default_V(N) : ((N % 3 == 0) ? (N >= 12 ? 12 : N) : (N >= 8 ? 8 : N));
}
// padded shared-memory index: one spare slot per 16 keeps stride-R writes
// of the Stockham stages on distinct 8-byte banks
__device__ __forceinline__ int pidx(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int padded_len(int N) { return N + N / 16; }
// slots of a column pass's line buffer: a padded line rounded up to 16 slots (128 bytes)
__host__ __device__ constexpr int col_line_slots(int N) { return (padded_len(N) + 15) & ~15; }
// pitch of the staged rows of the row passes: a padded line rounded to 2 (mod 8) slots, so
// that reading two rows x four columns per half-warp hits 16 distinct 8-byte banks
__host__ __device__ constexpr int row_pitch(int N) { return padded_len(N) + ((10 - padded_len(N) % 8) % 8); }

// ------------------------------------------------------------------ small DFTs
// Forward kernels use exp(-2 pi i / R); INV uses exp(+2 pi i / R).
template <int R, bool INV> struct Dft;

template <bool INV> struct Dft<2, INV> {
  static __device__ __forceinline__ void run(float2* a) {
    float2 t = a[0];
    a[0] = cadd(t, a[1]);
    a[1] = csub(t, a[1]);
  }
};

template <bool INV> struct Dft<3, INV> {
  static __device__ __forceinline__ void run(float2* a) {
    const float h = 0.86602540378443864676f;  // sin(2 pi / 3)
    float2 s = cadd(a[1], a[2]);
    float2 d = cscale(csub(a[1], a[2]), h);
    float2 m = make_float2(a[0].x - 0.5f * s.x, a[0].y - 0.5f * s.y);
    a[0] = cadd(a[0], s);
    float2 rd = rot90<INV>(d);       // -i d (forward)
    a[1] = cadd(m, rd);
    a[2] = csub(m, rd);
  }
};

template <bool INV> struct Dft<4, INV> {
  static __device__ __forceinline__ void run(float2* a) {
    float2 t0 = cadd(a[0], a[2]), t1 = csub(a[0], a[2]);
    float2 t2 = cadd(a[1], a[3]), t3 = rot90<INV>(csub(a[1], a[3]));
    a[0] = cadd(t0, t2);
    a[2] = csub(t0, t2);
    a[1] = cadd(t1, t3);
    a[3] = csub(t1, t3);
  }
};

// The 8- and 16-point DFTs, written once for one line (complex float2) and for two at a time (fft_pair.cuh).
// Rotations by odd multiples of pi/8 are taken as a scale times a shear (cos a (1 - i tan a)), and every scale goes
// into the fused multiply-adds of the butterfly that follows: 144 operations for 16 points (161 with the
// rotations as products), 52 for 8.
struct LineOps {
  using C = float2;
  using S = float;
  static __device__ __forceinline__ S re(const C& c) { return c.x; }
  static __device__ __forceinline__ S im(const C& c) { return c.y; }
  static __device__ __forceinline__ C mk(S r, S i) { return make_float2(r, i); }
  static __device__ __forceinline__ S add(S a, S b) { return a + b; }
  static __device__ __forceinline__ S sub(S a, S b) { return a - b; }
  static __device__ __forceinline__ S fma(float k, S a, S b) { return fmaf(k, a, b); }
};
template <class O> __device__ __forceinline__ typename O::C c_add(typename O::C a, typename O::C b) {
  return O::mk(O::add(O::re(a), O::re(b)), O::add(O::im(a), O::im(b)));
}
template <class O> __device__ __forceinline__ typename O::C c_sub(typename O::C a, typename O::C b) {
  return O::mk(O::sub(O::re(a), O::re(b)), O::sub(O::im(a), O::im(b)));
}
// a + k d
template <class O> __device__ __forceinline__ typename O::C c_fma(float k, typename O::C d, typename O::C a) {
  return O::mk(O::fma(k, O::re(d), O::re(a)), O::fma(k, O::im(d), O::im(a)));
}
// a + k s d, s = -i (forward) or +i (INV)
template <class O, bool INV>
__device__ __forceinline__ typename O::C c_fma_rot(float k, typename O::C d, typename O::C a) {
  return INV ? O::mk(O::fma(-k, O::im(d), O::re(a)), O::fma(k, O::re(d), O::im(a)))
             : O::mk(O::fma(k, O::im(d), O::re(a)), O::fma(-k, O::re(d), O::im(a)));
}
template <class O, bool INV>
__device__ __forceinline__ typename O::C c_add_rot(typename O::C a, typename O::C d) {
  return INV ? O::mk(O::sub(O::re(a), O::im(d)), O::add(O::im(a), O::re(d)))
             : O::mk(O::add(O::re(a), O::im(d)), O::sub(O::im(a), O::re(d)));
}
template <class O, bool INV>
__device__ __forceinline__ typename O::C c_sub_rot(typename O::C a, typename O::C d) {
  return c_add_rot<O, !INV>(a, d);
}
template <class O, bool INV>
__device__ __forceinline__ void dft4(typename O::C& a0, typename O::C& a1, typename O::C& a2, typename O::C& a3) {
  using C = typename O::C;
  const C t0 = c_add<O>(a0, a2), t1 = c_sub<O>(a0, a2), t2 = c_add<O>(a1, a3), d = c_sub<O>(a1, a3);
  a0 = c_add<O>(t0, t2);
  a2 = c_sub<O>(t0, t2);
  a1 = c_add_rot<O, INV>(t1, d);
  a3 = c_sub_rot<O, INV>(t1, d);
}
// v exp(-+ i pi/4) sqrt(2)
template <class O, bool INV> __device__ __forceinline__ typename O::C c_eighth(typename O::C v) {
  return c_add_rot<O, INV>(v, v);
}
template <class O, bool INV>
__device__ __forceinline__ void dft8(typename O::C* a) {
  using C = typename O::C;
  constexpr float c = 0.70710678118654752440f;
  dft4<O, INV>(a[0], a[2], a[4], a[6]);
  dft4<O, INV>(a[1], a[3], a[5], a[7]);
  const C e0 = a[0], e1 = a[2], e2 = a[4], e3 = a[6], o0 = a[1], o1 = c_eighth<O, INV>(a[3]), o2 = a[5], v = a[7];
  a[0] = c_add<O>(e0, o0);
  a[4] = c_sub<O>(e0, o0);
  a[1] = c_fma<O>(c, o1, e1);
  a[5] = c_fma<O>(-c, o1, e1);
  a[2] = c_add_rot<O, INV>(e2, o2);
  a[6] = c_sub_rot<O, INV>(e2, o2);
  // exp(-+ 3 i pi/4) v: forward c (im - re, -(re + im)), inverse c (-(re + im), re - im)
  const typename O::S s = O::add(O::re(v), O::im(v)), d = O::sub(O::im(v), O::re(v));
  if (INV) {
    a[3] = O::mk(O::fma(-c, s, O::re(e3)), O::fma(-c, d, O::im(e3)));
    a[7] = O::mk(O::fma(c, s, O::re(e3)), O::fma(c, d, O::im(e3)));
  } else {
    a[3] = O::mk(O::fma(c, d, O::re(e3)), O::fma(-c, s, O::im(e3)));
    a[7] = O::mk(O::fma(-c, d, O::re(e3)), O::fma(c, s, O::im(e3)));
  }
}

template <class O, bool INV>
__device__ __forceinline__ void dft16(typename O::C* a) {
  using C = typename O::C;
  using S = typename O::S;
  constexpr float c = 0.70710678118654752440f;     // cos(pi/4)
  constexpr float c1 = 0.92387953251128675613f;    // cos(pi/8)
  constexpr float tn = 0.41421356237309504880f;    // tan(pi/8)
  constexpr float T = INV ? -tn : tn;
  // 16 = 4 x 4: DFT4 over a[4 n1 + n2], twiddle W16^(n2 k1), DFT4 over n2
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4<O, INV>(a[n2], a[4 + n2], a[8 + n2], a[12 + n2]);
  // a[4 k1 + n2] holds y[n2][k1]
  dft4<O, INV>(a[0], a[1], a[2], a[3]);   // k1 = 0
  {   // k1 = 1: W16^1 y1 = c1 u1, W8 y2 = c z, W16^3 y3 = c1 u3
    const C y0 = a[4], y1 = a[5], y2 = a[6], y3 = a[7];
    const C u1 = O::mk(O::fma(T, O::im(y1), O::re(y1)), O::fma(-T, O::re(y1), O::im(y1)));
    const C z = c_eighth<O, INV>(y2);
    const C t0 = c_fma<O>(c, z, y0), t1 = c_fma<O>(-c, z, y0);
    // forward u3 = (tan re + im, -(re - tan im)), inverse u3 = (-(im - tan re), re + tan im)
    const S p = O::fma(tn, INV ? O::im(y3) : O::re(y3), INV ? O::re(y3) : O::im(y3));
    const S m = O::fma(-tn, INV ? O::re(y3) : O::im(y3), INV ? O::im(y3) : O::re(y3));
    const C s = INV ? O::mk(O::sub(O::re(u1), m), O::add(O::im(u1), p)) : O::mk(O::add(O::re(u1), p), O::sub(O::im(u1), m));
    const C d = INV ? O::mk(O::add(O::re(u1), m), O::sub(O::im(u1), p)) : O::mk(O::sub(O::re(u1), p), O::add(O::im(u1), m));
    a[4] = c_fma<O>(c1, s, t0);
    a[6] = c_fma<O>(-c1, s, t0);
    a[5] = c_fma_rot<O, INV>(c1, d, t1);
    a[7] = c_fma_rot<O, INV>(-c1, d, t1);
  }
  {   // k1 = 2: W8 y1, -+i y2, W8^3 y3: sum and difference of the first and last from y1 -+ y3
    const C y0 = a[8], y2 = a[10], p = c_sub<O>(a[9], a[11]), q = c_add<O>(a[9], a[11]);
    const C t0 = c_add_rot<O, INV>(y0, y2), t1 = c_sub_rot<O, INV>(y0, y2);
    const C s = c_add_rot<O, INV>(p, q), d = c_add_rot<O, INV>(q, p);
    a[8] = c_fma<O>(c, s, t0);
    a[10] = c_fma<O>(-c, s, t0);
    a[9] = c_fma_rot<O, INV>(c, d, t1);
    a[11] = c_fma_rot<O, INV>(-c, d, t1);
  }
  {   // k1 = 3: W16^3 y1 = c1 u1, W8^3 y2, W16^9 y3 = -c1 u3
    const C y0 = a[12], y1 = a[13], y2 = a[14], y3 = a[15];
    const S p = O::fma(tn, INV ? O::im(y1) : O::re(y1), INV ? O::re(y1) : O::im(y1));
    const S m = O::fma(-tn, INV ? O::re(y1) : O::im(y1), INV ? O::im(y1) : O::re(y1));
    const S r2 = O::add(O::re(y2), O::im(y2)), d2 = O::sub(O::im(y2), O::re(y2));
    const C t0 = INV ? O::mk(O::fma(-c, r2, O::re(y0)), O::fma(-c, d2, O::im(y0)))
                     : O::mk(O::fma(c, d2, O::re(y0)), O::fma(-c, r2, O::im(y0)));
    const C t1 = INV ? O::mk(O::fma(c, r2, O::re(y0)), O::fma(c, d2, O::im(y0)))
                     : O::mk(O::fma(-c, d2, O::re(y0)), O::fma(c, r2, O::im(y0)));
    const C u3 = O::mk(O::fma(T, O::im(y3), O::re(y3)), O::fma(-T, O::re(y3), O::im(y3)));
    // forward u1 = (p, -m), inverse u1 = (-m, p); sum u1 - u3, difference u1 + u3 (negated components folded below)
    if (INV) {
      const C s = O::mk(O::add(m, O::re(u3)), O::sub(p, O::im(u3)));   // (-(u1 - u3).re, (u1 - u3).im)
      const C d = O::mk(O::sub(O::re(u3), m), O::add(p, O::im(u3)));
      a[12] = O::mk(O::fma(-c1, O::re(s), O::re(t0)), O::fma(c1, O::im(s), O::im(t0)));
      a[14] = O::mk(O::fma(c1, O::re(s), O::re(t0)), O::fma(-c1, O::im(s), O::im(t0)));
      a[13] = c_fma_rot<O, INV>(c1, d, t1);
      a[15] = c_fma_rot<O, INV>(-c1, d, t1);
    } else {
      const C s = O::mk(O::sub(p, O::re(u3)), O::add(m, O::im(u3)));   // ((u1 - u3).re, -(u1 - u3).im)
      const C d = O::mk(O::add(p, O::re(u3)), O::sub(O::im(u3), m));
      a[12] = O::mk(O::fma(c1, O::re(s), O::re(t0)), O::fma(-c1, O::im(s), O::im(t0)));
      a[14] = O::mk(O::fma(-c1, O::re(s), O::re(t0)), O::fma(c1, O::im(s), O::im(t0)));
      a[13] = c_fma_rot<O, INV>(c1, d, t1);
      a[15] = c_fma_rot<O, INV>(-c1, d, t1);
    }
  }
  // a[4 k1 + k2] holds X[k1 + 4 k2]
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = i + 1; j < 4; ++j) {
      const C x = a[4 * i + j];
      a[4 * i + j] = a[4 * j + i];
      a[4 * j + i] = x;
    }
}

template <bool INV> struct Dft<8, INV> {
  static __device__ __forceinline__ void run(float2* a) { dft8<LineOps, INV>(a); }
};
template <bool INV> struct Dft<16, INV> {
  static __device__ __forceinline__ void run(float2* a) { dft16<LineOps, INV>(a); }
};

// 3 P-point DFT (P = 2, 4, 8) from P-point and 3-point ones without twiddles between them (Good's prime
// factor map): input 3 n1 + P n2, output K1 k1 + K2 k2 (mod 3 P), K1 = 1 mod P and 0 mod 3, K2 the reverse
template <int P, bool INV> struct DftPrime3 {
  static __device__ __forceinline__ void run(float2* a) {
    constexpr int K1 = (P == 2) ? 3 : 9, K2 = (P == 8) ? 16 : 4;
    float2 y[3][P];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < P; ++n1) y[n2][n1] = a[(3 * n1 + P * n2) % (3 * P)];
      Dft<P, INV>::run(y[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) {
      float2 t[3] = {y[0][k1], y[1][k1], y[2][k1]};
      Dft<3, INV>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) a[(K1 * k1 + K2 * k2) % (3 * P)] = t[k2];
    }
  }
};
template <bool INV> struct Dft<6, INV> : DftPrime3<2, INV> {};
template <bool INV> struct Dft<12, INV> : DftPrime3<4, INV> {};
template <bool INV> struct Dft<24, INV> : DftPrime3<8, INV> {};

// Twiddle tables.  Butterfly j of a stage with NS > 1 multiplies its input r by w^r,
// w = W_N^((j mod NS) N/(NS R)).  The table stores only the powers w^p for p in
// {1, 2, 4, 8, 16} below R (w and w^2 for radix 3), as rows of NS entries (the threads of a
// warp, consecutive j, read consecutive entries); the butterfly forms the other powers
// by at most three complex products (w^3 = w^2 w, w^5 = w^4 w, ..., w^15 = w^8 w^7).
// A 4096-point plan then needs 1088 entries (8.5 KB) instead of 4080, which stay in L1
// when a pass gives most of the SM's on-chip memory to shared memory.  Stages are
// concatenated in order; twiddle_offset(N, V, s) is where stage s starts.
// Narrow power-of-two lines up to 1024 points (V = 8; at most 1016 entries) store every power: their
// radix-8 stages are one more rounding than a wide line's, and exact powers make up for it (relative RMS
// error of 64 points 9.1e-8 with formed powers, 7.9e-8 with these, the wide plan 8.3e-8; 1024 points 12.0e-8,
// 10.7e-8, 11.6e-8).
// A caller may ask for every power (X) of another plan, with the table to match.
__host__ __device__ constexpr bool tw_every(int N, int V) { return V == 8 && N <= 1024; }
__host__ __device__ constexpr int tw_npow(int R, bool X) {
  return X ? R - 1 : R > 16 ? 5 : R > 8 ? 4 : R > 4 ? 3 : R > 2 ? 2 : 1;
}
__host__ __device__ constexpr int tw_pow(int q, bool X) { return X ? q + 1 : 1 << q; }   // the q-th stored power
__host__ __device__ constexpr int stage_ns(int N, int V, int s) {
  int ns = 1;
  for (int i = 0; i < s; ++i) ns *= radix_at(N, V, i);
  return ns;
}
__host__ __device__ constexpr int twiddle_offset(int N, int V, int s, bool X) {
  int off = 0;
  for (int i = 1; i < s; ++i) off += tw_npow(radix_at(N, V, i), X) * stage_ns(N, V, i);
  return off;
}
__host__ __device__ constexpr int twiddle_count(int N, int V, bool X) { return twiddle_offset(N, V, num_stages(N, V), X); }
__host__ __device__ constexpr int twiddle_count(int N, int V) { return twiddle_count(N, V, tw_every(N, V)); }
// exponent e (of W_N^e = exp(-2 pi i e / N)) of table entry i, 0 <= i < twiddle_count(N, V)
__host__ __device__ constexpr long long twiddle_exponent(int N, int V, int i, bool X) {
  const int S = num_stages(N, V);
  int s = 1;
  while (s + 1 < S && twiddle_offset(N, V, s + 1, X) <= i) ++s;
  const int NS = stage_ns(N, V, s), R = radix_at(N, V, s);
  const int local = i - twiddle_offset(N, V, s, X);
  const int q = local / NS, jm = local - q * NS;
  return ((long long)jm * tw_pow(q, X) * (N / (NS * R))) % N;
}
__host__ __device__ constexpr long long twiddle_exponent(int N, int V, int i) {
  return twiddle_exponent(N, V, i, tw_every(N, V));
}

// w^r for r = 1..R-1 of one butterfly from the stored powers (tws: this butterfly's
// first entry; rows NS apart); conjugated for the inverse transform
template <int R, bool INV, bool X>
__device__ __forceinline__ void twiddle_powers(float2 (&w)[R], const float2* __restrict__ tws, int NS) {
#pragma unroll
  for (int q = 0; q < tw_npow(R, X); ++q) {
    float2 x = __ldg(tws + q * NS);
    if (INV) x.y = -x.y;
    w[tw_pow(q, X)] = x;
  }
  if constexpr (X) return;
#pragma unroll
  for (int r = 3; r < R; ++r) {
    if ((r & (r - 1)) == 0) continue;          // stored
    const int hi = r >= 16 ? 16 : (r >= 8 ? 8 : (r >= 4 ? 4 : 2));   // largest stored power below r
    w[r] = cmul(w[hi], w[r - hi]);
  }
}

// Barrier over the threads that transform one line: the whole CTA (bid 0) or
// named barrier bid over the line's T threads, when each line owns whole warps
// and the CTA holds several lines, so that lines progress independently.
// bid < 0: the line is one warp, which synchronises alone.
template <int T>
__device__ __forceinline__ void line_sync(int bid) {
  if (bid == 0) {
    __syncthreads();
  } else if (bid < 0) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(bid), "n"(T) : "memory");
  }
}
// barrier id of line group g for line_sync: the line's own warp when a line is at most one warp
// (T divides 32, so no line straddles two warps), 1 + g when lines of T threads own several whole
// warps (at most 8 lines per CTA of up to 512 threads), else 0 (the CTA barrier)
template <int T>
__device__ __forceinline__ int line_bar(int g) {
  return (32 % T == 0) ? -1 : (T % 32 == 0) ? 1 + g : 0;
}

// ------------------------------------------------------------------ stages
// Stage S of the Stockham transform; NS = product of the radices before it.
// Butterfly j reads x[j + r N/R], multiplies by W_N^((j mod NS) r N/(NS R)),
// applies the R-point DFT and writes x[(j/NS) NS R + (j mod NS) + r NS].
// Thread t owns butterflies j = t + T b (b < V/R), whose inputs are its
// canonical slots b + r V/R; the last stage's outputs land in canonical slots.
template <int N, int V, int S, int NS, bool INV, bool TRAIL, bool X>
struct Stage {
  static __device__ __forceinline__ void run(float2 (&v)[V], float2* sm, int t, const float2* __restrict__ tw, int bid) {
    constexpr int R = radix_at(N, V, S);
    constexpr int T = N / V;
    constexpr int B = V / R;
    constexpr bool LAST = (S == num_stages(N, V) - 1);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      float2 a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) a[r] = v[b + r * B];
      const int j = t + T * b;
      if (NS > 1) {
        float2 w[R];
        twiddle_powers<R, INV, X>(w, tw + twiddle_offset(N, V, S, X) + (j % NS), NS);
#pragma unroll
        for (int r = 1; r < R; ++r) a[r] = cmul(a[r], w[r]);
      }
      Dft<R, INV>::run(a);
      if (LAST) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[b + r * B] = a[r];
      } else {
        const int p = (j / NS) * NS * R + (j % NS);
#pragma unroll
        for (int r = 0; r < R; ++r) sm[pidx(p + r * NS)] = a[r];
      }
    }
    if constexpr (!LAST) {
      line_sync<T>(bid);
#pragma unroll
      for (int m = 0; m < V; ++m) v[m] = sm[pidx(t + T * m)];
      // the buffer is written again by the next stage, or (after the last exchange) by the caller;
      // without TRAIL the caller synchronises before it reuses the buffer
      if constexpr (TRAIL || S + 2 < num_stages(N, V)) line_sync<T>(bid);
      Stage<N, V, S + 1, NS * R, INV, TRAIL, X>::run(v, sm, t, tw, bid);
    }
  }
};

// Unnormalised line DFT, sign -1 (forward) or +1 (INV).  Every thread of the
// CTA (bid 0) or of the line (bid = line_bar(g)) must call it: it synchronises
// with line_sync(bid) when the plan has >1 stage.  With TRAIL = false it returns
// while other threads of the line may still read sm: the caller must pass a
// barrier of those threads before anything writes sm again.
// tw: the stage-major twiddle table of (N, V, X) described above (exp(-2 pi i e/N)
// values).  sm: this line's padded buffer.
template <int N, int V, bool INV, bool TRAIL = true, bool X = tw_every(N, V)>
__device__ __forceinline__ void fft_line(float2 (&v)[V], float2* sm, int t, const float2* __restrict__ tw, int bid = 0) {
  static_assert(N % V == 0, "V must divide N");
  static_assert(num_stages(N, V) > 0, "no radix plan");
  Stage<N, V, 0, 1, INV, TRAIL, X>::run(v, sm, t, tw, bid);
}

}  // namespace fftenkf
