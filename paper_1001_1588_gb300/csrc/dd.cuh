// FP64 inputs and outputs without the FP64 unit.
//
// GB300's FP64 unit is slow even for single adds and conversions: forming chat + rhat in FP64 for every
// wavenumber and observed block (one add and two conversions, 16.8 M times at 4096^2 with two observed
// blocks) took 0.9 ms of the fused column pass's 5.4, nearly all of its gain step.  Here a double is split by
// integer operations into two floats, hi + lo with 48 of its 53 bits, sums and quotients are formed in
// float pairs (Knuth's two-sum, FMA products) and rounded to float once, as the FP64 results were.  Values
// whose exponent leaves no room for the pair (below 2^-74 or above 2^120, not 0) and denominators that
// are not comfortably normal floats take FP64, out of line.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fftenkf {

struct fpair {
  float h, l;
};

// x as hi + lo (hi its leading 24 bits, lo the next 24); false where x is neither 0 nor within 2^-74 .. 2^120
__device__ __forceinline__ bool split_double(double x, fpair& p) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ffu);
  const uint32_t sign = h & 0x80000000u;
  const bool zero = ((h << 1) | l) == 0u;
  const uint32_t hi = (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29);
  const float scale = __uint_as_float(((uint32_t)(e - 948) << 23) | sign);   // 2^(e - 1075), signed
  p.h = zero ? 0.f : __uint_as_float(hi | sign);
  p.l = zero ? 0.f : __uint2float_rn(l & 0x1fffffffu) * scale;
  return zero || (unsigned)(e - 949) <= 194u;
}

// x rounded to float (nearest, ties to even), as the conversion instruction does
__device__ __forceinline__ float to_float(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t e = (h >> 20) & 0x7ffu;
  if (e - 897u > 253u) return (float)x;   // 0, subnormal or out of a float's range
  uint32_t f = (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29);
  const uint32_t rest = l & 0x1fffffffu;
  f += (rest > 0x10000000u || (rest == 0x10000000u && (f & 1u))) ? 1u : 0u;
  return __uint_as_float(f | (h & 0x80000000u));
}

// x as a double
__device__ __forceinline__ double to_double(float x) {
  const uint32_t f = __float_as_uint(x);
  const uint32_t e = (f >> 23) & 0xffu;
  if (e - 1u > 253u) return (double)x;    // 0, subnormal, infinite or NaN
  return __hiloint2double((int)((((f & 0x7fffffffu) >> 3) + 0x38000000u) | (f & 0x80000000u)), (int)(f << 29));
}

__device__ __forceinline__ bool finite_double(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }

// a + b exactly, as sum and error
__device__ __forceinline__ fpair two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ fpair quick_two_sum(float a, float b) {   // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ fpair pair_add(fpair a, fpair b) {
  const fpair s = two_sum(a.h, b.h);
  return quick_two_sum(s.h, s.l + (a.l + b.l));
}
__device__ __forceinline__ fpair pair_mul(fpair a, fpair b) {
  const float p = __fmul_rn(a.h, b.h);
  return quick_two_sum(p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p))));
}
// 1 / a for a normal a well inside the float range
__device__ __forceinline__ fpair pair_recip(fpair a) {
  const float i = __frcp_rn(a.h);
  return {i, i * fmaf(-a.l, i, fmaf(-a.h, i, 1.f))};
}
// a b s rounded to float once
__device__ __forceinline__ float pair_product(fpair a, fpair b, float s) {
  const fpair p = pair_mul(a, b);
  const float t = __fmul_rn(p.h, s);
  return t + fmaf(p.l, s, fmaf(p.h, s, -t));
}
__device__ __forceinline__ bool well_inside(float x) { return fabsf(x) >= 1e-30f && fabsf(x) <= 1e30f; }

// chat + rhat rounded to float; false where it must be formed in FP64 (and where it is below FLT_MIN)
__device__ __forceinline__ bool denominator(float val, double rhat, float& den) {
  fpair r;
  const bool ok = split_double(rhat, r);
  const fpair s = two_sum(val, r.h);
  den = s.h + (s.l + r.l);
  return ok && den >= 1.17549435e-38f;
}
// inv_G / (val + rhat) in FP64, 0 where the denominator is exactly 0
static __device__ __noinline__ double quotient_fp64(float val, double rhat, float inv_G) {
  const double den = (double)val + rhat;
  return (den != 0.0) ? (double)inv_G / den : 0.0;
}

// scale / (a + rhat) for a caller's spectrum, and its products with entries of the spectrum, each rounded
// to float once
struct SpecQuotient {
  fpair inv;
  double inv64;
  float scale;
  bool pairs;
  __device__ __forceinline__ SpecQuotient(double a, double rhat, float s) : inv64(0.0), scale(s) {
    fpair ap, rp;
    const bool in = split_double(a, ap) & split_double(rhat, rp);
    const fpair den = pair_add(ap, rp);
    pairs = in && well_inside(den.h);
    inv = pair_recip(den);
    if (!pairs) slow(a + rhat);
  }
  __device__ __noinline__ void slow(double den) { inv64 = (den != 0.0) ? (double)scale / den : 0.0; }
  __device__ __forceinline__ float times(double x) const {
    fpair xp;
    if (pairs && split_double(x, xp)) return pair_product(xp, inv, scale);
    return slow_times(x);
  }
  __device__ __noinline__ float slow_times(double x) const {
    if (!pairs) return (float)(x * inv64);
    return (float)(x * ((double)inv.h + (double)inv.l) * (double)scale);
  }
};

}  // namespace fftenkf
