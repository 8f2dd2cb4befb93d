// FP64 inputs and outputs without the FP64 unit.
//
// GB300's FP64 unit is slow even for single adds and conversions: forming chat + rhat in FP64 for every
// wavenumber and observed block (one add and two conversions, 16.8 M times at 4096^2 with two observed
// blocks) took 0.9 ms of the fused column pass's 5.4, nearly all of its gain step.  Here a double is split by
// integer operations into floats (all 53 bits: 24 + 24 + 5), and sums, products and quotients are formed in
// float pairs (Knuth's two-sum, FMA products).  Every result is the exact value rounded to float once: sums by
// rounding to odd first (Boldo and Melquiond), quotients by Ziv's test, which takes FP64, out of line, where
// the pair's error could change the rounding.  So no result is further from the exact value than the same
// FP64 operations rounded to float.  Values whose exponent leaves no room for the pair (below 2^-74 or above
// 2^120, not 0), sums that cancel, and denominators that are not comfortably normal floats take FP64 too.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fftenkf {

struct fpair {
  float h, l;
};

// x as hi + lo (hi its leading 24 bits, lo the next 24, rounded), and the last bits' remainder in rest; false
// where x is neither 0 nor within 2^-74 .. 2^120
__device__ __forceinline__ bool split_double(double x, fpair& p, float& rest) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ffu);
  const uint32_t sign = h & 0x80000000u;
  const bool zero = ((h << 1) | l) == 0u;
  const uint32_t hi = (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29);
  const float scale = __uint_as_float(((uint32_t)(e - 948) << 23) | sign);   // 2^(e - 1075), signed
  p.h = zero ? 0.f : __uint_as_float(hi | sign);
  p.l = zero ? 0.f : __uint2float_rn(l & 0x1fffffe0u) * scale;
  rest = zero ? 0.f : __uint2float_rn(l & 0x1fu) * scale;
  return zero || (unsigned)(e - 949) <= 194u;
}
__device__ __forceinline__ bool split_double(double x, fpair& p) {
  float rest;
  return split_double(x, p, rest);
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
// a b s rounded to float; false where an error of 2^-42 cond in it could change the rounding (or it is tiny).
// The pair operations above and a truncated split are within 2^-44 of their values each.
__device__ __forceinline__ bool pair_product(fpair a, fpair b, float s, float cond, float& out) {
  const fpair p = pair_mul(a, b);
  const float t = __fmul_rn(p.h, s);
  const float e = fmaf(p.l, s, fmaf(p.h, s, -t));
  const float d = fabsf(t) * 0x1p-42f * cond;
  out = t + (e + d);
  return (out == t + (e - d) && fabsf(t) >= 1e-30f) || a.h == 0.f;
}
__device__ __forceinline__ bool well_inside(float x) { return fabsf(x) >= 1e-30f && fabsf(x) <= 1e30f; }

// chat + rhat rounded to float; false where it must be formed in FP64 (and where it is below FLT_MIN)
__device__ __forceinline__ bool denominator(float val, double rhat, float& den) {
  fpair r;
  float rest;
  const bool ok = split_double(rhat, r, rest);
  const fpair s = two_sum(val, r.h);
  // the tail s.l + r.l + rest rounded to odd: where t.l + rest is not 0, the neighbour on its side of an even t.h
  const fpair t = two_sum(s.l, r.l);
  const float low = t.l + rest;
  const uint32_t b = __float_as_uint(t.h), toward = ((b ^ __float_as_uint(low)) >> 31) ? ~0u : 1u;
  const float odd = __uint_as_float((low != 0.f && !(b & 1u)) ? b + toward : b);
  den = s.h + (t.h == 0.f ? low : odd);
  return ok && den >= 1.17549435e-38f && den >= 0.5f * fabsf(r.h);   // no cancellation
}
// inv_G / (val + rhat) in FP64, 0 where the denominator is exactly 0
static __device__ __noinline__ double quotient_fp64(float val, double rhat, float inv_G) {
  const double den = (double)val + rhat;
  return (den != 0.0) ? (double)inv_G / den : 0.0;
}
// a + b of two numbers split without their last bits; false where it cancels or is no comfortable float
__device__ __forceinline__ bool pair_sum(fpair a, fpair b, fpair& s) {
  s = pair_add(a, b);
  return well_inside(s.h) && fabsf(s.h) >= 0.5f * fmaxf(fabsf(a.h), fabsf(b.h));
}
// the same rounded to float
__device__ __forceinline__ float quotient(float val, double rhat, float inv_G) {
  fpair r, den;
  const bool in = split_double(rhat, r);
  float q;
  if (in && pair_sum({val, 0.f}, r, den) && pair_product({1.f, 0.f}, pair_recip(den), inv_G, 1.f, q)) return q;
  return (float)quotient_fp64(val, rhat, inv_G);
}

static __device__ __noinline__ double spec_quotient_fp64(double den, float scale) {
  return (den != 0.0) ? (double)scale / den : 0.0;
}
__device__ __forceinline__ int exponent_of(double x) { return (int)((uint32_t)__double2hiint(x) >> 20) & 0x7ff; }

// scale / (a + rhat) for a caller's spectrum, and its products with entries x of the spectrum, each rounded
// to float once.  Steep spectra (a squared-exponential one over most of the plane) hold entries below 2^-74:
// as a or rhat they count as 0 beside a sum of at least 2^-24 (2^-50 of it), as x their exponent is raised by
// 96 and the result lowered again.  (In FP64 such entries took the gain kernel 1.3 to 3 times as long: 512^2,
// one observed of three blocks, 26 us instead of 9; 12.5 us with FP64 throughout.)
struct SpecQuotient {
  fpair inv;
  double inv64;   // formed where the pairs do not hold it, or at the first product that needs it
  float scale;
  bool pairs, formed;
  __device__ __forceinline__ SpecQuotient(double a, double rhat, float s) : inv64(0.0), scale(s) {
    fpair ap, rp, den;
    const bool ta = exponent_of(a) < 949, tr = exponent_of(rhat) < 949;
    const bool in = (split_double(ta ? 0.0 : a, ap) & split_double(tr ? 0.0 : rhat, rp));
    pairs = pair_sum(ap, rp, den) && in && (!(ta | tr) || fabsf(den.h) >= 0x1p-24f);
    inv = pair_recip(den);
    formed = !pairs;
    if (!pairs) inv64 = spec_quotient_fp64(a + rhat, s);
  }
  __device__ __forceinline__ float times(double x, double a, double rhat) {
    if (!pairs) return (float)(x * inv64);
    const int e = exponent_of(x);
    const bool low = e < 949;
    fpair xp;
    float out;
    // (zeros, subnormals and exponents below 853 stay out of split_double's range when raised)
    const bool in = split_double(low ? __hiloint2double(__double2hiint(x) + (96 << 20), __double2loint(x)) : x, xp);
    const bool ok = pair_product(xp, inv, scale, 1.f, out);
    if (!low) {
      if (in && ok) return out;
    } else if (e < 853) {   // below 2^-170
      if (fabsf(inv.h) * scale < 0x1p18f) return 0.f;
    } else if (in) {
      if (fabsf(xp.h * inv.h * scale) < 0x1p-58f) return 0.f;   // below 2^-154
      if (ok && fabsf(out) >= 0x1p-30f) return out * 0x1p-96f;   // exact: a normal float
      // a subnormal float: out, rounded already, is rounded again to a multiple of 2^-149 (in this scale 2^-53),
      // which is wrong only where it lies half-way
      const float z = fabsf(out) * 0x1p53f, k = rintf(z);
      if (ok && fabsf(z - k) != 0.5f) return copysignf(__uint_as_float((uint32_t)k), out);
    }
    if (!formed) inv64 = spec_quotient_fp64(a + rhat, scale);
    formed = true;
    return (float)(x * inv64);
  }
};

// g A^-1 of the bracket A = [[a0 + r0, conj b], [b, a1 + r1]] of two coupled observed blocks: A^-1 when
// det A > 1e-6 a11 a22, the pseudo-inverse A / tr(A)^2 of a rank-1 bracket otherwise, 0 where tr(A) = 0; rounded
// to float.
struct Bracket {
  float s00, s11;
  float2 s01;
};
static __device__ __noinline__ Bracket bracket_fp64(float a0, float a1, float2 b, double r0, double r1, float g) {
  const double a = (double)a0 + r0, d = (double)a1 + r1;
  const double br = b.x, bi = b.y;
  const double det = a * d - (br * br + bi * bi);
  const double tr = a + d;
  double f = 0.0, q00 = 0.0, q11 = 0.0, q01r = 0.0, q01i = 0.0;   // A^-1 = f [[q00, q01], [conj q01, q11]]
  if (det > 1e-6 * a * d) {
    f = (double)g / det;
    q00 = d; q11 = a; q01r = -br; q01i = bi;      // [[d, -conj b], [-b, a]] / det
  } else if (tr > 0.0) {
    f = (double)g / (tr * tr);
    q00 = a; q11 = d; q01r = br; q01i = -bi;      // [[a, conj b], [b, d]] / tr^2
  }
  return {(float)(f * q00), (float)(f * q11), make_float2((float)(f * q01r), (float)(f * q01i))};
}
// The same in float pairs, FP64 where their error could change a result's rounding.  The determinant's relative
// error grows with cond = a11 a22 / det, which is at most 2^10 here (up to 1e6 where it is used).
__device__ __forceinline__ Bracket bracket(float a0, float a1, float2 b, double r0, double r1, float g) {
  fpair p0, p1, a, d;
  bool in = split_double(r0, p0) & split_double(r1, p1);
  in &= pair_sum({a0, 0.f}, p0, a);
  in &= pair_sum({a1, 0.f}, p1, d);
  const fpair ad = pair_mul(a, d);
  const fpair bb = pair_add(pair_mul({b.x, 0.f}, {b.x, 0.f}), pair_mul({b.y, 0.f}, {b.y, 0.f}));
  const fpair det = pair_add(ad, {-bb.h, -bb.l});
  const fpair f = pair_recip(det);
  const float cond = ad.h * f.h;
  Bracket k;
  in &= well_inside(det.h) && a.h > 0.f && cond > 0.f && cond <= 1024.f;
  in &= pair_product(d, f, g, cond, k.s00);
  in &= pair_product(a, f, g, cond, k.s11);
  in &= pair_product({-b.x, 0.f}, f, g, cond, k.s01.x);
  in &= pair_product({b.y, 0.f}, f, g, cond, k.s01.y);
  return in ? k : bracket_fp64(a0, a1, b, r0, r1, g);
}

}  // namespace fftenkf
