"""The gains' arithmetic without the FP64 unit (csrc/dd.cuh), compiled for the host: on random operands, exact
floats, few-bit numbers, all 53 bits and (caller's spectra) vanishing entries, no result may be further from the exact value (113 bits) than the same
FP64 operations rounded to float, and a denominator is the exact sum rounded to float."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1588_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
#define __noinline__
struct float2 { float x, y; };
static float2 make_float2(float a, float b) { return {a, b}; }
template <class T, class U> T bits(U u) { T t; static_assert(sizeof t == sizeof u, ""); std::memcpy(&t, &u, sizeof t); return t; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __frcp_rn(float a) { return 1.0f / a; }
static float __uint_as_float(uint32_t u) { return bits<float>(u); }
static uint32_t __float_as_uint(float f) { return bits<uint32_t>(f); }
static int __double2hiint(double d) { return (int)(bits<uint64_t>(d) >> 32); }
static int __double2loint(double d) { return (int)(uint32_t)bits<uint64_t>(d); }
static double __hiloint2double(int h, int l) { return bits<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static float __uint2float_rn(uint32_t u) { return (float)u; }
#include "dd.cuh"
#ifdef __x86_64__
typedef __float128 quad;
#else
typedef long double quad;
#endif
static quad mag(quad a) { return a < 0 ? -a : a; }
"""

MAIN = SHIM + r"""
using namespace fftenkf;
int main() {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(0, 1);
  auto value = [&] {
    double v = std::exp2(60 * U(g) - 40);
    const int kind = g() % 4;
    int e;
    if (kind == 1) v = (float)v;
    if (kind == 2) v = std::ldexp(std::floor(std::frexp(v, &e) * (1 << (1 + (int)(20 * U(g))))) + 1, e - 12);
    if (kind == 3) v = (float)v * (1 + std::ldexp(std::floor(32 * U(g)), -52));
    return v;
  };
  long den_off = 0, quot_worse = 0, spec_worse = 0, bracket_worse = 0, conversions = 0, fp64_used = 0;
  for (int i = 0; i < 1000000; ++i) {
    const double r = value(), a = value(), x = i % 3 ? value() : a;
    float val = (float)value(), s = 1.0f / (1 << (int)(24 * U(g))), den;
    if (i % 2) s /= 3;
    if (g() % 8 == 0) val = -val * (float)U(g);
    if (denominator(val, r, den)) den_off += (float)((quad)val + r) != den;
    const quad q = (quad)s / ((quad)val + r);
    quot_worse += mag((quad)quotient(val, r, s) - q) > mag((quad)(float)(s / (val + r)) - q);
    const quad p = (quad)x * s / ((quad)a + r);
    spec_worse += mag((quad)SpecQuotient(a, r, s).times(x, a, r) - p) > mag((quad)(float)(x * (s / (a + r))) - p);
    // a steep spectrum beside an ordinary rhat, and both anywhere
    const double tiny = i % 16 ? std::exp2(-320 * U(g)) * (1 + U(g)) : 0.0, y = i % 3 ? tiny : -tiny * U(g);
    const double rr = i % 5 ? std::exp2(-10 * U(g)) : std::exp2(-160 * U(g));
    SpecQuotient st(tiny, rr, s);
    const quad py = (quad)y * s / ((quad)tiny + rr);
    spec_worse += mag((quad)st.times(y, tiny, rr) - py) > mag((quad)(float)(y * (s / (tiny + rr))) - py);
    fp64_used += i % 5 && !st.pairs;
    conversions += to_float(r) != (float)r || to_double(val) != (double)val;
    const float a0 = (float)std::exp2(10 * U(g) - 8), a1 = (float)std::exp2(10 * U(g) - 8);
    const double r0 = i % 5 ? std::exp2(12 * U(g) - 12) : 0.0, r1 = i % 5 ? std::exp2(12 * U(g) - 12) : 0.0;
    const double rho = i % 3 ? U(g) : 1 - std::exp2(-20 * U(g)), ph = 6.2831853 * U(g);
    const double m = rho * std::sqrt((a0 + r0 * (i % 2)) * (a1 + r1 * (i % 2)));
    const float2 b = {(float)(m * std::cos(ph)), (float)(m * std::sin(ph))};
    const quad A = (quad)a0 + r0, D = (quad)a1 + r1, det = A * D - ((quad)b.x * b.x + (quad)b.y * b.y);
    if (det > (quad)2e-6 * A * D) {
      const Bracket k = bracket(a0, a1, b, r0, r1, s), f = bracket_fp64(a0, a1, b, r0, r1, s);
      const quad e[4] = {s * D / det, s * A / det, -(quad)b.x * s / det, (quad)b.y * s / det};
      const float u[4] = {k.s00, k.s11, k.s01.x, k.s01.y}, v[4] = {f.s00, f.s11, f.s01.x, f.s01.y};
      for (int t = 0; t < 4; ++t) bracket_worse += mag((quad)u[t] - e[t]) > mag((quad)v[t] - e[t]);
    }
  }
  std::printf("%ld %ld %ld %ld %ld %ld\n", den_off, quot_worse, spec_worse, bracket_worse, conversions, fp64_used);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_no_result_is_further_off_than_fp64(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text("")
    (tmp_path / "t.cc").write_text(MAIN)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-I", str(tmp_path), "-I", CSRC,
                    str(tmp_path / "t.cc"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    assert [int(x) for x in out.split()] == [0, 0, 0, 0, 0, 0], out
