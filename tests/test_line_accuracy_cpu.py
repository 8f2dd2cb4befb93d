"""Accuracy of the line transforms (csrc/fft_core.cuh), stage by stage on the host: a narrow plan (radix 8, more
stages) is no further from the 64-bit transform than the wide plan of the same length, for white lines and for
lines with a steep spectrum, so that a pass may choose either by speed; and a wide plan with every twiddle power in
its table (the sine passes) is no further off than the one with formed powers."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1001_1588_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <random>
#include <vector>
struct float2 { float x, y; };
static float2 make_float2(float a, float b) { return {a, b}; }
#define __device__
#define __host__
#define __forceinline__ inline
#define __restrict__
template <class T> T __ldg(const T* p) { return *p; }
static void __syncthreads() {}
static void __syncwarp() {}
#include "fft_core.cuh"
using namespace fftenkf;
typedef std::complex<double> C;

template <int N, int V, int S, int NS, bool X>
void stages(std::vector<float2>& x, const float2* tw) {
  constexpr int R = radix_at(N, V, S);
  std::vector<float2> y(N);
  for (int j = 0; j < N / R; ++j) {
    float2 a[R], w[R];
    for (int r = 0; r < R; ++r) a[r] = x[j + r * (N / R)];
    if (NS > 1) {
      twiddle_powers<R, false, X>(w, tw + twiddle_offset(N, V, S, X) + j % NS, NS);
      for (int r = 1; r < R; ++r) a[r] = cmul(a[r], w[r]);
    }
    Dft<R, false>::run(a);
    for (int r = 0; r < R; ++r) y[(j / NS) * NS * R + j % NS + r * NS] = a[r];
  }
  x.swap(y);
  if constexpr (S + 1 < num_stages(N, V)) stages<N, V, S + 1, NS * R, X>(x, tw);
}
std::vector<C> exact(const std::vector<C>& a) {
  const size_t n = a.size();
  if (n == 1) return a;
  std::vector<C> e, o, z(n);
  for (size_t i = 0; i < n; i += 2) { e.push_back(a[i]); o.push_back(a[i + 1]); }
  e = exact(e); o = exact(o);
  for (size_t k = 0; k < n; ++k) z[k] = e[k % (n / 2)] + std::polar(1.0, -2 * M_PI * k / n) * o[k % (n / 2)];
  return z;
}
template <int N, int V, bool X> double error(int steep) {
  std::vector<float2> tw;
  for (int i = 0; i < twiddle_count(N, V, X); ++i) {
    const double a = 2 * M_PI * twiddle_exponent(N, V, i, X) / N;
    tw.push_back({(float)std::cos(a), (float)-std::sin(a)});
  }
  tw.push_back({0, 0});
  std::mt19937 g(7);
  std::normal_distribution<double> d;
  double off = 0, all = 0;
  for (int it = 0; it < 40960 / N; ++it) {
    std::vector<C> z(N);
    for (int k = 0; k < N; ++k) {
      const int q = k < N / 2 ? k : k - N;
      z[k] = C(d(g), d(g)) * (steep ? 64.0 / (1 + q * q) : 1.0);
    }
    if (steep == 1) z = exact(z);   // a smooth line; 2: a line of steep coefficients
    std::vector<float2> x(N);
    for (int k = 0; k < N; ++k) {
      x[k] = {(float)z[k].real(), (float)z[k].imag()};
      z[k] = C(x[k].x, x[k].y);
    }
    z = exact(z);
    stages<N, V, 0, 1, X>(x, tw.data());
    for (int k = 0; k < N; ++k) { off += std::norm(C(x[k].x, x[k].y) - z[k]); all += std::norm(z[k]); }
  }
  return std::sqrt(off / all);
}
template <int N> void line() {
  for (int s = 0; s < 3; ++s) std::printf("%d %d %.4e %.4e %.4e\n", N, s,
    error<N, plan_V(N, 1), tw_every(N, plan_V(N, 1))>(s), error<N, plan_V(N, 0), false>(s), error<N, plan_V(N, 0), true>(s));
}
int main() { line<32>(); line<64>(); line<128>(); line<256>(); line<512>(); line<1024>(); }
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_narrow_lines_are_as_accurate_as_wide_ones(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text("")
    (tmp_path / "t.cc").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-I", str(tmp_path), "-I", CSRC,
                    str(tmp_path / "t.cc"), "-o", exe], check=True)
    rows = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")[:-1]
    assert len(rows) == 18
    for row in rows:
        narrow, wide, exact = (float(x) for x in row.split()[2:])
        assert narrow <= wide and exact <= wide, row
