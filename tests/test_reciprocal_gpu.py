"""The reciprocals of the density that the collision and the boundary use in place of a
division, over the densities a run meets and far beyond, plain and scaled as 16-bit
states are: their error in units of the last place of the result against a reciprocal
in more bits.

Bounds: an approximation r with 1 - a r = e is improved to r (1 + e + e^2), error e^3,
in double, and to r (1 + e), error e^2, in float.  The double approximation keeps 20
bits of the fraction (|e| < 2^-19): 2^-57 and the last rounding, below 0.5 + 2^-57 /
2^-53 = 0.5625 of a last place.  The float one is documented to 2^-23 for arguments in
[1, 2], two last places (|e| < 2^-22): 2 as it is, and 0.5 + 2^-44 / 2^-24, below 0.51,
improved.  An IEEE division: 0.5."""
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "lbm_kernels.cuh"
namespace lbmk { Shift<double> far_field_shift(const double*) { return {}; } }

// kind 0: v_rcp, 1: rcp_full
template <typename C>
__global__ void eval(const C* a, C* r, int n, int kind) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) r[k] = kind ? lbmk::rcp_full(a[k]) : lbmk::v_rcp(a[k]);
}

// 1 / a - r in last places of 1 / a, from the exact residual 1 - a r (one fma in C's next wider arithmetic)
static double off(float a, float r) {
  const double x = 1.0 / (double)a;
  const float f = (float)x;
  return std::fabs((double)r - x) / ((double)std::nextafterf(std::fabs(f), INFINITY) - std::fabs(f));
}
static double off(double a, double r) {
  const double q = 1.0 / a, ulp = std::nextafter(std::fabs(q), INFINITY) - std::fabs(q);
  const double e = std::fma(-a, r, 1.0);  // exact but for its own rounding
  return std::fabs(e / a) / ulp;
}

template <typename C>
static int measure(const char* name, int kind, double lo, double hi, double bound) {
  constexpr int N = 1 << 22;
  std::vector<C> a(N), r(N);
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> d(std::log(lo), std::log(hi));
  for (C& v : a) v = (C)std::exp(d(g));
  C *da, *dr;
  cudaMalloc(&da, N * sizeof(C));
  cudaMalloc(&dr, N * sizeof(C));
  cudaMemcpy(da, a.data(), N * sizeof(C), cudaMemcpyHostToDevice);
  eval<C><<<N / 256, 256>>>(da, dr, N, kind);
  if (cudaMemcpy(r.data(), dr, N * sizeof(C), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  double worst = 0;
  int misrounded = 0;
  for (int k = 0; k < N; ++k) {
    worst = std::fmax(worst, off(a[k], r[k]));
    misrounded += r[k] != (C)(C(1) / a[k]);
  }
  std::printf("%s [%g, %g]: %.6f last places, %.2g not as a division rounds\n", name, lo, hi, worst,
              (double)misrounded / N);
  cudaFree(da);
  cudaFree(dr);
  return worst > bound;
}

int main() {
  int bad = 0;
  const double ranges[][2] = {{0.9, 1.1}, {0.25, 4.0}, {0.25 * 4096, 4.0 * 4096}, {1e-6, 1e6}};
  for (const auto& q : ranges) {
    bad |= measure<double>("double v_rcp", 0, q[0], q[1], 0.5625);
    bad |= measure<double>("double rcp_full", 1, q[0], q[1], 0.5625);
    bad |= measure<float>("float v_rcp", 0, q[0], q[1], 2.0);
    bad |= measure<float>("float rcp_full", 1, q[0], q[1], 0.51);
  }
  return bad;
}
"""


def test_reciprocals(tmp_path):
    from paper_2005_08674_gb300 import build
    src, exe = tmp_path / "rcp.cu", tmp_path / "rcp"
    src.write_text(SRC)
    r = subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                        "-I", build.INCLUDE, str(src), "-o", str(exe)], capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
