"""rcp_newton and rsqrt_newton (csrc/common.cuh) against CUDA's 1.0 / x and, in extended precision, 1 / sqrt(x),
over random mantissas (and runs of them next to powers of two) and the exponents their callers use."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1704_02357_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
#include "common.cuh"
constexpr int n = 1 << 22;
__global__ void k(const double* x, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = pspec::rcp_newton(x[i]);
  out[n + i] = 1.0 / x[i];
  out[2 * n + i] = pspec::rsqrt_newton(x[i]);
}
int main() {
  std::vector<double> x(n), y(3 * (size_t)n);
  std::mt19937_64 g(11);
  for (int i = 0; i < n; i++) {
    unsigned long long m = g() & 0xfffffffffffffull, e = 1023 - 100 + g() % 200;
    if (i < 3000) m = i % 2 ? 0xfffffffffffffull - i / 2 : (unsigned long long)i / 2;
    const unsigned long long b = (e << 52) | m;
    std::memcpy(&x[i], &b, 8);
  }
  double *dx, *dy;
  if (cudaMalloc(&dx, 8 * (size_t)n) != cudaSuccess || cudaMalloc(&dy, 24 * (size_t)n) != cudaSuccess) return 1;
  cudaMemcpy(dx, x.data(), 8 * (size_t)n, cudaMemcpyHostToDevice);
  k<<<n / 256, 256>>>(dx, dy);
  if (cudaMemcpy(y.data(), dy, 24 * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  long differ = 0;
  double worst = 0, worst_rsqrt = 0;
  for (int i = 0; i < n; i++) {
    const double ulp = std::nextafter(y[n + i], INFINITY) - y[n + i];
    differ += y[i] != y[n + i];
    worst = std::fmax(worst, std::fabs(y[i] - y[n + i]) / ulp);
    const long double r = 1.0L / std::sqrt((long double)x[i]);
    worst_rsqrt = std::fmax(worst_rsqrt, (double)(std::fabs(y[2 * (size_t)n + i] - r) / (std::nextafter((double)r, INFINITY) - (double)r)));
  }
  std::printf("%ld %.17g %.17g\n", differ, worst, worst_rsqrt);
}
"""


def test_newton_against_the_library(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    (tmp_path / "t.cu").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", CSRC, str(tmp_path / "t.cu"), "-o", exe], check=True)
    differ, worst, worst_rsqrt = (float(v) for v in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split())
    # two steps leave 2^-80 before the last rounding: another result than the division's needs a quotient that close to
    # halfway between two numbers; a product and a sum are rounded in the last step of 1/sqrt(x)
    assert differ <= 4 and worst <= 1.0
    assert worst_rsqrt < 1.5
