"""The ion-ion pass's special functions (csrc/sfu.cuh) against the host's 64-bit ones: each instruction within 2^-22,
e^x with two more roundings of its exponent, |x| 2^-23, over the arguments whose results are normal numbers."""
import subprocess

import pytest

from paper_2509_24742_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "sfu.cuh"
__global__ void k(int n, const float *x, const float *p, float *y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = srbe::exp_n(x[i]);
  y[n + i] = srbe::rsqrt_n(p[i]);
  y[2 * n + i] = srbe::rcp_n(p[i]);
}
int main() {
  const int n = 1 << 20;
  std::vector<float> x(n), p(n), y(3 * n);
  for (int i = 0; i < n; ++i) {
    x[i] = -87.0f * i / n;
    p[i] = std::exp2(-30.0f + 60.0f * i / n);
  }
  float *d = nullptr;
  if (cudaMalloc(&d, sizeof(float) * 5 * n) != cudaSuccess) return 2;
  cudaMemcpy(d, x.data(), sizeof(float) * n, cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, p.data(), sizeof(float) * n, cudaMemcpyHostToDevice);
  k<<<n / 256, 256>>>(n, d, d + n, d + 2 * n);
  if (cudaMemcpy(y.data(), d + 2 * n, sizeof(float) * 3 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  cudaFree(d);
  double w[3] = {0, 0, 0};                       // errors in units of their bounds
  for (int i = 0; i < n; ++i) {
    const double u = std::ldexp(1.0, -22);
    w[0] = std::fmax(w[0], std::fabs(y[i] / std::exp((double)x[i]) - 1) / (u + std::fabs(x[i]) * u / 2));
    w[1] = std::fmax(w[1], std::fabs(y[n + i] * std::sqrt((double)p[i]) - 1) / u);
    w[2] = std::fmax(w[2], std::fabs(y[2 * n + i] * (double)p[i] - 1) / u);
  }
  printf("%.3f %.3f %.3f\n", w[0], w[1], w[2]);
}
"""


def test_special_functions_within_their_bounds(tmp_path):
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0
    print("errors of exp, rsqrt and reciprocal in units of their bounds:", r.stdout)
    assert all(float(v) <= 1.0 for v in r.stdout.split())


QUOTIENT = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <vector>
#include "sfu.cuh"
__global__ void k(int n, const float *a, const float *d, float *y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = srbe::quotient(a[i], d[i], srbe::rcp_n(d[i]));
}
int main() {
  const int n = 1 << 20;
  std::vector<float> a(n), d(n), y(n);
  uint64_t w = 1;
  for (int i = 0; i < n; ++i) {
    w = w * 6364136223846793005ull + 1442695040888963407ull;
    const double u = (double)(w >> 11) / 9007199254740992.0;
    d[i] = 1.0f + (float)std::exp2(-30.0 + 90.0 * i / n);
    a[i] = (float)((u - 0.5) * std::exp2((i % 61) - 30));
  }
  float *m = nullptr;
  if (cudaMalloc(&m, sizeof(float) * 3 * n) != cudaSuccess) return 2;
  cudaMemcpy(m, a.data(), sizeof(float) * n, cudaMemcpyHostToDevice);
  cudaMemcpy(m + n, d.data(), sizeof(float) * n, cudaMemcpyHostToDevice);
  k<<<n / 256, 256>>>(n, m, m + n, m + 2 * n);
  if (cudaMemcpy(y.data(), m + 2 * n, sizeof(float) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  cudaFree(m);
  double worst = 0;
  for (int i = 0; i < n; ++i)
    if (a[i] != 0.0f) worst = std::fmax(worst, std::fabs((double)y[i] * d[i] / a[i] - 1) * 16777216.0);
  printf("%.6f\n", worst);
}
"""


def test_quotient_is_left_with_its_own_rounding(tmp_path):
    """Reciprocal (2^-22) and product (2^-24) leave a quotient within 1.25 2^-22, its residual times a reciprocal
    that far off corrects it to 2^-43, and the last rounding is 2^-24."""
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(QUOTIENT)
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0
    print("error of the quotient in units of 2^-24:", r.stdout)
    assert float(r.stdout) <= 1.0 + 2.0 ** -18
