"""The FP64 form's radial tables on the host (csrc/pairfix.cuh compiled by the host compiler) against long double
arithmetic, over the cutoffs and splittings where the period, the octave or the screening changes.

Bounds.  A factor is a polynomial of four 62-bit integer coefficients (truncated products, 3 units of 2^-62 each) with
a tail rounded in FP32 below 2^-53 of 1 / r^3, S is rounded to 2^-64 of R1^2 and the result to a double: 2^-53 three
times over, and 1e-15 leaves a factor of three.  Every entry has to keep its last unit, 2^(E - 62), and a value of
one such unit (E - 62 - 63 in the assembled exponent) within the normal doubles."""
import os
import shutil
import subprocess

import pytest

from paper_2509_24742_gb300 import build

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "pairfix.cuh"
using namespace srbe;
static long double g(long double a, long double r) {
  return (erfcl(a * r) / r + 1.12837916709551257389615890312154517L * a * expl(-a * a * r * r)) / (r * r);
}
static long double f(long double a, long double r) { return erfcl(a * r) / r; }
int main() {
  double worst[3] = {0, 0, 0};
  int low = 0;
  for (double rc : {0.98, 0.99, 1.2, 1.6, 2.5}) for (double alpha : {0.9, 1.87, 3.5, 8.0, 17.0, 25.9, 26.2})
    for (double ie : {3.0, 19.79, 40.0}) {
      const double R1 = std::exp2(std::ceil(std::log2(rc + 0.01)));
      std::vector<PairCoef> t[3];
      for (int i = 0; i < kPtSize; ++i) {
        double s0, half;
        pair_interval(i, R1, s0, half);
        RadialTaylor a, b;
        radial_taylor(s0, alpha, half, a);
        radial_taylor(s0, ie, half, b);
        t[0].push_back(pair_coef(a.g, nullptr, 1.0));
        t[1].push_back(pair_coef(a.g, b.g, 1.0));
        t[2].push_back(pair_coef(a.f, b.f, 1.0));
        for (auto &v : t) low = std::min(low, (int)(pf_bits(v.back().c7) & 4095) - 2048);
      }
      for (int k = 0; k < 20000; ++k) {
        const double x = (R1 / 64 + (rc - R1 / 64) * (k + 0.5) / 20000) / R1;
        const uint64_t S = (uint64_t)(x * x * 9223372036854775808.0);
        if (S < kPtMin) continue;
        const PairArg p = pair_arg(S);
        const long double r = sqrtl((long double)S / 9223372036854775808.0L) * R1;
        const long double ref[3] = {g(alpha, r), g(alpha, r) - g(ie, r), f(alpha, r) - f(ie, r)};
        for (int w = 0; w < 3; ++w) {
          const double e = (double)(fabsl(pair_poly(t[w][p.idx], p) - ref[w]) * (w < 2 ? r * r * r : r));
          if (!(e <= worst[w])) worst[w] = e;
        }
      }
    }
  printf("%.3e %.3e %.3e %d\n", worst[0], worst[1], worst[2], low);
}
"""


def test_radial_tables_on_the_host(tmp_path):
    cxx = shutil.which("g++")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    if cxx is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-w", "-I", cuda, "-I", build.CSRC, str(src), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    print("worst error of the ion-ion and ion-electrode force factors and the potential:", out[:3], "lowest E:", out[3])
    assert all(float(v) < 1e-15 for v in out[:3])
    assert 1023 + int(out[3]) - 63 >= 1
