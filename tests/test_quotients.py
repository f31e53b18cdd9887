"""Quotients by a precomputed reciprocal (csrc/divide.cuh), built for the host
with g++ and compared with division bit for bit: every FP32 numerator of a
binade and random FP64 numerators over many binades, for divisors that the
solvers use (smoother constants, time steps, theta) and the extreme mantissas;
infinities, NaN, zeros and an infinite divisor's stand-in {1, 0}.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_2204_06083_gb300", "csrc")

PROG = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
#include "divide.cuh"
using namespace ebk;
template <class A>
static bool same(A x, A y) { return x == y || (std::isnan(x) && std::isnan(y)); }
int main() {
  long bad = 0;
  const double h = 2.0 / 1021;
  const double divisors[] = {0.5 * (1.1 + 1.0 / 30) * 2.0, 0.5 * (1.1 + 1.0 / 30) * 1.9375, 0.5 * (1.1 + 1.0 / 30) * 3.7e5,
                             h, 0.5, 1.0 / 12, 0.1, 3.0, 1.0 + 0x1p-23, 2.0 - 0x1p-23, 1.0 + 0x1p-52, 2.0 - 0x1p-52};
  std::mt19937_64 g(7);
  for (double d : divisors) {
    const DivBy<float> cf = DivBy<float>::of(d);
    for (uint32_t m = 0; m < (1u << 23); ++m) {
      const uint32_t bits = 0x3f800000u | m;
      float a;
      std::memcpy(&a, &bits, 4);
      if (!same(div_by(a, cf), a / cf.d)) ++bad;
    }
    const DivBy<double> cd = DivBy<double>::of(d);
    for (int i = 0; i < 1000000; ++i) {
      const uint64_t e = 1023 - 600 + g() % 1200, bits = (g() & 0x800fffffffffffffull) | e << 52;
      double a;
      std::memcpy(&a, &bits, 8);
      if (!same(div_by(a, cd), a / cd.d)) ++bad;
    }
    const double inf = std::numeric_limits<double>::infinity();
    for (double a : {0.0, inf, -inf, std::nan("")}) {
      if (!same(div_by(a, cd), a / cd.d)) ++bad;
      if (!same(div_by((float)a, cf), (float)a / cf.d)) ++bad;
    }
  }
  const DivBy<double> never{1.0, 0.0};
  for (double a : {1.0, -3.5e10, 0.0}) if (div_by(a, never) != 0.0) ++bad;
  std::printf("%ld\n", bad);
  return 0;
}
"""


def test_quotients_are_those_of_division(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(PROG)
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-I", HDR, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert int(out) == 0
