"""The integer exponential, logarithm and float conversions of the log-sums,
compiled for the host, against long double arithmetic (no GPU)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1701_03038_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fixmath.cuh"
using namespace fstgpu;
typedef long double ld;
// the worst error of 400,000 arguments of one kind, in the unit its bound has
int main(int, char** v) {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(0, 1);
  const int kind = atoi(v[1]);
  ld worst = 0;
  for (long i = 0; i < 400000; ++i) {
    ld e = 0;
    if (kind < 4) {  // terms: exp(x) in units of 2^-40
      double x = kind == 0 ? -30 * U(g) : kind == 1 ? -exp(-45 * U(g)) : 0;
      if (kind == 2) x = -(double)(i % 5400) * 0.69314718055994531 / 128 * (1 + 1e-15 * (double)(i % 7 - 3));
      const double edge[] = {-0.0, 0.0, -5e-324, -1e-300, -0x1p-59, -0x1p-58, -28.4, -28.5, -31.99, -32.0, -1e300, -INFINITY};
      if (kind == 3) x = edge[i % 12];
      e = fabsl((ld)fx_exp40(x) - expl((ld)x) * 0x1p40L);
    } else if (kind < 7) {  // sums: log(s 2^-40), s from 2^40 to 2^64
      const int b = 40 + (int)(g() % 24);
      uint64_t s = (1ull << b) | (g() & ((1ull << b) - 1));
      if (kind == 5) s = (1ull << 40) + (g() & ((1ull << (g() % 40)) - 1));
      if (kind == 6) s = i & 1 ? ~0ull - (g() & 255) : (1ull << b) + (uint64_t)(i % 3) - 1;
      if (s < (1ull << 40)) s = 1ull << 40;
      const ld w = logl((ld)s) - 40 * logl(2.0L);
      e = fabsl((ld)fx_add_log40(0.0, s) - w);
    } else {  // conversions: the same bits
      uint64_t u = g();
      if (i % 2) u = (u & ~(0x7ffull << 52)) | ((uint64_t)(870 + g() % 290) << 52);
      if (i % 5 == 0) u &= ~0xfffffffull;
      const float f = fx_float((uint32_t)(g() >> 32) & (i % 8 ? ~0u : 0x807fffffu));
      const double d = i == 0 ? -INFINITY : i == 1 ? -0.0 : fx_double(u);
      if (d == d && fx_bits32(fx_narrow(d)) != fx_bits32((float)d)) e = 1;
      if (f == f && fx_bits(fx_widen(f)) != fx_bits((double)f)) e = 1;
    }
    if (e > worst) worst = e;
  }
  printf("%.6Lg\n", worst);
}
"""

# terms: the rounding (0.5) and 1/16 of a unit for the arithmetic; logarithms
# (below 16.7): half an ulp of the float64 result, 1.8e-15, and 1e-15
BOUNDS = [0.5625, 0.5625, 0.5625, 0.5625, 2.8e-15, 2.8e-15, 2.8e-15, 0.0]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("fixmath")
    (d / "t.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("kind", range(len(BOUNDS)))
def test_errors_within_bounds(harness, kind):
    got = float(subprocess.run([harness, str(kind)], check=True, capture_output=True, text=True).stdout)
    assert got <= BOUNDS[kind], got
