"""The exponentials and the logarithm of the scaled matrix products, compiled
for the host, against long double arithmetic (no GPU)."""
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
#include "logprod.cuh"
using namespace fstgpu;
typedef long double ld;
// the worst and the mean error of 400,000 arguments of one kind, in units of 2^-24
int main(int, char** v) {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(0, 1);
  const int kind = atoi(v[1]);
  ld worst = 0, sum = 0;
  long n = 0;
  auto add = [&](ld e) {
    e *= 0x1p24L;
    if (fabsl(e) > worst) worst = fabsl(e);
    sum += e;
    ++n;
  };
  for (long i = 0; i < 400000; ++i) {
    if (kind == 0 || kind == 1) {  // exp(x), relative: over its range, near 0
      const float x = kind == 0 ? (float)(-87 * U(g)) : -(float)exp(-20 * U(g));
      add((ld)exp_neg(x) / expl((ld)x) - 1);
    } else if (kind <= 4) {  // exp(x - m), relative: scales below 0, above, of any size
      const float s = kind == 2 ? (float)(-200 * U(g)) : kind == 3 ? (float)(200 * U(g)) : (float)(1e7 * (U(g) - 0.5));
      const float m = scale_of(s), x = s - (float)(60 * U(g));
      if (x > m || x - m < -80) continue;
      add((ld)exp_below(x, m) / expl((ld)x - (ld)m) - 1);
    } else {  // r + c + log x, beyond half a rounding of the result
      const float R = kind == 5 ? 60.f : 1e6f;
      const float r = scale_of(R * (float)(U(g) - 0.5)), c = scale_of(i % 3 ? -r + (float)(50 * U(g)) : R * (float)(U(g) - 0.5));
      const float x = (float)exp(-60 * U(g)) * (float)(1 + U(g));
      const ld w = (ld)r + (ld)c + logl((ld)x);
      const float y = add_log(r, c, x);
      const ld half = 0.5L * (nextafterf(fabsf(y), INFINITY) - fabsf(y)), e = (ld)y - w;
      add(fabsl(e) <= half ? 0 : (fabsl(e) - half));
    }
  }
  const float inf = INFINITY;
  const float zero = exp_neg(-inf) + exp_neg(NAN) + exp_neg(-87.4f) + exp_neg(-3e38f) + exp_below(-inf, -inf) +
                     exp_below(-inf, 0.f) + exp_below(-inf, 3e38f) + exp_below(-3e38f, 3e38f) + exp_below(-inf, -2e6f);
  printf("%.6Lg %.6Lg %ld %g %g\n", worst, sum / n, n, zero, exp_neg(0.f) + exp_neg(-0.f));
}
"""

# the exponential: its last rounding (1 of 2^-24 below 1, relative), its
# argument's (a quarter) and the series'; a difference with its error term a
# rounding more; the mean a tenth of expf's 0.1 to 0.18.  r + c + log x: the
# logarithm of f and the small parts, of size below 0.36 and 0.01, within 1/2
WORST = [1.5, 1.5, 1.5, 2.5, 2.5, 0.5, 0.5]
MEAN = [0.02, 0.02, 0.02, 0.02, 0.02, 0.5, 0.5]


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("logprod")
    (d / "t.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")],
                   check=True)
    return str(d / "t")


@pytest.mark.parametrize("kind", range(len(WORST)))
def test_errors_within_bounds(harness, kind):
    out = subprocess.run([harness, str(kind)], check=True, capture_output=True, text=True).stdout.split()
    worst, mean, n, zero, two = (float(x) for x in out)
    assert n > 100_000 and zero == 0.0 and two == 2.0, out
    assert worst <= WORST[kind] and abs(mean) <= MEAN[kind], out
