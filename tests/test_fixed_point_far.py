"""Neighbours of any relative size in the hop sums of the fixed-point stencil (csrc/fixed.cuh, hop_round): the functions
that the kernel calls, on the host, under the undefined-behaviour checker."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1712_01505_gb300", "csrc")

SRC = r"""
#include <math.h>
#include <stdio.h>
#include <random>
#include "fixed.cuh"
using namespace qcd::fx;
int main() {
  std::mt19937_64 rng(1);
  const int64_t most = (int64_t)ldexpl(5.0L / 4 * sqrtl(6.0L), 61);  // the bound on |HH|
  std::uniform_int_distribution<int64_t> all(-most, most);
  double sum = 0;
  long n = 0;
  for (int diff = 0; diff <= 2000; ++diff) {  // E - e, all that exponent fields allow
    const int d = (diff < 100 ? diff : 100) + 3;
    for (int k = 0; k < 2000; ++k) {
      const int64_t H = k == 0 ? most : k == 1 ? -most : k == 2 ? 0 : k == 3 ? -1 : all(rng);
      const float C = ldexpf((float)(rng() % 2001) / 1000.f - 1.f, 33);
      const long double exact = ldexpl((long double)H, -d - (diff > 100 ? diff - 100 : 0));
      long double got = 0;
      if (d < kFar) got = (long double)hop_round(H + hop_half(d, k & 1), 0.f, ldexpf(1.f, -d), d);
      if (fabsl(got - exact) > (d < kFar ? 0.5L : 1.6L)) return printf("d %d H %lld: %Lg, exact %Lg\n", d, (long long)H, got, exact), 1;
      if (d < kFar) {
        const long double both = (long double)hop_round(H + hop_half(d, k & 1), C, ldexpf(1.f, -d), d);
        if (fabsl(both - exact - ldexpl((long double)C, -d)) > 1.0L) return printf("d %d: C\n", d), 1;
      }
      if (d == 3) sum += (double)(got - exact), ++n;
    }
  }
  // no bias: the mean of n errors uniform on (-1/2, 1/2), ties alternating, 0.29 / sqrt(n) rms
  if (fabs(sum / n) > 6 * 0.29 / sqrt((double)n)) return printf("mean error %g\n", sum / n), 1;
  return 0;
}
"""


def test_hop_sums_of_far_neighbours(tmp_path):
    src, exe = tmp_path / "far.cpp", tmp_path / "far"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=undefined", "-I", CSRC,
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
