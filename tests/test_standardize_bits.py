"""Host check of the standardised values (csrc/fp_bits.cuh, std_value): formed
from pairs of floats they must be the float that rounding (x - mean) * inv in
FP64 gives, bit for bit -- over random data, data whose mean is large against
its spread, values next to the mean, integers, zeros, infinities and the ends
of the range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2106_09382_gb300", "csrc")

PROGRAM = r"""
#include "fp_bits.cuh"
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
using namespace concord;
static long bad = 0, seen = 0;
static void check(float x, double mean, double inv) {
  const StdCol c = std_col(mean, inv);
  volatile double d = (double)x - mean;
  volatile double v = d * inv;
  volatile float want = (float)v;
  const float got = std_value(x, c), w = want;
  ++seen;
  if (std::isnan(w) ? !std::isnan(got) : std::memcmp(&w, &got, 4) != 0)
    if (bad++ < 5) printf("x %a mean %a inv %a: %a, not %a\n", x, mean, inv, got, w);
}
int main() {
  std::mt19937_64 g(7);
  std::normal_distribution<double> nd;
  std::uniform_real_distribution<double> ud(0.0, 1.0);
  for (int col = 0; col < 4000; ++col) {
    const double spread = std::pow(10.0, 12.0 * ud(g) - 6.0);
    const double mean0 = (col % 4 == 0 ? 0.0 : (col % 4 == 1 ? 1.0 : 1e4 * ud(g))) * spread * nd(g);
    const double mean = col % 7 == 0 ? 0.0 : mean0 * (1.0 + 1e-9 * nd(g));
    const double inv = col % 5 == 0 ? 1.0 : 1.0 / (spread * (0.5 + ud(g)));
    for (int k = 0; k < 5000; ++k) {
      float x = (float)(mean0 + spread * nd(g));
      if (k % 50 == 0) x = std::nearbyintf(x);
      if (k % 50 == 1) x = (float)mean;
      if (k % 50 == 2) x = std::nextafterf((float)mean, 1e30f);
      if (k % 50 == 3) x = 0.f;
      check(x, mean, inv);
    }
  }
  const float ends[] = {0.f, -0.f, 1e-45f, 1e-38f, 3.4e38f, -3.4e38f, INFINITY, -INFINITY, NAN, 1.f};
  const double means[] = {0.0, 1e-300, 1e-40, 1.0, 1e38, 1e300}, invs[] = {1.0, 1e-40, 1e40, 1e-300, 1e300};
  for (float x : ends)
    for (double m : means)
      for (double i : invs) check(x, m, i);
  printf("%ld of %ld differ\n", bad, seen);
  return bad ? 1 : 0;
}
"""


def test_standardised_values_are_the_fp64_ones(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "s.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "s")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, "-gencode", "arch=compute_103a,code=sm_103a",
                    "-Xcompiler", "-ffp-contract=off", "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
