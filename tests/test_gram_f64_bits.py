"""Host checks of the integer arithmetic of the FP64 Gram
(csrc/gram_f64.cu): the fixed-point columns, their balanced base-256 digits
and the rounded division by n, against Python's exact integers and
fractions.  The functions are host-and-device code; the test builds a small
host program around them with nvcc (no GPU needed)."""
import math
import os
import random
import shutil
import struct
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2106_09382_gb300", "csrc")

PROGRAM = r"""
#include "gram_f64.cu"
#include <cstdio>
namespace concord {
void note_launches(unsigned) {}
int col_stats_chunks(int) { return 1; }
cudaError_t launch_col_stats_chunked(const void*, int, int, int, int, int, double*, double*, int*,
                                     double*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_apply_prep(const void*, int, int, int, int, const double*, const double*, void*,
                              int, int, cudaStream_t, const int*) { return cudaSuccess; }
cudaError_t launch_syrk_f64(const double*, int, int, int, double*, int, double, cudaStream_t,
                            const int*) { return cudaSuccess; }
}
int main() {
  char op;
  while (scanf(" %c", &op) == 1) {
    if (op == 'f') {
      unsigned long long b; int e;
      if (scanf("%llx %d", &b, &e) != 2) return 1;
      const long long F = concord::f64_to_fixed(concord::fb_u2d(b), e);
      printf("%lld", F);
      for (int s = 0; s < 7; ++s) printf(" %d", concord::fixed_digit(F, s));
      printf("\n");
    } else {
      long long h; int x, n;
      if (scanf("%lld %d %d", &h, &x, &n) != 3) return 1;
      int k = 0;
      while ((1ll << k) < n) ++k;
      const unsigned long long r = (unsigned long long)(
          (((unsigned __int128)1 << (63 + k)) + (unsigned)n / 2) / (unsigned)n);
      printf("%016llx\n", concord::fb_d2u(concord::fixed_over_n(h, x, r, k)));
    }
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("gram_f64")
    src = d / "t.cu"
    src.write_text(PROGRAM)
    exe = str(d / "t")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", exe, str(src)], check=True)
    return lambda lines: subprocess.run([exe], input="\n".join(lines), text=True, check=True,
                                        capture_output=True).stdout.splitlines()


def test_fixed_point_and_digits(program):
    rng = random.Random(1)
    cases = []
    for e in (-3, 0, 1, 2, 5):
        for z in (0.0, 2.0 ** e, -2.0 ** e, math.nextafter(2.0 ** e, 0), 2.0 ** (e - 57),
                  2.0 ** (e - 58), 5e-324, -2.0 ** (e - 1)):
            cases.append((z, e))
        for _ in range(400):
            cases.append((rng.uniform(-1, 1) * 2.0 ** (e - rng.randint(0, 60)), e))
    out = program("f %016x %d" % (struct.unpack("<Q", struct.pack("<d", z))[0], e) for z, e in cases)
    assert len(out) == len(cases)
    for (z, e), line in zip(cases, out):
        F, *dig = map(int, line.split())
        assert abs(F - Fraction(z) * Fraction(2) ** (56 - e)) <= Fraction(1, 2)
        assert F == sum(d * 256 ** (6 - s) for s, d in enumerate(dig))
        assert -256 <= dig[0] <= 256 and all(-128 <= d <= 127 for d in dig[1:])


def test_division_by_n_rounds_once(program):
    rng = random.Random(2)
    cases = []
    for n in (32, 33, 64, 100, 2000, 2001, 4096, 16384, 99991):
        for h in (0, 1, -1, 2 ** 62, -2 ** 62, 2 ** 53 + 1, n, -n, 3 * n):
            cases.append((h, -30, n))
        for _ in range(300):
            cases.append((rng.randint(-2 ** 62, 2 ** 62) >> rng.randint(0, 61),
                          rng.randint(-800, 700), n))
    out = program("d %d %d %d" % c for c in cases)
    for (h, x, n), line in zip(cases, out):
        got = struct.unpack("<d", struct.pack("<Q", int(line, 16)))[0]
        want = Fraction(h) * Fraction(2) ** x / n
        # the reciprocal carries 2^-64 and the truncated product 2^-63: half
        # an ulp (2^-53 relative) and those
        assert abs(Fraction(got) - want) <= abs(want) * (Fraction(1, 2 ** 53) + Fraction(1, 2 ** 61))
