"""The wave form's quotient (csrc/wave.cuh, wave_quotient: products with a
correctly rounded reciprocal and their residuals) against the division: the
same bits wherever wave_plain holds, over random pairs, pairs of neighbouring
and extreme mantissas, and the ends of wave_plain's range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2106_09382_gb300", "csrc")

PROGRAM = r"""
#include "wave.cuh"
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
using namespace concord;
static uint64_t state = 88172645463325252ull;
static uint32_t rnd() { state ^= state << 13; state ^= state >> 7; state ^= state << 17; return (uint32_t)(state >> 16); }
static float of(uint32_t b) { float f; memcpy(&f, &b, 4); return f; }
static uint32_t bits(float f) { uint32_t b; memcpy(&b, &f, 4); return b; }
static long bad = 0, seen = 0;
static void check(float n, float d) {
  if (!wave_plain(n, d)) return;
  ++seen;
  volatile float q = n / d, y = 1.f / d;
  if (bits(q) != bits(wave_quotient(n, d, y)) && bad++ < 5) printf("%a / %a\n", n, d);
}
int main() {
  for (long k = 0; k < 20000000; ++k) {
    const int en = 127 - 70 + (int)(rnd() % 141), ed = 127 - 40 + (int)(rnd() % 81);
    const uint32_t sn = (rnd() & 1) << 31;
    uint32_t mn = rnd() & 0x7fffff, md = rnd() & 0x7fffff;
    switch (k % 5) {  // random; extreme and neighbouring mantissas
      case 1: md = (rnd() & 1) ? rnd() & 7 : 0x7fffff - (rnd() & 7); break;
      case 2: mn = (rnd() & 1) ? rnd() & 7 : 0x7fffff - (rnd() & 7); break;
      case 3: mn = (md + (rnd() & 15) - 7) & 0x7fffff; break;
      case 4: md = (rnd() & 7) << 20 | (rnd() & 3); break;
    }
    check(of(sn | (uint32_t)en << 23 | mn), of((uint32_t)ed << 23 | md));
  }
  for (uint32_t md = 0; md < 0x800000; md += 1)  // every mantissa of the denominator
    check(of(0x3f800000u | (rnd() & 0x7fffff)), of(0x40000000u | md));
  check(0.f, 1.5f);
  if (bits(wave_quotient(0.f, 1.5f, 1.f / 1.5f)) != 0) ++bad;
  printf("%ld of %ld differ\n", bad, seen);
  return bad || seen < 25000000 ? 1 : 0;
}
"""


def test_quotient_is_the_division(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "q.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "q")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler",
                    "-ffp-contract=off", "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
