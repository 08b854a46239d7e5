"""Host check of the wave form's tile schedule (csrc/wave.cuh, wave_tile): the
tiles a sweep's owners walk cover every pair exactly once, give each row its
pairs in the colour order of the circle method (Section 3.2), agree between
the two owners of a tile on the exchange slot, use no slot twice, and never
wait in a circle -- neither for a partner's entries nor, in the tiles with
vertex 0's pairs, for its changes in the blocks above."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2106_09382_gb300", "csrc")

PROGRAM = r"""
#include "wave.cuh"
#include <cstdio>
#include <cstdlib>
#include <set>
#include <vector>
using namespace concord;
static void die(const char* what, int p, int a, int b) { printf("%s p=%d %d %d\n", what, p, a, b); exit(1); }
static void check(int p) {
  const int P = p + (p & 1) - 1, nb = wave_blocks(p), slots = wave_slots(p);
  std::vector<std::vector<WaveTile>> seq(nb);
  for (int I = 0; I < nb; ++I) {
    std::set<int> used;
    for (int v = 0;; ++v) {
      const WaveTile t = wave_tile(I, nb, P, v);
      if (t.J < 0) break;
      if (t.J >= nb || t.slot < 0 || t.slot >= slots || !used.insert(t.slot).second) die("slot", p, I, v);
      if (t.hi - t.lo > 63) die("range", p, I, v);
      seq[I].push_back(t);
    }
  }
  // every row's partners in colour order (each pair seen from both rows)
  for (int I = 0; I < nb; ++I)
    for (int l = 0; l < kWaveB; ++l) {
      const int i = kWaveB * I + l;
      if (i < 1 || i >= p) continue;
      std::vector<int> got;
      for (const WaveTile& t : seq[I])
        for (int s = t.hi; s >= t.lo; s -= 2) {
          const int j = s - i;
          if (j < kWaveB * t.J || j >= kWaveB * t.J + kWaveB || j < 1 || j > P) continue;
          const int q = j == i ? 0 : j;  // would meet itself: vertex 0
          if (q == 0 || j < p) got.push_back(q);
        }
      size_t n = 0;
      for (int c = 0; c < P; ++c) {
        const int q = cm_partner(i, c, P);
        if (q >= p) continue;
        if (n >= got.size() || got[n] != q) die("order", p, i, c);
        ++n;
      }
      if (n != got.size()) die("extra", p, i, (int)got.size());
    }
  // progress: an owner's next tile needs its partner's entries (published
  // when the partner stands at the same tile) and, with vertex 0's pairs,
  // every such pair of the blocks above
  std::vector<size_t> at(nb, 0);
  std::vector<int> zleft(nb, 0);
  for (int b = 0; b < nb; ++b)
    for (int v = kWaveB * b; v < kWaveB * b + kWaveB; ++v) zleft[b] += v >= 1 && v < p;
  for (bool moved = true; moved;) {
    moved = false;
    for (int I = 0; I < nb; ++I) {
      if (at[I] >= seq[I].size()) continue;
      const WaveTile& t = seq[I][at[I]];
      if (t.J == I) {
        bool ready = true;
        if ((t.hi & 1) == 0)
          for (int b = I + 1; b < nb; ++b) ready = ready && zleft[b] == 0;
        if (!ready) continue;
        if ((t.hi & 1) == 0)
          for (int s = t.hi; s >= t.lo; s -= 2) {
            const int v = s / 2;
            if (v / kWaveB == I && v >= 1 && v < p) --zleft[I];
          }
        ++at[I];
        moved = true;
      } else if (at[t.J] < seq[t.J].size()) {
        const WaveTile& u = seq[t.J][at[t.J]];
        if (u.J == I && u.slot == t.slot) {
          if (u.lo != t.lo || u.hi != t.hi) die("sums", p, I, t.J);
          ++at[I];
          ++at[t.J];
          moved = true;
        }
      }
    }
  }
  for (int I = 0; I < nb; ++I)
    if (at[I] != seq[I].size() || zleft[I] != 0) die("stuck", p, I, (int)at[I]);
}
int main() {
  for (int p = 2; p <= 330; ++p) check(p);
  for (int p : {511, 512, 513, 999, 1000, 1001, 1023, 1024, 1025, 2047, 2048}) check(p);
  printf("ok\n");
}
"""


def test_wave_tiles_cover_every_pair_in_colour_order(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "t.cu"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-I", CSRC,
                    "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
