"""The streamed adjoint row pass's sharing of (band of rows, frame) pairs, run as
host code: every pair is summed once, no FP32 partial sum is longer than a chunk
of eight frames, whole chunks are stored by one CTA, and the slots of split ones
are exactly those that are zeroed first, with two parts each."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "adjoint_share.h"
int main() {
  int bands, nt, ctas, bad_total = 0, used = 0;
  while (scanf("%d %d %d", &bands, &nt, &ctas) == 3) {
    const ssoct::RowsAdjShare s{bands, nt, ctas, 8};
    if (!s.fits()) continue;
    ++used;
    const int slots = (nt + 7) / 8;
    std::vector<int> frames(bands * nt, 0), stores(bands * slots, 0), adds(bands * slots, 0), zeroed(bands * slots, 0);
    for (int c = 1; c < ctas; ++c)
      if (s.splits(c)) ++zeroed[s.band(s.first(c)) * slots + s.slot(s.first(c))];
    int bad = s.first(0) != 0 || s.first(ctas) != bands * nt;
    for (int c = 0; c < ctas; ++c) {
      const int lo = s.first(c), hi = s.first(c + 1);
      int run = 0;
      for (int i = lo; i < hi; ++i) {
        ++frames[i];
        bad += ++run > 8;
        if (!s.closes(i, hi)) continue;
        ++(s.whole(i, lo, hi) ? stores : adds)[s.band(i) * slots + s.slot(i)];
        run = 0;
      }
      bad += run != 0;
    }
    for (int f : frames) bad += f != 1;
    for (int k = 0; k < bands * slots; ++k)
      bad += !((stores[k] == 1 && adds[k] == 0 && zeroed[k] == 0) || (stores[k] == 0 && adds[k] == 2 && zeroed[k] == 1));
    if (bad) printf("%d bands, %d frames, %d CTAs: %d\n", bands, nt, ctas, bad);
    bad_total += bad;
  }
  printf("%d\n", used);
  return bad_total != 0;
}
"""


def test_parts_of_eight_frames(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "s.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, str(tmp_path / "s.cu"), "-o", str(tmp_path / "s")], check=True)
    cases = [(b, n, c) for b in (2, 4, 8, 16, 24, 32, 48, 64, 80, 96, 128) for n in (16, 32, 64, 96, 128, 160, 200, 256, 512, 100)
             for c in (1, 7, 132, 148, 152, 160)]
    r = subprocess.run([str(tmp_path / "s")], input="\n".join("%d %d %d" % c for c in cases), capture_output=True, text=True)
    assert r.returncode == 0 and int(r.stdout.split()[-1]) > 100, r.stdout
