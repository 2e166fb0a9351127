"""The lateral kernel's default schedule (lateral_pick), run as host code: for
every kind of frame count, items per frame and ring size, each item is handed
out once, every dependency has a lower ticket, and the ring is not exceeded."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "ssoct_internal.h"
int main() {
  int frames, nr, nc, most;
  while (scanf("%d %d %d %d", &frames, &nr, &nc, &most) == 4) {
    const ssoct::LateralPick p = ssoct::lateral_pick(frames, nr + nc, most);
    ssoct::LateralSchedule s{frames, nr, nc, p.lag, p.slots};
    std::vector<long long> row(frames * nr, -1), col(frames * nc, -1);
    int bad = 0;
    for (long long t = 0; t < s.total(); ++t) {
      int kind, f, item;
      s.decode((unsigned)t, kind, f, item);
      std::vector<long long>& v = kind == 0 ? row : col;
      const int n = kind == 0 ? nr : nc;
      if (f < 0 || f >= frames || item < 0 || item >= n || v[f * n + item] != -1) { ++bad; continue; }
      v[f * n + item] = t;
    }
    for (int f = 0; f < frames; ++f) {
      for (int c = 0; c < nc; ++c)
        for (int r = 0; r < nr; ++r) bad += row[f * nr + r] >= col[f * nc + c];
      if (f >= p.slots)
        for (int c = 0; c < nc; ++c)
          for (int r = 0; r < nr; ++r) bad += col[(f - p.slots) * nc + c] >= row[f * nr + r];
    }
    printf("%d %d %d\n", p.lag, p.slots, bad);
  }
  return 0;
}
"""

# frames, row items, column items, ring slots: 1024^2 (8 slots of 64 MiB), 640^2
# with a window, 256^2 with the ring larger and smaller than the sweep, 64^2
# (every frame in the ring), and the passes over one to a few new frames
CASES = [(256, 128, 128, 8), (13, 128, 128, 8), (1, 128, 128, 8), (2, 128, 1, 8), (160, 80, 50, 23), (512, 16, 16, 128),
         (64, 16, 16, 128), (64, 16, 16, 13), (32, 2, 1, 2048), (16, 2, 2, 6), (3, 2, 2, 6), (4, 2, 2, 6), (5, 96, 96, 14)]


@pytest.fixture(scope="module")
def picks(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("pick")
    (d / "s.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, str(d / "s.cu"), "-o", str(d / "s")], check=True)
    text = "\n".join(" ".join(map(str, c)) for c in CASES) + "\n"
    out = subprocess.run([str(d / "s")], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    return {c: tuple(map(int, line.split())) for c, line in zip(CASES, out)}


@pytest.mark.parametrize("case", CASES)
def test_default_schedule_drains(picks, case):
    frames, _, _, most = case
    lag, slots, bad = picks[case]
    assert bad == 0
    assert 0 <= lag < max(slots, 1) <= max(most, 1) and lag <= max(0, frames - 1)
