"""The taps of Eq. 5 as the host builds them are those that the device builds for
the no-allocation path: the source position c + (i - c) s is one fused step,
rounded once, on either side.  Staging is sized from the host's taps, so another
rounding there could leave it a row short.  Compiled as host code and compared
with exact rational arithmetic."""

import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "ssoct_internal.h"
int main() {
  int n;
  double s;
  while (scanf("%d %la", &n, &s) == 2)
    for (int i = 0; i < n; ++i) {
      const ssoct::Tap t = ssoct::eq5_tap(i, n, s);
      printf("%d %a %a\n", t.base, (double)t.w0, (double)t.w1);
    }
  return 0;
}
"""


def _tap(i, n, s):
    c = Fraction(n, 2)
    u = Fraction(float(c + (i - c) * Fraction(s)))  # rounded once, as by a fused multiply-add
    i0 = u.numerator // u.denominator
    a = float(u - i0)
    w = {i0: np.float32(1.0 - a), i0 + 1: np.float32(a)}
    base = min(max(i0, 0), n - 2)
    inside = {k: v for k, v in w.items() if 0 <= k < n}
    return base, float(inside.get(base, 0)), float(inside.get(base + 1, 0))


# sweeps (first and last wavelength, frames) with ratios below and above 1; 800 to
# 880 nm puts source positions of 384 pixels next to whole numbers
@pytest.mark.parametrize("n,first,last,frames", [(384, 800e-9, 880e-9, 16), (64, 800e-9, 850e-9, 16), (640, 800e-9, 700e-9, 16),
                                                 (128, 800e-9, 1600e-9, 16)])
def test_host_taps_are_fused(tmp_path, n, first, last, frames):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "t.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-O3", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")], check=True)
    lam = [first + (last - first) * t / (frames - 1) for t in range(frames)]
    ratios = [v / lam[0] for v in lam]
    text = "\n".join(f"{n} {r.hex()}" for r in ratios) + "\n"
    out = subprocess.run([str(tmp_path / "t")], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    got = [(int(b), float.fromhex(x), float.fromhex(y)) for b, x, y in (line.split() for line in out if line)]
    want = [_tap(i, n, r) for r in ratios for i in range(n)]
    assert len(got) == len(want)
    assert got == want
