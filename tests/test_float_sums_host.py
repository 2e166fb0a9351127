"""The sums over the volume (sum of P, sum of P^2) in expansions of floats, run as
host code, against exact values, also where one value outweighs all others.

Bound: the error terms of four values (at most 2^-24 of a partial sum each, seven of
them) are added in FP32, six roundings of at most 2^-25 relative: with random signs
an RMS below 2^-49 of the four's sum, and of the total.  (FP64 sums that meet by
atomics, 304 of them, leave 2^-51; a pair of floats leaves 2^-45 where small values
follow a large one.)"""

import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "float_sums.cuh"
// in: int32 trials, values (a multiple of 4), then the values.  out: S1, S2
int main(int, char** a) {
  FILE* f = fopen(a[1], "rb");
  int n[2];
  if (fread(n, 4, 2, f) != 2) return 1;
  std::vector<float> v((size_t)n[0] * n[1]);
  if (fread(v.data(), 4, v.size(), f) != v.size()) return 1;
  f = fopen(a[2], "wb");
  for (int i = 0; i < n[0]; ++i) {
    const float* x = v.data() + (size_t)i * n[1];
    // four threads' sums, joined as lanes are
    ssoct::FloatSums t[4] = {};
    for (int k = 0; k < n[1]; k += 4) t[k / 4 % 4].add4(x[k], x[k + 1], x[k + 2], x[k + 3]);
    for (int o = 2; o; o >>= 1)
      for (int k = 0; k < o; ++k) { t[k].p.add(t[k + o].p); t[k].q.add(t[k + o].q); }
    const double out[2] = {t[0].p.value(), t[0].q.value()};
    fwrite(out, 8, 2, f);
  }
  fclose(f);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("sums")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-O3", "-std=c++17", "-I", CSRC, str(d / "h.cu"), "-o", str(d / "h")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("kind", ["uniform", "speckle", "one large first", "one large later", "decades"])
def test_sums_against_exact(program, tmp_path, kind):
    rng = np.random.default_rng(7)
    trials, n = 400, 576
    v = rng.exponential(1.0, (trials, n)) if kind != "uniform" else rng.uniform(0.5, 1.0, (trials, n))
    if kind == "one large first":
        v[:, 1] = rng.uniform(1e4, 1e7, trials)
    elif kind == "one large later":
        v[:, 301] = rng.uniform(1e4, 1e7, trials)
    elif kind == "decades":
        v *= 10.0 ** rng.uniform(-8, 4, (trials, n))
    v = v.astype(np.float32)
    with open(tmp_path / "in", "wb") as f:
        f.write(np.array([trials, n], dtype=np.int32).tobytes() + v.tobytes())
    subprocess.run([program, str(tmp_path / "in"), str(tmp_path / "out")], check=True)
    got = np.fromfile(tmp_path / "out").reshape(trials, 2)
    err = np.zeros((trials, 2))
    for i in range(trials):
        x = [Fraction(float(t)) for t in v[i]]
        s1, s2 = sum(x), sum(t * t for t in x)
        for k, s in enumerate((s1, s2)):
            err[i, k] = float((Fraction(float(got[i, k])) - s) / s)
    rms = np.sqrt(np.mean(err ** 2, axis=0))
    assert rms.max() <= 2.0 ** -49, rms
