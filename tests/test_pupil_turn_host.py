"""The exponential of the pupil table, run as host code over phases of up to 1e5
half turns: within half a unit in the last place of a float of the exact value,
plus 2^-35.  (Its one rounding to float32, and the terms that are kept in single
precision: cos d - 1, at most 7.6e-5 in size and off by a few 2^-25 of that.)"""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include "pupil_turn.cuh"
int main() {
  std::vector<float4> cis(256);
  for (int k = 0; k < 256; ++k) {
    const double a = 3.14159265358979323846 * k / 128.0, c = std::cos(a), s = std::sin(a);
    cis[k] = make_float4((float)c, (float)(c - (float)c), (float)s, (float)(s - (float)s));
  }
  std::mt19937_64 gen(5);
  std::uniform_real_distribution<double> log_size(-6.0, 5.0), unit(-1.0, 1.0);
  const long double pi = 3.14159265358979323846264338327950288L;
  double worst = 0.0;
  for (int i = 0; i < 400000; ++i) {
    double t = unit(gen) * std::pow(10.0, log_size(gen));
    if (i % 4 == 0) t = std::rint(t * 256.0) / 256.0 + 1e-12 * unit(gen);  // ends of the remainder's range, zeros
    const int odd = i & 1;
    const float2 v = ssoct::cis_turn(t, odd, cis.data());
    const double r = t - 2.0 * std::rint(t / 2.0);  // exact
    const long double c = std::cos(pi * r) * (odd ? -1 : 1), s = std::sin(pi * r) * (odd ? -1 : 1);
    for (int k = 0; k < 2; ++k) {
      const long double exact = k ? s : c, got = k ? v.y : v.x;
      const float f = std::fabs((float)exact);
      const double half = 0.5 * (std::nextafter(f, 2.f) - f);
      worst = std::fmax(worst, (double)std::fabs(got - exact) - half);
    }
  }
  printf("%a\n", worst);
  return 0;
}
"""


def test_exponential_is_rounded_once(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "t.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")], check=True)
    worst = float.fromhex(subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout)
    print(worst)
    assert worst <= 2.0 ** -35
