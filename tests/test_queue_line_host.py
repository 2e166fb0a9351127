"""Where non-square frames and the aberration path change from the two passes to
the work queue: on either side of the line, sizes at which the path taken measured
no slower than the other one (run as host code; whether a plan's staging fits is
asked separately)."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "ssoct_internal.h"
int main() {
  int nx, ny, nl;
  while (scanf("%d %d %d", &nx, &ny, &nl) == 3)
    printf("%d %d\n", (int)ssoct::pair_queue_pays(nx, ny, (long long)nx * ny * nl), (int)ssoct::pupil_queue_pays(nx, (long long)nx * ny * nl));
  return 0;
}
"""

# nx, ny, frames: two passes, queue (us a call)
PAIRS = [((256, 64, 200), 32.9, 43.1), ((256, 64, 512), 85.1, 90.3), ((64, 256, 512), 81.5, 94.3), ((1024, 64, 512), 314.5, 338.6),
         ((512, 64, 256), 88.1, 100.7), ((384, 64, 512), 131.5, 137.0), ((64, 384, 512), 128.0, 131.7), ((64, 1024, 64), 48.5, 56.5),
         ((64, 1024, 200), 147.4, 139.8), ((64, 512, 512), 177.1, 173.6), ((64, 768, 256), 140.7, 133.6), ((768, 64, 256), 137.7, 131.1),
         ((640, 64, 128), 61.5, 63.7), ((640, 64, 256), 115.1, 111.7), ((256, 128, 128), 41.0, 45.1), ((256, 128, 256), 82.0, 75.9),
         ((512, 128, 96), 66.6, 70.8), ((128, 512, 96), 74.9, 69.7), ((512, 256, 32), 38.0, 45.3), ((512, 256, 64), 87.5, 83.2),
         ((1024, 256, 16), 39.9, 45.2), ((256, 1024, 16), 41.8, 43.5), ((1024, 512, 16), 98.1, 76.1), ((384, 128, 96), 50.6, 58.2),
         ((384, 256, 32), 34.0, 35.0), ((384, 256, 64), 68.8, 66.0), ((128, 640, 64), 66.5, 61.8), ((640, 256, 32), 55.3, 54.1),
         ((512, 384, 16), 36.1, 39.1), ((640, 384, 16), 43.7, 41.1), ((640, 384, 160), 386.4, 333.0)]
PUPILS = [((256, 256, 96), 223.2, 238.9), ((256, 256, 128), 266.8, 276.1), ((256, 256, 200), 421.6, 414.1), ((384, 384, 32), 219.5, 235.5),
          ((384, 384, 64), 348.0, 343.4), ((512, 512, 16), 237.5, 240.4), ((512, 512, 64), 484.2, 449.7), ((640, 640, 16), 327.5, 331.1),
          ((768, 768, 16), 426.1, 405.0), ((1024, 1024, 16), 620.7, 580.8)]


@pytest.fixture(scope="module")
def routes(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("line")
    (d / "l.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, str(d / "l.cu"), "-o", str(d / "l")], check=True)
    sizes = [c[0] for c in PAIRS + PUPILS]
    out = subprocess.run([str(d / "l")], input="\n".join("%d %d %d" % s for s in sizes), capture_output=True, text=True, check=True)
    return dict(zip(sizes, (tuple(map(int, line.split())) for line in out.stdout.splitlines())))


@pytest.mark.parametrize("size,two,queue", PAIRS)
def test_non_square_frames_take_the_faster_path(routes, size, two, queue):
    assert routes[size][0] == (queue < two)


@pytest.mark.parametrize("size,two,queue", PUPILS)
def test_aberration_path_takes_the_faster_path(routes, size, two, queue):
    assert routes[size][1] == (queue < two)
