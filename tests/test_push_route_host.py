"""Which pushed frames the copy kernel takes: memory of the plan's own device, on a
16-byte boundary, with that device current.  Frames of another GPU, managed or
host memory handed in as device frames, and pointers CUDA does not know are
copied by the runtime, which reaches memory that a kernel here may not."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_08960_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "ssoct_internal.h"
int main() {
  const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged};
  for (cudaMemoryType t : types)
    for (int device = 0; device < 2; ++device)
      for (int current = 0; current < 2; ++current)
        for (int shift = 0; shift < 32; shift += 2) {
          cudaPointerAttributes a = {};
          a.type = t;
          a.device = device;
          const bool k = ssoct::push_by_kernel(a, 1, current, (const char*)4096 + shift);
          const bool want = t == cudaMemoryTypeDevice && device == 1 && current == 1 && shift % 16 == 0;
          if (k != want) { printf("type %d device %d current %d shift %d: %d\n", (int)t, device, current, shift, k); return 1; }
        }
  return 0;
}
"""


def test_copy_kernel_takes_the_plans_own_memory_only(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    (tmp_path / "p.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, str(tmp_path / "p.cu"), "-o", str(tmp_path / "p")], check=True)
    r = subprocess.run([str(tmp_path / "p")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
