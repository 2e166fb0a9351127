"""Frames of up to 128 x 128 are transformed whole in shared memory and keep no
frames in flight: beside the pushed frames (2 bytes a voxel), the intermediate (8)
and the tables, their workspace holds no more ring than the work queue needs when
a stall is injected (79 frames of 128 x 128, 9.9 MiB)."""

import os

import numpy as np
import pytest

import paper_2003_08960_gb300 as ss

pytestmark = pytest.mark.skipif(not os.path.exists(ss._abi.LIB_PATH), reason="libssoct.so is not built")


@pytest.mark.parametrize("shape", [(64, 64, 512), (128, 64, 256), (64, 128, 512), (128, 128, 128), (128, 128, 256), (128, 128, 512)])
def test_workspace_of_small_frames(shape):
    nx, ny, nl = shape
    st, h = ss.ssoct_create_plan(nx, ny, nl, 20e-6, 0.3, np.linspace(800e-9, 850e-9, nl))
    assert st == ss.SSOCT_OK
    try:
        st, size = ss.ssoct_workspace_size(h)
        assert st == ss.SSOCT_OK
        tables = 16 * nl * (nx + ny) + (1 << 16) + 8 * nx * ny  # taps, the other tables, the running cut
        assert size <= (2 + 8) * nx * ny * nl + tables + 10 * (1 << 20)
    finally:
        ss.ssoct_destroy_plan(h)
