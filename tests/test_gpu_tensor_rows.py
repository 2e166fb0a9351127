"""Rows of the tensor-core axial kernel: the tensor copy (row pitch a multiple of
16 bytes), clipped at the window's last columns, and the plain stores
of every other volume write the same values, and nothing outside the volume."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


# widths: one half-tile, clipped in its first and second half-tile, an empty last
# half-tile, the whole frame; and widths whose rows are not on 16-byte boundaries
@pytest.mark.parametrize("wx", [4, 16, 20, 36, 48, 64, 1, 15, 33, 62])
@pytest.mark.parametrize("magnitude", [False, True])
def test_copied_and_stored_rows_agree(wx, magnitude):
    import paper_2003_08960_gb300 as ss
    nx = ny = 64
    nl, wy = 256, 5
    lam = np.linspace(800e-9, 850e-9, nl)
    flags = ss.SSOCT_FLAG_TC_AXIAL | (ss.SSOCT_FLAG_MAGNITUDE if magnitude else 0)
    gen = torch.Generator(device="cuda").manual_seed(wx)
    frames = torch.randint(0, 4096, (nl, ny, nx), dtype=torch.int16, device="cuda", generator=gen)
    whole = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam, flags=flags).reconstruct(frames)
    x0, y0 = nx - wx, 3
    plan = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam, window=(x0, y0, wx, wy), flags=flags)
    n = nl * wy * wx
    for shift in (0, 4):
        flat = torch.full((n + 64,), -1.0, device="cuda")
        vol = flat[shift:shift + n].view(nl, wy, wx)
        plan.reconstruct(frames, out=(vol, None))
        plan.sync()
        assert torch.equal(vol, whole[:, y0:y0 + wy, x0:x0 + wx])
        assert bool((flat[:shift] == -1).all()) and bool((flat[shift + n:] == -1).all())
