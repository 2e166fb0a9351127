"""The order that whole volumes of plans without a flag run in: axial-first for the
whole plane (the volume of a plan made with that flag, bit for bit), the paper's
for any cropped window (the sliding gate's volume, bit for bit), with and without
the complex volume."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("window", [None, (0, 0, 256, 256), (0, 0, 256, 255), (0, 0, 255, 256), (3, 5, 250, 241)])
@pytest.mark.parametrize("complex_out", [False, True])
def test_order_of_default_volumes(window, complex_out):
    import paper_2003_08960_gb300 as ss
    nx, nl = 256, 64
    lam = np.linspace(800e-9, 850e-9, nl)
    gen = torch.Generator(device="cuda").manual_seed(2)
    frames = torch.randint(0, 4096, (nl, nx, nx), dtype=torch.int16, device="cuda", generator=gen)
    plan = ss.Plan(nx, nx, nl, 20e-6, 0.3, lam, window=window)
    got = plan.reconstruct(frames, complex_out=complex_out)
    if window is None or window[2:] == (nx, nx):
        ref = ss.Plan(nx, nx, nl, 20e-6, 0.3, lam, window=window, flags=ss.SSOCT_FLAG_AXIAL_FIRST).reconstruct(
            frames, complex_out=complex_out)
    else:
        plan.push(frames)
        ref = plan.reconstruct_sliding(complex_out=complex_out)
    torch.cuda.synchronize()
    for a, b in zip(got if complex_out else (got,), ref if complex_out else (ref,)):
        assert torch.equal(a, b)
