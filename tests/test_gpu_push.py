"""Frames pushed from device memory: the copy kernel (16-byte aligned sources, a
last block that is not full, a run that wraps the ring) and the plain copy of
frames at any other address fill the ring with the same frames."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


@pytest.mark.parametrize("shape", [(64, 64, 16), (128, 64, 16), (640, 384, 16)])
@pytest.mark.parametrize("shift", [0, 1, 8])
def test_push_from_device_memory(shape, shift):
    import paper_2003_08960_gb300 as ss
    nx, ny, nl = shape
    lam = np.linspace(800e-9, 850e-9, nl)
    plan = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam)
    gen = torch.Generator(device="cuda").manual_seed(nx + shift)
    frames = torch.randint(0, 4096, (nl, ny, nx), dtype=torch.int16, device="cuda", generator=gen)
    ref = plan.reconstruct(frames)
    flat = torch.empty(frames.numel() + shift, dtype=torch.int16, device="cuda")
    flat[shift:] = frames.reshape(-1)
    moved = flat[shift:].view(frames.shape)
    plan.push(moved[:5])          # stray frames, so that the sweep wraps the ring
    plan.push(moved[:7])
    plan.push(moved[7:])
    vol = plan.reconstruct_ring()
    torch.cuda.synchronize()
    assert torch.equal(vol, ref)
