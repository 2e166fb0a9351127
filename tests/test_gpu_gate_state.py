"""The running xy cut that a plan keeps between sliding gates does not outlive the
gate it belongs to: a dropped sequence and a new workspace start it over."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

NX, NL = 64, 16
LAM = np.linspace(800e-9, 850e-9, NL)


def _frames(seed, n=NL):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, 4096, (n, NX, NX), dtype=torch.int16, device="cuda", generator=gen)


def _plan(ss):
    return ss.Plan(NX, NX, NL, 20e-6, 0.3, LAM)


def _cuts_of(ss, frames):
    plan = _plan(ss)
    plan.push(frames)
    cuts = plan.sliding_cuts(5, 6, 3)
    plan.sync()
    return cuts


@pytest.mark.parametrize("restart", ["drop", "workspace"])
@pytest.mark.parametrize("volume_first", [True, False])
def test_running_cut_starts_over(restart, volume_first):
    import paper_2003_08960_gb300 as ss
    old, new = _frames(1), _frames(2)
    plan = _plan(ss)
    plan.push(old, first_seq=0)
    plan.sliding_cuts(5, 6, 3)
    plan.sync()
    keep = None
    if restart == "drop":
        assert plan.push(new, first_seq=1000) == ss.SSOCT_EDROPPED
    else:
        keep = torch.zeros(plan.info.workspace_bytes, dtype=torch.uint8, device="cuda")
        assert ss.ssoct_set_workspace(plan.handle, keep.data_ptr(), keep.numel()) == ss.SSOCT_OK
        plan.push(new, first_seq=0)
    if volume_first:
        plan.reconstruct_sliding()
    cuts = plan.sliding_cuts(5, 6, 3)
    plan.sync()
    for a, b in zip(cuts, _cuts_of(ss, new)):
        assert torch.equal(a, b)
