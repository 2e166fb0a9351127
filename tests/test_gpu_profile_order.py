"""Stage times of plans whose whole volumes run axial-first while their sliding
gates keep the paper's order: every call's intervals go to the stage that they
measured, whichever order the plan has when the times are read."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def _plan(ss, tmp_path, frames, lam):
    """A plan tuned to the axial-first order (through its cache entry)."""
    nl, ny, nx = frames.shape
    cache = tmp_path / "tune.json"
    ss.Plan(nx, ny, nl, 20e-6, 0.3, lam).autotune(frames, cache)
    cache.write_text(cache.read_text().replace('"axial_first": 0', '"axial_first": 1').replace('"tc_axial": 1', '"tc_axial": 0'))
    plan = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam)
    assert plan.autotune(frames, cache)["axial_first"] == 1
    return plan


def test_sliding_gates_of_an_axial_first_plan(tmp_path):
    import paper_2003_08960_gb300 as ss
    nx, nl = 512, 128
    lam = np.linspace(800e-9, 850e-9, nl)
    gen = torch.Generator(device="cuda").manual_seed(1)
    frames = torch.randint(0, 4096, (nl, nx, nx), dtype=torch.int16, device="cuda", generator=gen)
    plan = _plan(ss, tmp_path, frames, lam)
    plan.push(frames)
    out = plan.empty_volume()
    for _ in range(3):
        plan.reconstruct_sliding(out=out)
    plan.sync()

    def profile(calls):
        assert ss.ssoct_profile(plan.handle, True) == 0
        for c in calls:
            c()
        st, lat, ax, n = ss.ssoct_profile_read(plan.handle)
        assert st == 0 and n == len(calls)
        return lat, ax

    gate = lambda: plan.reconstruct_sliding(out=out)  # no new frames: its lateral interval is empty
    volume = lambda: plan.reconstruct(frames, out=out)
    lat, ax = profile([gate] * 3)
    # the axial kernel reads 268 MB and writes 134 MB a call: over 40 us at the memory's
    # nominal 7.9 TB/s; two events recorded one after the other are a few us apart
    assert ax > 3 * 0.040 and lat < ax / 3, (lat, ax)
    # a mix of both kinds: the volume's lateral pass is the longer of its two stages, and
    # the gates' empty lateral intervals leave it so
    volume()
    vlat, vax = profile([volume] * 3)
    gate()
    mlat, max_ = profile([volume, gate, gate, gate])
    assert vlat > vax
    assert max_ > 3 * 0.040 and mlat < vlat
