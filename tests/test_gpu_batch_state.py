"""What a batch's graph launch does to the state its plans keep."""

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


def test_batch_relaunch_between_gates():
    import paper_2003_08960_gb300 as ss
    stream, other = _frames(3, 2 * NL), _frames(4)
    plan, ref = _plan(ss), _plan(ss)
    vol = plan.empty_volume()[0]
    batch = ss.Batch([plan])
    for p in (plan, ref):
        p.push(stream[:NL])
    batch.run([other], [vol])
    batch.sync()
    plan.reconstruct_sliding()
    ref.reconstruct_sliding()
    for p in (plan, ref):
        p.push(stream[NL:NL + 3])
    batch.run([other], [vol])  # the same pointers: the captured graph again
    batch.sync()
    assert batch.captures == 1
    a, b = plan.reconstruct_sliding(), ref.reconstruct_sliding()
    torch.cuda.synchronize()
    assert torch.equal(a, b)


def test_batch_follows_a_new_workspace():
    import paper_2003_08960_gb300 as ss
    frames = _frames(5)
    plan = _plan(ss)
    vol = plan.empty_volume()[0]
    batch = ss.Batch([plan])
    batch.run([frames], [vol])
    batch.sync()
    first = vol.clone()
    moved = torch.zeros(plan.info.workspace_bytes, dtype=torch.uint8, device="cuda")
    assert ss.ssoct_set_workspace(plan.handle, moved.data_ptr(), moved.numel()) == ss.SSOCT_OK
    batch.run([frames], [vol])
    batch.sync()
    assert batch.captures == 2 and torch.equal(vol, first)
    batch.run([frames], [vol])
    batch.sync()
    assert batch.captures == 2
