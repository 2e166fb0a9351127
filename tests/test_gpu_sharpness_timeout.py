"""A wait that runs out inside the aberration path is the call's own status: no
loss and gradient of an incomplete pass are handed back as good ones, no earlier
failure is lost, and the next call is exact again."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]


def test_a_stalled_queue_is_reported_by_the_call():
    import paper_2003_08960_gb300 as ss
    nx, nl = 512, 32  # long enough for the work queue
    lam = np.linspace(800e-9, 850e-9, nl)
    gen = torch.Generator(device="cuda").manual_seed(9)
    frames = torch.randint(0, 4096, (nl, nx, nx), dtype=torch.int16, device="cuda", generator=gen)
    plan = ss.Plan(nx, nx, nl, 20e-6, 0.3, lam, flags=ss.SSOCT_FLAG_PUPIL)
    coeffs = [0.1 * j for j in range(15)]
    loss, grad, vol = plan.sharpness(frames, coeffs, 0.304)
    stream = torch.cuda.current_stream().cuda_stream
    assert ss.ssoct_inject_stall(plan.handle, 1, 50_000_000) == ss.SSOCT_OK
    out = torch.empty_like(vol)
    st, res = ss.ssoct_sharpness(plan.handle, frames.data_ptr(), out.data_ptr(), stream)
    assert st == ss.SSOCT_ETIMEOUT and not res.any()  # the output is untouched
    assert "gave up" in ss.ssoct_last_error(plan.handle)
    assert ss.ssoct_inject_stall(plan.handle, 0, 0) == ss.SSOCT_OK
    assert ss.ssoct_sync(plan.handle, stream) == ss.SSOCT_OK  # reported once
    loss2, grad2, vol2 = plan.sharpness(frames, coeffs, 0.304)
    assert torch.equal(vol2, vol)
    # the FP64 block sums are atomics, so two calls agree to rounding
    assert abs(loss2 - loss) <= 1e-12 * abs(loss) and np.allclose(grad2, grad, rtol=0, atol=1e-9 * np.linalg.norm(grad))


def test_an_earlier_failure_is_left_to_sync():
    import paper_2003_08960_gb300 as ss
    nx, nl = 512, 32
    lam = np.linspace(800e-9, 850e-9, nl)
    frames = torch.zeros((nl, nx, nx), dtype=torch.int16, device="cuda")
    frames[:, 100:200, 50:300] = 1000
    plan = ss.Plan(nx, nx, nl, 20e-6, 0.3, lam, flags=ss.SSOCT_FLAG_PUPIL)
    stream = torch.cuda.current_stream().cuda_stream
    vol = plan.empty_volume()[0]
    assert ss.ssoct_inject_stall(plan.handle, 1, 50_000_000) == ss.SSOCT_OK
    plan.reconstruct(frames, out=(vol, None))
    assert ss.ssoct_inject_stall(plan.handle, 0, 0) == ss.SSOCT_OK
    plan.sharpness(frames, [], 0.3, out=vol)  # a good call of its own
    assert ss.ssoct_sync(plan.handle, stream) == ss.SSOCT_ETIMEOUT
    assert ss.ssoct_sync(plan.handle, stream) == ss.SSOCT_OK
