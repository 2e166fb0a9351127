"""The aberration path's sums over the volume and the sensor at the sizes where
their kernels' grids change: widths that take 64, 128 or 256 threads per row,
volumes whose voxel count is no multiple of four, a single-voxel window, and
many chunks of the sensor sum; loss and gradient against the FP64 oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

import synth
from oracle import aberration as ab


@pytest.mark.parametrize("shape,window", [((64, 64, 16), (5, 7, 1, 1)), ((64, 128, 16), (3, 1, 33, 21)),
                                          ((384, 64, 32), (100, 2, 77, 55)), ((640, 64, 16), None), ((256, 64, 128), None)])
def test_loss_and_gradient_at_grid_edges(shape, window):
    import paper_2003_08960_gb300 as ss
    nx, ny, nl = shape
    w = synth.workload("custom", nx=nx, ny=ny, nlambda=nl, kind="points", seed=nx + ny)
    rng = np.random.default_rng(nl)
    coeffs = (0.3 * rng.standard_normal(15)).tolist()
    plan = ss.Plan(nx, ny, nl, w.pitch, 0.3, w.lambdas, window=window, flags=ss.SSOCT_FLAG_PUPIL)
    frames = torch.from_numpy(np.ascontiguousarray(w.frames).view(np.int16)).cuda()
    loss, grad, vol = plan.sharpness(frames, coeffs, 0.304)
    ref_loss, ref = ab.sharpness_gradient(w.frames, w.pitch, 0.304, w.lambdas, coeffs, window)
    # the FP32 bounds of the path: 2e-5 for the volume's squares, 1e-4 for the gradient
    assert abs(loss - ref_loss) <= 2e-5 * abs(ref_loss)
    assert np.linalg.norm(grad[1:] - ref[1:]) <= 1e-4 * np.linalg.norm(ref[1:])
    assert abs(grad[0] - ref[0]) <= 1e-4 * np.linalg.norm(ref)
    # the two sums themselves, from the volume the call returned: 48-bit sums
    p = vol.double()
    assert abs(loss + float((p * p).sum() / p.sum() ** 2)) <= 1e-12 * abs(loss)
