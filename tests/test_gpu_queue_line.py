"""Non-square frames just on either side of the line between the two passes and the
work queue, against the FP64 oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

import oracle
import synth

TOL = 1e-5  # relative L2 of the complex volume over the whole plane, the bound of the FP32 path


@pytest.mark.parametrize("shape,window", [((256, 512, 32), None), ((256, 512, 64), (3, 5, 201, 333)), ((64, 512, 256), (1, 100, 63, 311)),
                                          ((768, 64, 128), (0, 3, 700, 1)), ((1024, 64, 128), None), ((512, 384, 32), (30, 0, 97, 384))])
def test_both_sides_of_the_line(shape, window):
    import paper_2003_08960_gb300 as ss
    nx, ny, nl = shape
    f = np.random.default_rng(nx + ny).integers(0, 4096, (nl, ny, nx), dtype=np.uint16)
    lam = synth.interferograms.sweep_wavelengths(800e-9, 850e-9, nl)
    plan = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam, window=window)
    _, cplx = plan.reconstruct(torch.from_numpy(f.view(np.int16)).cuda(), complex_out=True)
    plan.sync()
    full = oracle.reconstruct(f, 20e-6, 0.3, lam, method="fft")
    x0, y0, wx, wy = window or (0, 0, nx, ny)
    err = cplx.cpu().numpy().astype(np.complex128) - full[:, y0:y0 + wy, x0:x0 + wx]
    assert np.sqrt(np.mean(oracle.intensity(err))) <= TOL * np.sqrt(np.mean(oracle.intensity(full)))
