"""Non-square frames: the work queue (long enough sweeps), the two passes through
the frame buffer (short sweeps, and rescale ratios whose rows do not fit the
queue's staging), and the aberration path on the queue, from aligned and from
unaligned frames."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

import oracle
import synth

TOL = 1e-5  # relative L2 of the complex volume over the whole plane, the bound of the FP32 path


def _frames(shape, seed):
    nx, ny, nl = shape
    return np.random.default_rng(seed).integers(0, 4096, (nl, ny, nx), dtype=np.uint16)


# (shape, window, last wavelength): the two lengths' splits differ in every pair;
# 1024 x 128 with ratios up to 12 stages 98 rows an item and takes the two passes
@pytest.mark.parametrize("shape,window,last", [
    ((256, 512, 32), (3, 5, 201, 333), 850e-9), ((1024, 64, 64), None, 850e-9), ((384, 768, 16), (100, 700, 33, 68), 850e-9),
    ((640, 1024, 16), (639, 0, 1, 1024), 850e-9), ((512, 384, 16), None, 780e-9), ((64, 256, 16), None, 850e-9),
    ((1024, 128, 32), (11, 13, 97, 101), 9600e-9)])
def test_non_square_frames(shape, window, last):
    import paper_2003_08960_gb300 as ss
    nx, ny, nl = shape
    f = _frames(shape, nx + ny)
    lam = synth.interferograms.sweep_wavelengths(800e-9, last, nl)
    plan = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam, window=window)
    vol, cplx = plan.reconstruct(torch.from_numpy(f.view(np.int16)).cuda(), complex_out=True)
    plan.sync()
    full = oracle.reconstruct(f, 20e-6, 0.3, lam, method="fft")
    x0, y0, wx, wy = window or (0, 0, nx, ny)
    ref = full[:, y0:y0 + wy, x0:x0 + wx]
    rms = float(np.sqrt(np.mean(oracle.intensity(full))))
    err = cplx.cpu().numpy().astype(np.complex128) - ref
    assert np.sqrt(np.mean(oracle.intensity(err))) <= TOL * rms
    e = TOL * rms * np.sqrt(ref.size)
    assert np.all(np.abs(vol.cpu().numpy().astype(np.float64) - oracle.intensity(ref)) <= 2 * e * np.abs(ref) + e * e)


# rows whose second-stage transforms are dealt out over a group's threads: whole rows,
# and windows that begin or end inside a thread's run of outputs
@pytest.mark.parametrize("n", [384, 640, 768])
@pytest.mark.parametrize("axial_first", [False, True])
@pytest.mark.parametrize("crop", [None, (0, 0, 1, 3), (19, 23, 33, 40), (-1, -7, 1, 7)])
def test_uneven_splits_of_square_frames(n, axial_first, crop):
    import paper_2003_08960_gb300 as ss
    nl = 16
    f = _frames((n, n, nl), n)
    lam = synth.interferograms.sweep_wavelengths(800e-9, 850e-9, nl)
    window = crop and (crop[0] % n, crop[1] % n, crop[2], crop[3])
    plan = ss.Plan(n, n, nl, 20e-6, 0.3, lam, window=window, flags=ss.SSOCT_FLAG_AXIAL_FIRST if axial_first else 0)
    vol, cplx = plan.reconstruct(torch.from_numpy(f.view(np.int16)).cuda(), complex_out=True)
    plan.sync()
    full = oracle.reconstruct(f, 20e-6, 0.3, lam, method="fft")
    x0, y0, wx, wy = window or (0, 0, n, n)
    ref = full[:, y0:y0 + wy, x0:x0 + wx]
    rms = float(np.sqrt(np.mean(oracle.intensity(full))))
    err = cplx.cpu().numpy().astype(np.complex128) - ref
    assert np.sqrt(np.mean(oracle.intensity(err))) <= TOL * rms
    e = TOL * rms * np.sqrt(ref.size)
    assert np.all(np.abs(vol.cpu().numpy().astype(np.float64) - oracle.intensity(ref)) <= 2 * e * np.abs(ref) + e * e)


@pytest.mark.parametrize("window", [None, (100, 40, 301, 222)])
def test_aberration_path_from_any_alignment(window):
    import paper_2003_08960_gb300 as ss
    w = synth.workload("custom", nx=512, ny=512, nlambda=32, kind="speckle", seed=4)
    plan = ss.Plan(w.nx, w.ny, w.nlambda, w.pitch, 0.3, w.lambdas, window=window, flags=ss.SSOCT_FLAG_PUPIL)
    flat = torch.empty(w.frames.size + 1, dtype=torch.int16, device="cuda")
    aligned = torch.from_numpy(np.ascontiguousarray(w.frames).view(np.int16)).cuda()
    flat[1:] = aligned.reshape(-1)
    shifted = flat[1:].view(aligned.shape)
    assert aligned.data_ptr() % 16 == 0 and shifted.data_ptr() % 16 != 0
    coeffs = (0.2 * np.random.default_rng(3).standard_normal(15)).tolist()
    l0, g0, v0 = plan.sharpness(aligned, coeffs, 0.303)
    v0 = v0.clone()
    l1, g1, v1 = plan.sharpness(shifted, coeffs, 0.303)   # plain loads instead of bulk copies
    # two FP32 evaluations of the same sums
    assert float((v0.double() - v1.double()).norm()) <= 2e-5 * float(v1.double().norm())
    assert abs(l0 - l1) <= 2e-5 * abs(l1)
    assert np.linalg.norm(g0[1:] - g1[1:]) <= 2e-4 * np.linalg.norm(g1[1:])


# streamed adjoint row pass (aligned frames) against the plain one (any alignment):
# bands that end inside a CTA's share, mixed-radix rows, a band of eight rows, the
# last share shorter
@pytest.mark.parametrize("shape,window", [((256, 256, 128), (30, 7, 101, 200)), ((640, 384, 64), None),
                                          ((1024, 64, 200), (1, 3, 1000, 55)), ((384, 256, 160), None)])
def test_adjoint_rows_streamed_and_plain(shape, window):
    import paper_2003_08960_gb300 as ss
    nx, ny, nl = shape
    lam = synth.interferograms.sweep_wavelengths(800e-9, 850e-9, nl)
    plan = ss.Plan(nx, ny, nl, 20e-6, 0.3, lam, window=window, flags=ss.SSOCT_FLAG_PUPIL)
    aligned = torch.from_numpy(_frames(shape, nx * nl).view(np.int16)).cuda()
    flat = torch.empty(aligned.numel() + 1, dtype=torch.int16, device="cuda")
    flat[1:] = aligned.reshape(-1)
    coeffs = (0.2 * np.random.default_rng(nl).standard_normal(15)).tolist()
    l0, g0, _ = plan.sharpness(aligned, coeffs, 0.301)
    l1, g1, _ = plan.sharpness(flat[1:].view(aligned.shape), coeffs, 0.301)
    # two FP32 evaluations of the same sums
    assert abs(l0 - l1) <= 2e-5 * abs(l1)
    assert np.linalg.norm(g0[1:] - g1[1:]) <= 2e-4 * np.linalg.norm(g1[1:])
    assert abs(g0[0] - g1[0]) <= 2e-4 * np.linalg.norm(g1)
