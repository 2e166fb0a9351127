"""Sweep lengths of the streaming axial kernel on their own splits (96, 160, 200)
and in half tiles (512), with windows that leave ragged last units and with
fewer units than SMs; the cuts of sliding gates on the same splits; and the
no-allocation path, whose taps are built on the device."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a GPU")]

import oracle
import synth

TOL = 1e-5  # relative L2 of the complex volume over the whole plane, the bound of the FP32 path


def _plan(shape, window, **kw):
    import paper_2003_08960_gb300 as ss
    nx, ny, nl = shape
    w = synth.workload("custom", nx=nx, ny=ny, nlambda=nl, kind="points", seed=nl + nx)
    frames = torch.from_numpy(np.ascontiguousarray(w.frames).view(np.int16)).cuda()
    return ss, w, frames, ss.Plan(nx, ny, nl, w.pitch, w.z, w.lambdas, window=window, **kw)


SHAPES = [((64, 64, 96), (3, 5, 33, 41)), ((64, 64, 160), (0, 0, 1, 1)), ((128, 64, 200), (17, 1, 97, 63)),
          ((64, 64, 512), (9, 2, 17, 30)), ((64, 64, 512), (9, 2, 49, 2)), ((64, 128, 512), None)]


@pytest.mark.parametrize("shape,window", SHAPES)
def test_streaming_splits_against_the_oracle(shape, window):
    ss, w, frames, plan = _plan(shape, window)
    vol, cplx = plan.reconstruct(frames, complex_out=True)
    plan.sync()
    # every output of the transforms mixes every input, so the rounding error of a
    # voxel goes with the RMS of the whole plane's volume, not with its own size
    full = oracle.reconstruct(w.frames, w.pitch, w.z, w.lambdas, method="fft")
    x0, y0, wx, wy = window or (0, 0, w.nx, w.ny)
    ref = full[:, y0:y0 + wy, x0:x0 + wx]
    rms = float(np.sqrt(np.mean(oracle.intensity(full))))
    err = cplx.cpu().numpy().astype(np.complex128) - ref
    assert np.sqrt(np.mean(oracle.intensity(err))) <= TOL * rms
    # |V|^2 = (|V| + e)^2: twice the error times |V|, plus its square
    p_err = np.abs(vol.cpu().numpy().astype(np.float64) - oracle.intensity(ref))
    e = TOL * rms * np.sqrt(ref.size)  # no voxel's error exceeds the whole window's
    assert np.all(p_err <= 2 * e * np.abs(ref) + e * e)


@pytest.mark.parametrize("shape,window", SHAPES)
def test_sliding_lines_equal_the_volume(shape, window):
    ss, w, frames, plan = _plan(shape, window)
    other = ss.Plan(w.nx, w.ny, w.nlambda, w.pitch, w.z, w.lambdas, window=window)
    nl, wy, wx = plan.volume_shape()
    for p in (plan, other):
        p.push(frames)
    for new in (0, 1, 9, 17):  # slots read ahead in eights by the running xy cut
        if new:
            for p in (plan, other):
                p.push(frames[5:5 + new] if new + 5 <= nl else frames[:new])
        vol = plan.reconstruct_sliding()
        xy, xz, yz = other.sliding_cuts(wx - 1, wy // 2, nl // 3)
        torch.cuda.synchronize()
        assert torch.equal(xz, vol[:, wy // 2, :]) and torch.equal(yz, vol[:, :, wx - 1])
        # one bin summed frame by frame against the FFT: FP32 rounding of nl terms
        assert float((xy - vol[nl // 3]).norm()) <= 1e-4 * float(vol[nl // 3].norm()) + 1e-6 * float(vol.amax())


@pytest.mark.parametrize("shape,window", [((64, 128, 16), None), ((128, 64, 200), (3, 2, 101, 57)),
                                          ((256, 256, 32), (100, 90, 31, 77)), ((64, 64, 512), None)])
def test_noalloc_tables_built_on_the_device(shape, window):
    ss, w, frames, plan = _plan(shape, window)
    ref = plan.reconstruct(frames)
    st, h = ss.ssoct_create_plan(w.nx, w.ny, w.nlambda, w.pitch, w.z, w.lambdas, window)
    assert st == ss.SSOCT_OK
    try:
        vol = torch.full_like(ref, float("nan"))
        stream = torch.cuda.current_stream().cuda_stream
        assert ss.ssoct_reconstruct_frames_noalloc(h, frames.data_ptr(), vol.data_ptr(), 0, stream) == ss.SSOCT_OK
        assert ss.ssoct_sync(h, stream) == ss.SSOCT_OK
        # the taps may differ from the host's in the last bit of a float
        assert float((vol.double() - ref.double()).norm()) <= 1e-6 * float(ref.double().norm())
    finally:
        ss.ssoct_destroy_plan(h)
