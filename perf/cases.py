"""Workloads of the reconstruction library for timing: what a program that links
libssoct has it do, through the public calls of ``paper_2003_08960_gb300``.

A case is a dict of plain values.  ``prepare`` builds what such a program holds
before the call (plan, workspace, frames on the device, output buffers), ``run``
makes one call sequence on it, ``work`` counts the bytes and operations of one
``run`` that no implementation can avoid, and ``exact`` evaluates Eq. 5 - Eq. 7
(and the sharpness gradient) in float64 with plain torch.

Fields: op (volume, noalloc, sliding, sliding_cuts, sharpness, batch); nx, ny, nl
(frame and sweep); x0, y0, wx, wy (window); order (paper, axial_first,
tensor_core); complex (also the complex volume); magnitude (|V| instead of
|V|^2); cuts (the three cuts after the volume); new (frames pushed per gate);
volumes (sizes of a batch); scene (points, speckle).
"""

import math

import numpy as np
import torch

import paper_2003_08960_gb300 as ss

# Sweep 800 -> 850 nm linear in wavenumber, 20 um pixels, object at 0.3 m, fringes
# of a quarter of the frame: the optics of the repository's tests and benchmark.
LAMBDA_START, LAMBDA_END, PITCH, Z = 800e-9, 850e-9, 20e-6, 0.3

FRAMES_1D = (64, 128, 256, 384, 512, 640, 768, 1024)
SWEEPS = (16, 32, 64, 96, 128, 160, 200, 256, 512)
VOXELS_MOST = 1024 * 1024 * 256

# The eight uneven volumes of the benchmark's batch.
BATCH = "256x256x64,384x384x96,512x512x128,512x512x128,640x640x160,768x768x200,1024x1024x256,1024x1024x256"


def _case(op, nx, ny, nl, window=None, order="paper", **more):
    x0, y0, wx, wy = window or (0, 0, nx, ny)
    return dict(op=op, nx=nx, ny=ny, nl=nl, x0=x0, y0=y0, wx=wx, wy=wy, order=order,
                **{"complex": False, "magnitude": False, "cuts": False, "new": 0, "volumes": "",
                   "scene": "points", **more})


def listed():
    return [
        # A region of interest small enough that launches and latency are all of it
        # (alignment loops, the size of the smoke test); ragged, with phase.
        dict(_case("volume", 64, 64, 32, (36, 40, 23, 17), complex=True), name="tiny_64x64x32_window"),
        # Acquisition code that may not allocate device memory; the largest sizes
        # its fixed scratch holds are about these.
        dict(_case("noalloc", 256, 256, 64), name="noalloc_256x256x64"),
        # Off-axis holography as it is used: one window of the hologram plane (odd
        # offsets), phase-resolved, mixed-radix frame.
        dict(_case("volume", 640, 640, 160, (100, 60, 400, 300), complex=True), name="window_640x640x160_complex"),
        # A camera that is not square: the two-pass lateral path.
        dict(_case("volume", 640, 384, 160), name="two_pass_640x384x160"),
        # The longest sweep (deep imaging range) on a small frame.
        dict(_case("volume", 256, 256, 512), name="long_sweep_256x256x512"),
        # The paper's headline volume with a plan as created, and its display cuts.
        dict(_case("volume", 1024, 1024, 256, cuts=True), name="paper_1024x1024x256"),
        # The same volume in the order that the autotuner chooses for it.
        dict(_case("volume", 1024, 1024, 256, order="axial_first", cuts=True), name="axial_first_1024x1024x256"),
        # The tensor-core option of Eq. 7.
        dict(_case("volume", 512, 512, 256, order="tensor_core"), name="tensor_core_512x512x256"),
        # The paper's acquisition pattern, 13 new frames per rendered volume.
        dict(_case("sliding", 1024, 1024, 256, new=13), name="sliding_1024x1024x256"),
        # The same for a live display: only the three cuts of each gate.
        dict(_case("sliding_cuts", 1024, 1024, 256, new=13), name="sliding_cuts_1024x1024x256"),
        # One step of aberration correction: loss, gradient and volume.
        dict(_case("sharpness", 512, 512, 128, scene="speckle"), name="sharpness_512x512x128"),
        # A queue of uneven volumes as one graph launch, in the autotuner's order.
        dict(_case("batch", 0, 0, 0, order="axial_first", volumes=BATCH), name="batch_8_volumes"),
    ]


def _persistent(nx, ny):
    return nx == ny or (nx, ny) in ((128, 64), (64, 128))


def draw(rng):
    op = rng.choice(("volume", "volume", "volume", "volume", "noalloc", "sliding", "sliding_cuts", "sharpness", "batch"))
    scene = rng.choice(("points", "speckle")) if op == "sharpness" else "points"
    if op == "batch":
        sizes, total = [], 0
        for _ in range(rng.randint(2, 6)):
            n, nl = rng.choice(FRAMES_1D), rng.choice((64, 96, 128, 160, 200, 256))
            if total + n * n * nl <= 2 * VOXELS_MOST:
                sizes.append("%dx%dx%d" % (n, n, nl))
                total += n * n * nl
        return _case(op, 0, 0, 0, order=rng.choice(("paper", "axial_first")), volumes=",".join(sizes or ["64x64x64"]))
    while True:
        nx = rng.choice(FRAMES_1D)
        ny = nx if op not in ("volume", "sharpness") or rng.random() < 0.7 else rng.choice(FRAMES_1D)
        order = rng.choice(("paper", "paper", "axial_first", "tensor_core")) if op == "volume" else "paper"
        nl = 256 if order == "tensor_core" else rng.choice(SWEEPS)
        if order == "axial_first" and not _persistent(nx, ny):
            continue
        if op == "noalloc" and (nx > 256 or nx * ny * nl > 256 * 256 * 64):
            continue  # beyond the fixed scratch of that call
        if nx * ny * nl <= (VOXELS_MOST if op != "sharpness" else VOXELS_MOST // 4):
            break
    window = None
    if rng.random() < 0.5:
        wx, wy = rng.randint(nx // 4, nx), rng.randint(ny // 4, ny)
        window = (rng.randint(0, nx - wx), rng.randint(0, ny - wy), wx, wy)
    more = {}
    if op in ("volume", "noalloc"):
        more = dict(complex=rng.random() < 0.4, cuts=op == "volume" and rng.random() < 0.5)
    if op != "sharpness":
        more["magnitude"] = rng.random() < 0.2
    if op in ("sliding", "sliding_cuts"):
        more["new"] = max(1, min(nl, int(round(math.exp(rng.uniform(0.0, math.log(nl)))))))
    return _case(op, nx, ny, nl, window, order, scene=scene, **more)


# ------------------------------------------------------------------ inputs

def _wavelengths(nl):
    ka, kb = 2.0 * np.pi / LAMBDA_START, 2.0 * np.pi / LAMBDA_END
    return 2.0 * np.pi / (ka + np.arange(nl, dtype=np.float64) * (kb - ka) / (nl - 1))


def _scene(kind, gen):
    """Scatterers (X, Y, depth, amplitude): five points, or fifty over a diffuse layer."""
    fov = LAMBDA_START * Z / PITCH

    def uniform(n, lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)

    n = 5 if kind == "points" else 50
    x, y, depth = uniform(n, -fov / 8, fov / 8), uniform(n, -fov / 8, fov / 8), uniform(n, 0.0, 0.5e-3)
    amp = torch.polar(torch.exp(uniform(n, math.log(1e-3), 0.0)) / n, uniform(n, 0.0, 2 * math.pi))
    if kind == "speckle":
        m = 1024
        d = (torch.arange(64, device="cuda", dtype=torch.float64) + 0.5).repeat_interleave(16) * (1.2e-3 / 64)
        re = torch.randn(m, 2, generator=gen, device="cuda", dtype=torch.float64)
        sigma = 0.02 * torch.exp(-d / 0.6e-3) / math.sqrt(2.0)
        x = torch.cat([x, uniform(m, -fov / 8, fov / 8)])
        y = torch.cat([y, uniform(m, -fov / 8, fov / 8)])
        depth = torch.cat([depth, d])
        amp = torch.cat([amp, torch.complex(sigma * re[:, 0], sigma * re[:, 1])])
    return x, y, depth, amp


def _frames(nx, ny, nl, kind, gen):
    """uint16 interferograms (as int16 bits) |E + E_LO|^2 in camera counts: 12 bits with
    read noise for points, shot noise around 2000 counts for speckle."""
    x, y, depth, amp = _scene(kind, gen)
    xs = (torch.arange(nx, device="cuda", dtype=torch.float64) - nx / 2) * PITCH
    ys = (torch.arange(ny, device="cuda", dtype=torch.float64) - ny / 2) * PITCH
    sx, sy = LAMBDA_START * (nx / 4) / (nx * PITCH), LAMBDA_START * (ny / 4) / (ny * PITCH)
    k_all = torch.from_numpy(2.0 * np.pi / _wavelengths(nl)).cuda()
    out = torch.empty((nl, ny, nx), device="cuda", dtype=torch.int16)
    qx = (xs[None, :] - x[:, None]) ** 2 / (2 * Z)                       # [S][nx]
    qy = (ys[:, None] - y[None, :]) ** 2 / (2 * Z)                       # [ny][S]
    step = 16
    for t in range(0, nl, step):
        k = k_all[t:t + step, None, None]
        one = torch.ones((), device="cuda", dtype=torch.float64)
        u = torch.polar(one, k * qx + 2.0 * k * depth[:, None]) * amp[:, None]   # [b][S][nx]
        v = torch.polar(one, k * qy)                                             # [b][ny][S]
        lo_x, lo_y = torch.polar(one, k * sx * xs[None, :]), torch.polar(one, k * sy * ys[:, None])
        u = torch.cat([u, lo_x], dim=1).to(torch.complex64)
        v = torch.cat([v, lo_y], dim=2).to(torch.complex64)
        e = torch.bmm(v, u)
        c = e.real * e.real + e.imag * e.imag
        noise = torch.randn(c.shape, generator=gen, device="cuda")
        if kind == "points":
            c = (c.mul_(1000.0) + noise.mul_(2.0)).round_().clamp_(0, 4095)
        else:
            c = c.mul_(2000.0)
            c = (c + noise.mul_(c.sqrt())).round_().clamp_(0, 32767)
        out[t:t + step] = c.to(torch.int16)
    return out


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _flags(case):
    return ({"paper": 0, "axial_first": ss.SSOCT_FLAG_AXIAL_FIRST, "tensor_core": ss.SSOCT_FLAG_TC_AXIAL}[case["order"]]
            | (ss.SSOCT_FLAG_MAGNITUDE if case["magnitude"] else 0)
            | (ss.SSOCT_FLAG_PUPIL if case["op"] == "sharpness" else 0))


def _window(case):
    return case["x0"], case["y0"], case["wx"], case["wy"]


def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["volumes"].split(",")]


def _position(case):
    """Where the cuts are taken: off the middle of the window, at an odd place."""
    return (case["wx"] * 5) // 8, (case["wy"] * 3) // 8, (case["nl"] * 3) // 16


def _stream(case, seed):
    """Frames of a sliding acquisition: two sweeps of different scenes, repeated (the
    first frames again at the end, so that every push is one contiguous run)."""
    gen = _generator(seed)
    two = torch.cat([_frames(case["nx"], case["ny"], case["nl"], case["scene"], gen) for _ in range(2)])
    return torch.cat([two, two[:case["new"]]])


def _pupil(seed):
    rng = np.random.default_rng(seed)
    return (0.5 * rng.standard_normal(15)).tolist(), Z + 0.005 * float(rng.uniform(-1.0, 1.0))


# ------------------------------------------------------------------ the calls

class _Handle:
    """A plan of the C interface that has no workspace (released with the state)."""

    def __init__(self, case):
        st, self.h = ss.ssoct_create_plan(case["nx"], case["ny"], case["nl"], PITCH, Z, _wavelengths(case["nl"]),
                                          _window(case), _flags(case))
        if st != ss.SSOCT_OK:
            raise ss.SsoctError(st, "create_plan")

    def __del__(self):
        ss.ssoct_destroy_plan(self.h)


def prepare(case, seed):
    s = {"case": case}
    op, nl = case["op"], case["nl"]
    if op == "batch":
        gen = _generator(seed)
        sizes = _sizes(case)
        s["frames"] = [_frames(nx, ny, n, case["scene"], gen) for nx, ny, n in sizes]
        s["plans"] = [ss.Plan(nx, ny, n, PITCH, Z, _wavelengths(n), flags=_flags(case)) for nx, ny, n in sizes]
        s["vols"] = [p.empty_volume()[0] for p in s["plans"]]
        s["batch"] = ss.Batch(s["plans"])
        return s
    shape = (nl, case["wy"], case["wx"])
    if op == "noalloc":
        s["frames"] = _frames(case["nx"], case["ny"], nl, case["scene"], _generator(seed))
        s["handle"] = _Handle(case)
        s["vol"] = torch.empty(shape, device="cuda", dtype=torch.float32)
        s["cplx"] = torch.empty(shape, device="cuda", dtype=torch.complex64) if case["complex"] else None
        return s
    s["plan"] = ss.Plan(case["nx"], case["ny"], nl, PITCH, Z, _wavelengths(nl), window=_window(case), flags=_flags(case))
    s["out"] = s["plan"].empty_volume(case["complex"]) if op != "sliding_cuts" else None
    if op in ("sliding", "sliding_cuts"):
        # the acquisition is running: a whole sweep has been pushed and rendered
        s["stream"] = _stream(case, seed)
        s["plan"].push(s["stream"][:nl])
        s["pos"] = nl
        if op == "sliding":
            s["plan"].reconstruct_sliding(out=s["out"])
        else:
            s["plan"].sliding_cuts(*_position(case))
        return s
    s["frames"] = _frames(case["nx"], case["ny"], nl, case["scene"], _generator(seed))
    if op == "sharpness":
        s["coeffs"], s["z"] = _pupil(seed)
    return s


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "volume":
        plan = s["plan"]
        plan.reconstruct(s["frames"], out=s["out"])
        outs = [v for v in s["out"] if v is not None]
        return outs + list(plan.cuts(s["out"][0], *_position(case))) if case["cuts"] else outs
    if op == "noalloc":
        st = ss.ssoct_reconstruct_frames_noalloc(s["handle"].h, s["frames"].data_ptr(), s["vol"].data_ptr(),
                                                 s["cplx"].data_ptr() if s["cplx"] is not None else 0,
                                                 torch.cuda.current_stream().cuda_stream)
        if st != ss.SSOCT_OK:
            raise ss.SsoctError(st, ss.ssoct_last_error(s["handle"].h))
        return [v for v in (s["vol"], s["cplx"]) if v is not None]
    if op == "batch":
        s["batch"].run(s["frames"], s["vols"])
        return s["vols"]
    if op == "sharpness":
        # a descent loop keeps its parameters, and so the gradient, in float32
        loss, grad, vol = s["plan"].sharpness(s["frames"], s["coeffs"], s["z"], out=s["out"][0])
        return [loss, float(grad[0]), torch.from_numpy(grad[1:]).float(), vol]
    # sliding gates: the next frames of the stream, then the gate that ends with them
    plan, nl, pos = s["plan"], case["nl"], s["pos"]
    plan.push(s["stream"][pos:pos + case["new"]])
    s["pos"] = (pos + case["new"]) % (2 * nl)
    if op == "sliding":
        plan.reconstruct_sliding(out=s["out"])
        return s["out"][0]
    return list(plan.sliding_cuts(*_position(case)))


def _volume_work(nx, ny, nl, wx, wy, per_voxel):
    return {"bytes": 2.0 * nx * ny * nl + per_voxel * wx * wy * nl,
            "flops": 5.0 * nx * ny * nl * math.log2(nx * ny) + 5.0 * wx * wy * nl * math.log2(nl)}


def work(case):
    """Frames read once, results written once; 5 N log2 N operations per transform."""
    nx, ny, nl, wx, wy, op = case["nx"], case["ny"], case["nl"], case["wx"], case["wy"], case["op"]
    if op == "batch":
        each = [_volume_work(x, y, n, x, y, 4.0) for x, y, n in _sizes(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    cuts = 4.0 * (wx * wy + nl * wx + nl * wy)
    if op in ("volume", "noalloc"):
        w = _volume_work(nx, ny, nl, wx, wy, 12.0 if case["complex"] else 4.0)
        if case["cuts"]:
            w["bytes"] += 2 * cuts
        return w
    if op == "sharpness":
        # forward and adjoint transforms; frames are used by both
        w = _volume_work(nx, ny, nl, wx, wy, 4.0)
        return {"bytes": w["bytes"], "flops": 2 * w["flops"]}
    # sliding: the new frames' holograms, then the whole gate over its window (the
    # other holograms of the gate are read) or one bin of it and two lines
    new = 2.0 * nx * ny * case["new"]
    lateral = 5.0 * nx * ny * case["new"] * math.log2(nx * ny)
    if op == "sliding":
        return {"bytes": new + 12.0 * wx * wy * nl, "flops": lateral + 5.0 * wx * wy * nl * math.log2(nl)}
    return {"bytes": new + 16.0 * wx * wy * case["new"] + 8.0 * nl * (wx + wy) + cuts,
            "flops": lateral + 16.0 * wx * wy * case["new"] + 5.0 * (wx + wy) * nl * math.log2(nl)}


# ------------------------------------------------------------------ float64 values

def _taps(n, ratio):
    """Eq. 5 along one axis: the two source pixels of each output pixel and their weights
    (0 outside the frame), origin at pixel n / 2."""
    c = n / 2.0
    u = c + (torch.arange(n, device="cuda", dtype=torch.float64) - c) * ratio
    i0 = torch.floor(u)
    a = u - i0
    i0 = i0.long()
    w0 = torch.where((i0 >= 0) & (i0 < n), 1.0 - a, torch.zeros_like(a))
    w1 = torch.where((i0 >= -1) & (i0 < n - 1), a, torch.zeros_like(a))
    return i0.clamp(0, n - 1), (i0 + 1).clamp(0, n - 1), w0, w1


def _rescaled(frames, nl):
    """Eq. 5 of every frame, float64 [nl][ny][nx]."""
    lam = _wavelengths(nl)
    out = torch.empty(frames.shape, device="cuda", dtype=torch.float64)
    for t in range(nl):
        f = frames[t].double()
        ratio = lam[t] / lam[0]
        a, b, wa, wb = _taps(f.shape[1], ratio)
        f = f[:, a] * wa + f[:, b] * wb
        a, b, wa, wb = _taps(f.shape[0], ratio)
        out[t] = f[a] * wa[:, None] + f[b] * wb[:, None]
    return out


def _chirp(n, d, scale):
    """exp(-i pi scale (d (k - n/2))^2), k = 0 .. n-1."""
    k = torch.arange(n, device="cuda", dtype=torch.float64) - n / 2.0
    return torch.polar(torch.ones_like(k), -math.pi * scale * (d * k) ** 2)


def _holograms(u, case, screen):
    """Eq. 6 without prefactor and output chirp: the centred DFT (+) of screen x u over
    the window's pixels, complex128 [nl][wy][wx]."""
    x0, y0, wx, wy = _window(case)
    nl, ny, nx = u.shape
    out = torch.empty((nl, wy, wx), device="cuda", dtype=torch.complex128)
    for t in range(nl):
        h = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(u[t] * screen)))
        out[t] = h[y0:y0 + wy, x0:x0 + wx] * (nx * ny)
    return out


def _exact_volume(frames, case):
    """(V, |V|^2 or |V|) of Eq. 5 - Eq. 7 in float64; frames [nl][ny][nx]."""
    nl, ny, nx = frames.shape
    x0, y0, wx, wy = _window(case)
    lam = float(_wavelengths(nl)[0])
    screen = _chirp(ny, PITCH, 1 / (lam * Z))[:, None] * _chirp(nx, PITCH, 1 / (lam * Z))[None, :]
    v = torch.fft.fft(_holograms(_rescaled(frames, nl), case, screen), dim=0)
    mag = PITCH * PITCH / (lam * Z)
    phase = math.pi / 2 - 2 * math.pi * math.fmod(Z / lam, 1.0)
    # reconstructed pixel lambda_1 z / (N d) along each axis (Eq. 4)
    ox = _chirp(nx, lam * Z / (nx * PITCH), 1 / (lam * Z))[x0:x0 + wx]
    oy = _chirp(ny, lam * Z / (ny * PITCH), 1 / (lam * Z))[y0:y0 + wy]
    k = complex(mag * math.cos(phase), mag * math.sin(phase))
    v *= (k * oy)[:, None] * ox[None, :]
    p = v.real ** 2 + v.imag ** 2
    return v, (p.sqrt() if case["magnitude"] else p)


def _zernike(nx, ny):
    """Noll's Z_1 .. Z_15 over the frame, RMS-normalised on the disk of radius min(nx, ny) / 2."""
    x = (torch.arange(nx, device="cuda", dtype=torch.float64) - nx / 2)[None, :] * (2.0 / min(nx, ny))
    y = (torch.arange(ny, device="cuda", dtype=torch.float64) - ny / 2)[:, None] * (2.0 / min(nx, ny))
    x, y = x.expand(ny, nx), y.expand(ny, nx)
    r2, th = x * x + y * y, torch.atan2(y, x)
    r = r2.sqrt()
    s = math.sqrt
    return torch.stack([
        torch.ones_like(r), 2 * x, 2 * y, s(3) * (2 * r2 - 1), s(6) * r2 * torch.sin(2 * th), s(6) * r2 * torch.cos(2 * th),
        s(8) * (3 * r2 - 2) * y, s(8) * (3 * r2 - 2) * x, s(8) * r2 * r * torch.sin(3 * th), s(8) * r2 * r * torch.cos(3 * th),
        s(5) * (6 * r2 * r2 - 6 * r2 + 1), s(10) * (4 * r2 - 3) * r2 * torch.cos(2 * th), s(10) * (4 * r2 - 3) * r2 * torch.sin(2 * th),
        s(10) * r2 * r2 * torch.cos(4 * th), s(10) * r2 * r2 * torch.sin(4 * th)])


def _exact_sharpness(frames, case, coeffs, z):
    """[loss, dL/dz, dL/dc_1..15, |V|^2]: autograd through the float64 screen, the transforms
    differentiated by their adjoint (linear in the screen, so one frame at a time)."""
    nl, ny, nx = frames.shape
    x0, y0, wx, wy = _window(case)
    lam = float(_wavelengths(nl)[0])
    u = _rescaled(frames, nl)
    zern = _zernike(nx, ny)
    c = torch.tensor(coeffs, device="cuda", dtype=torch.float64, requires_grad=True)
    zt = torch.tensor(z, device="cuda", dtype=torch.float64, requires_grad=True)
    kx = torch.arange(nx, device="cuda", dtype=torch.float64) - nx / 2.0
    ky = torch.arange(ny, device="cuda", dtype=torch.float64) - ny / 2.0
    r2 = (ky[:, None] ** 2 + kx[None, :] ** 2) * (PITCH * PITCH)
    phi = torch.tensordot(c, zern, dims=1) - math.pi * r2 / (lam * zt)
    screen = torch.polar(torch.ones_like(phi), phi)
    with torch.no_grad():
        v = torch.fft.fft(_holograms(u, case, screen.detach()), dim=0)
        k2 = (PITCH * PITCH / (lam * z)) ** 2
        p = (v.real ** 2 + v.imag ** 2) * k2
        s1, s2 = p.sum(), (p * p).sum()
        loss = -s2 / (s1 * s1)
        # dL/d conj(V), then back through Eq. 7, the window and the DFT of Eq. 6
        w = v * (2 * k2 * (-2 * p / s1 ** 2 + 2 * s2 / s1 ** 3))
        w = torch.fft.ifft(w, dim=0) * nl
        g = torch.zeros((ny, nx), device="cuda", dtype=torch.complex128)
        full = torch.zeros((ny, nx), device="cuda", dtype=torch.complex128)
        for t in range(nl):
            full[y0:y0 + wy, x0:x0 + wx] = w[t]
            g += torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(full))) * u[t]
    # real part of <g, d screen>; |K| also depends on z but the loss does not on |K|
    (g.real * screen.real + g.imag * screen.imag).sum().backward()
    return [float(loss), float(zt.grad), c.grad, p]


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        gen = _generator(seed)
        stacks = [_frames(nx, ny, n, case["scene"], gen) for nx, ny, n in _sizes(case)]
        out = []
        while stacks:
            f = stacks.pop(0)
            n, ny, nx = f.shape
            out.append(_exact_volume(f, dict(case, nx=nx, ny=ny, nl=n, x0=0, y0=0, wx=nx, wy=ny))[1])
        return out
    nl = case["nl"]
    if op in ("sliding", "sliding_cuts"):
        # the gate after one push: its first `new` slots hold the second sweep
        stream = _stream(case, seed)
        gate = torch.cat([stream[nl:nl + case["new"]], stream[case["new"]:nl]])
        p = _exact_volume(gate, case)[1]
    else:
        frames = _frames(case["nx"], case["ny"], nl, case["scene"], _generator(seed))
        if op == "sharpness":
            return _exact_sharpness(frames, case, *_pupil(seed))
        v, p = _exact_volume(frames, case)
    if op == "sliding":
        return p
    x, y, q = _position(case)
    cuts = [p[q].clone(), p[:, y].clone(), p[:, :, x].clone()]
    if op == "sliding_cuts":
        return cuts
    return [p] + ([v] if case["complex"] else []) + (cuts if case["cuts"] else [])
