"""What this framework is timed on: whole reconstructions through its public entry points.

Every pass is one call (or one batch call) as a user's program makes it: the inputs, the context or
batch handle and the output buffer are in hand, the call returns chi (or the field map).  Inputs are
brachytherapy-like volumes: smooth tissue inside an elliptical mask, a few titanium seeds and needles
of 120-200 ppm, the dipole field of that with 0.02 ppm of noise.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2006_09808_gb300 as pcs

#: 1/L with L = sqrt(4/9 + 8) (2-D) and sqrt(4/9 + 12) (3-D): bounds on ||K|| for every 0/1 mask.
STEP_2D = 1.0 / math.sqrt(4.0 / 9.0 + 8.0)
STEP_3D = 1.0 / math.sqrt(4.0 / 9.0 + 12.0)
COMPILED = (64, 128, 192, 256, 384, 512)
SHAPES_3D = ((32, 64), (64, 64), (32, 128), (64, 128), (128, 128), (32, 256), (64, 256), (128, 256))
B0_TESLA, T_SHIFT = 3.0, 0.6e-3
THRESHOLD = 0.1
RAD_PER_PPM = 2.0 * math.pi * 42.577478518 * B0_TESLA * T_SHIFT
POWER_ITERS = 300


def _case(kind, H, W, S, N=0, lam=5e-4, tv=0, axis=0, weighted=False, voxel="", volumes="", name=None):
    c = {"kind": kind, "H": H, "W": W, "S": S, "N": N, "lam": lam, "tv": tv, "axis": axis, "weighted": weighted,
         "voxel": voxel, "volumes": volumes}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one 64 x 64 slice, the smallest reconstruction: a chain of 300 iterations, latency alone
        _case("slices", 64, 64, 1, 300, lam=1e-3, name="slice_64"),
        # one slice of an interventional scan, reconstructed as it arrives
        _case("slices", 256, 256, 1, 500, name="slice_256"),
        # the needle phantom's volume, rounded to the compiled size: fewer slices than the GPU holds
        _case("slices", 128, 128, 42, 500, name="volume_128"),
        # the headline volume: 64 slices of 256 x 256, 500 iterations
        _case("slices", 256, 256, 64, 500, name="volume_256"),
        # magnitude weighting and isotropic TV, as QSM users run it, on a radix-3 size
        _case("slices", 192, 192, 24, 400, tv=1, weighted=True, name="weighted_iso_192"),
        # host buffers in, host buffers out (copies inside the call), a large slice size
        _case("host", 384, 384, 32, 200, name="host_384"),
        # volumes of mixed sizes and lambdas waiting together: one batch call
        _case("batch", 0, 0, 0, 400, volumes="128x128x40@0.0002,192x192x30@0.0005,256x256x64@0.0005,"
              "384x384x24@0.001,512x512x16@0.0002", name="batch_uneven"),
        # the stent acquisition's own shape (row length 258 = 2 x 3 x 43), through a context
        _case("slices", 256, 258, 25, 500, name="native_258"),
        # the seeds acquisition's own shape (row length 132 = 4 x 3 x 11), the one-call form
        _case("generic", 128, 132, 12, 500, name="native_132"),
        # the literal 3-D reading on the headline volume
        _case("volume3d", 256, 256, 64, 500, name="volume3d_256"),
        # a small 3-D volume with the acquisition's 2 x 0.72 x 0.72 mm voxel and a magnitude weighting
        _case("volume3d", 128, 128, 32, 300, weighted=True, voxel="2,0.72,0.72", name="volume3d_128"),
        # the field map of two acquisitions, before the solve: one pass over memory
        _case("fieldmap", 256, 256, 64, name="fieldmap_256"),
    ]


def _smooth(n):
    """Even, in the any-size path's range, prime factors at most 61."""
    if n % 2 or not 8 <= n <= 512:
        return False
    for q in range(2, 62):
        while n % q == 0:
            n //= q
    return n == 1


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["slices", "slices", "slices", "native", "native", "host", "batch", "volume3d", "fieldmap"])
    lam = rng.choice([2e-4, 5e-4, 1e-3])
    tv, axis = rng.choice([0, 0, 1]), rng.choice([0, 0, 1])
    if kind in ("slices", "host"):
        n = rng.choice(COMPILED)
        N = rng.randrange(100, 501)
        most = max(1, int(2.0e9 / (n * n * N)))
        S = _log_int(rng, 1, min(96, most))
        return _case(kind, n, n, S, N, lam, tv, axis, weighted=kind == "slices" and rng.random() < 0.3)
    if kind == "native":
        while True:
            H, W = 2 * _log_int(rng, 16, 256), 2 * _log_int(rng, 16, 256)
            if _smooth(H) and _smooth(W) and not (H == W and H in COMPILED):
                break
        N = rng.randrange(100, 501)
        S = _log_int(rng, 1, max(1, min(48, int(8.0e8 / (H * W * N)))))
        return _case(rng.choice(["slices", "generic"]), H, W, S, N, lam, tv, axis, weighted=rng.random() < 0.3)
    if kind == "batch":
        vols = []
        for _ in range(rng.randrange(2, 6)):
            H, W = rng.choice([(n, n) for n in COMPILED] + [(256, 258), (128, 132)])
            S = _log_int(rng, 4, 40)
            vols.append("%dx%dx%d@%g" % (H, W, S if H < 512 else min(S, 12), rng.choice([2e-4, 5e-4, 1e-3])))
        return _case("batch", 0, 0, 0, rng.randrange(100, 301), axis=axis, volumes=",".join(vols))
    if kind == "volume3d":
        S, n = rng.choice(SHAPES_3D)
        N = rng.randrange(50, 501) if n < 256 else rng.randrange(50, 251)
        voxel = rng.choice(["", "", "2,0.72,0.72", "%.2f,1,1" % rng.uniform(0.8, 3.0)])
        return _case("volume3d", n, n, S, N, lam, tv, weighted=rng.random() < 0.3, voxel=voxel)
    H, W = rng.randrange(33, 400), rng.randrange(33, 400)
    return _case("fieldmap", H, W, _log_int(rng, 1, max(1, min(96, 4000000 // (H * W)))))


# --------------------------------------------------------------------------- inputs


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _freq(n, dev):
    return torch.fft.fftfreq(n, dtype=torch.float64, device=dev)


def _dipole_2d(H, W, axis, dev):
    ky, kx = _freq(H, dev)[:, None], torch.fft.rfftfreq(W, dtype=torch.float64, device=dev)[None, :]
    kp = ky if axis == 0 else kx
    k2 = kx * kx + ky * ky
    return torch.where(k2 > 0, 1.0 / 3.0 - kp * kp / torch.where(k2 > 0, k2, 1.0), 0.0)


def _dipole_3d(S, H, W, voxel, dev):
    dz, dy, dx = voxel
    kz, ky = _freq(S, dev)[:, None, None] / dz, _freq(H, dev)[None, :, None] / dy
    kx = torch.fft.rfftfreq(W, dtype=torch.float64, device=dev)[None, None, :] / dx
    k2 = kx * kx + ky * ky + kz * kz
    return torch.where(k2 > 0, 1.0 / 3.0 - kz * kz / torch.where(k2 > 0, k2, 1.0), 0.0)


def _lowpass(x, sigma):
    H, W = x.shape[-2:]
    ky, kx = _freq(H, x.device)[:, None], torch.fft.rfftfreq(W, dtype=torch.float64, device=x.device)[None, :]
    g = torch.exp(-2.0 * (math.pi * sigma) ** 2 * (kx * kx + ky * ky)).to(x.dtype)
    return torch.fft.irfft2(torch.fft.rfft2(x) * g, s=(H, W))


def _volume(S, H, W, seed, axis=0, voxel=None):
    """(field float32, mask uint8) [S][H][W] of one acquisition."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(seed)
    rng = random.Random(seed)
    y = torch.arange(H, device=dev, dtype=torch.float32)[:, None]
    x = torch.arange(W, device=dev, dtype=torch.float32)[None, :]
    inside = ((x - (W - 1) / 2) / (0.45 * W)) ** 2 + ((y - (H - 1) / 2) / (0.35 * H)) ** 2 <= 1.0
    if S == 1 and H <= 64:
        inside = torch.ones_like(inside)  # the small phantom is reconstructed with a full mask
    tissue = _lowpass(torch.randn((S, H, W), generator=gen, device=dev), 4.0)
    tissue = tissue - tissue.mean()
    chi = tissue * (0.5 / tissue.std().clamp_min(1e-12)) * inside
    for _ in range(6 if S > 1 else 3):
        r, t = 0.85 * math.sqrt(rng.random()), rng.uniform(0, 2 * math.pi)
        ci, cj = (H - 1) / 2 + r * 0.35 * H * math.sin(t), (W - 1) / 2 + r * 0.45 * W * math.cos(t)
        if rng.random() < 0.5:
            shape, run = (y - ci) ** 2 + (x - cj) ** 2 <= 4.0, min(3, S)
        else:
            a, half = rng.uniform(0, math.pi), 0.5 * min(rng.uniform(20, 60), H / 3)
            along = (x - cj) * math.cos(a) + (y - ci) * math.sin(a)
            across = (y - ci) * math.cos(a) - (x - cj) * math.sin(a)
            shape, run = (along.abs() <= half) & (across.abs() <= 1.0), min(rng.randrange(8, 65), S)
        s0 = rng.randrange(0, S - run + 1)
        part = chi[s0:s0 + run]
        chi[s0:s0 + run] = torch.where(shape, torch.full_like(part, rng.uniform(120.0, 200.0)), part)
    if voxel is None:
        f = torch.fft.irfft2(torch.fft.rfft2(chi) * _dipole_2d(H, W, axis, dev).float(), s=(H, W))
    else:
        f = torch.fft.irfftn(torch.fft.rfftn(chi) * _dipole_3d(S, H, W, voxel, dev).float(), s=(S, H, W))
    f = f + 0.02 * torch.randn((S, H, W), generator=gen, device=dev)
    return f.contiguous(), inside.to(torch.uint8).expand(S, H, W).contiguous()


def _magnitude(mask, seed):
    """A smooth magnitude image in [0.2, 1] inside the mask, 0 outside."""
    gen = torch.Generator(device=mask.device).manual_seed(seed + 7)
    w = _lowpass(torch.randn(mask.shape, generator=gen, device=mask.device), 6.0)
    w = 0.2 + 0.8 * (w - w.min()) / (w.max() - w.min()).clamp_min(1e-12)
    return (w.clamp(0.2, 1.0) * mask).float().contiguous()


def _echoes(S, H, W, seed):
    """The two complex acquisitions, without and with the readout shift."""
    field, mask = _volume(S, H, W, seed)
    gen = torch.Generator(device=field.device).manual_seed(seed + 13)
    mag = torch.where(mask != 0, _magnitude(mask, seed), torch.full_like(field, 0.02))
    phase = _lowpass(torch.randn((S, H, W), generator=gen, device=field.device), 8.0)
    phase = phase * (math.pi / phase.abs().max().clamp_min(1e-12))
    s0, s1 = torch.polar(mag, phase), torch.polar(mag, phase + RAD_PER_PPM * field)

    def noise():
        return 0.002 * torch.view_as_complex(torch.randn((S, H, W, 2), generator=gen, device=field.device))

    return s0 + noise(), s1 + noise()


def _voxel(case):
    return tuple(float(v) for v in case["voxel"].split(",")) if case["voxel"] else (1.0, 1.0, 1.0)


def _volumes(case):
    """[(H, W, S, lambda)] of a batch."""
    out = []
    for v in case["volumes"].split(","):
        shape, lam = v.split("@")
        H, W, S = (int(n) for n in shape.split("x"))
        out.append((H, W, S, float(lam)))
    return out


def _inputs(case, seed):
    if case["kind"] == "fieldmap":
        return _echoes(case["S"], case["H"], case["W"], seed)
    if case["kind"] == "batch":
        return [_volume(S, H, W, seed + 101 * k, case["axis"]) for k, (H, W, S, _) in enumerate(_volumes(case))]
    voxel = _voxel(case) if case["kind"] == "volume3d" else None
    field, mask = _volume(case["S"], case["H"], case["W"], seed, case["axis"], voxel)
    return field, mask, _magnitude(mask, seed) if case["weighted"] else None


# --------------------------------------------------------------------------- a pass


class _Handle:
    """A context or batch that a user's program keeps; released with the state."""

    def __init__(self, h, release):
        self.h, self._release = h, release

    def __del__(self):
        if self.h is not None:
            self._release(self.h)
            self.h = None


def _context(case):
    kernel = pcs.KERNEL_STREAMING if case["weighted"] and case["H"] == case["W"] and case["H"] in COMPILED else 0
    h = pcs.pcs_create(case["H"], case["W"], case["S"], b0_axis=case["axis"], tv=case["tv"], kernel=kernel)
    return _Handle(h, pcs.pcs_destroy)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fieldmap":
        s0, s1 = _inputs(case, seed)
        return {"case": case, "s0": s0, "s1": s1, "field": torch.empty(s0.shape, device=s0.device),
                "weight": torch.empty(s0.shape, device=s0.device),
                "mask": torch.empty(s0.shape, dtype=torch.uint8, device=s0.device)}
    if kind == "batch":
        vols = [(f, m, lam, torch.empty_like(f))
                for (f, m), (_, _, _, lam) in zip(_inputs(case, seed), _volumes(case))]
        batch = _Handle(pcs.pcs_batch_create(autotune=True, b0_axis=case["axis"]), pcs.pcs_batch_destroy)
        pcs.pcs_batch_solve(batch.h, vols, 0)  # contexts, tuning and step sizes of these slice sizes
        return {"case": case, "batch": batch, "volumes": vols}
    field, mask, weight = _inputs(case, seed)
    st = {"case": case, "field": field, "mask": mask, "weight": weight, "chi": torch.empty_like(field)}
    if kind == "host":
        st["ctx"] = _context(case)
        for key in ("field", "mask", "chi"):
            st[key] = st[key].cpu().pin_memory().numpy()
    elif kind == "slices":
        st["ctx"] = _context(case)
    return st


def run(state):
    case = state["case"]
    kind, lam, N = case["kind"], case["lam"], case["N"]
    if kind == "fieldmap":
        pcs.pcs_field_map(state["s0"], state["s1"], T_SHIFT, B0_TESLA, THRESHOLD, state["field"], state["weight"],
                          state["mask"])
        return {"field": state["field"], "weight": state["weight"], "mask": state["mask"]}
    if kind == "batch":
        pcs.pcs_batch_solve(state["batch"].h, state["volumes"], N)
        return [v[3] for v in state["volumes"]]
    f, m, w, chi = state["field"], state["mask"], state["weight"], state["chi"]
    if kind == "host":
        pcs.pcs_solve_slices_host(state["ctx"].h, f, m, lam, STEP_2D, STEP_2D, N, chi)
    elif kind == "generic":
        pcs.pcs_solve_slices_generic(f, m, lam, STEP_2D, STEP_2D, N, chi, tv=case["tv"], weight=w,
                                     b0_axis=case["axis"])
    elif kind == "volume3d":
        pcs.pcs_solve_volume_3d(f, m, lam, STEP_3D, STEP_3D, N, chi, tv=case["tv"], weight=w,
                                voxel=_voxel(case) if case["voxel"] else None)
    elif w is not None:
        pcs.pcs_solve_slices_weighted(state["ctx"].h, f, m, w, lam, STEP_2D, STEP_2D, N, chi)
    else:
        pcs.pcs_solve_slices(state["ctx"].h, f, m, lam, STEP_2D, STEP_2D, N, chi)
    return chi


def work(case):
    """Field and mask (and weighting) in, chi out, once each; per voxel and iteration two round trips of
    a real FFT over the slice (10 log2 of its size) or the volume, and about 30 pointwise operations."""
    if case["kind"] == "fieldmap":
        n = case["S"] * case["H"] * case["W"]
        return {"bytes": 25 * n, "flops": 40 * n}
    vols = _volumes(case) if case["kind"] == "batch" else [(case["H"], case["W"], case["S"], case["lam"])]
    nbytes = flops = 0.0
    for H, W, S, _ in vols:
        n = S * H * W
        points = n if case["kind"] == "volume3d" else H * W
        nbytes += n * (13 if case["weighted"] else 9)
        flops += n * case["N"] * (10.0 * math.log2(points) + (40 if case["kind"] == "volume3d" else 30))
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------- 64-bit values


def _grad(x, dims):
    out = []
    for d in dims:
        g = torch.zeros_like(x)
        n = x.shape[d]
        g.narrow(d, 0, n - 1).copy_(x.narrow(d, 1, n - 1) - x.narrow(d, 0, n - 1))
        out.append(g)
    return out


def _grad_adjoint(q, dims):
    out = torch.zeros_like(q[0])
    for a, d in zip(q, dims):
        n = a.shape[d]
        out.narrow(d, 1, n - 1).add_(a.narrow(d, 0, n - 1))
        out.narrow(d, 0, n - 1).sub_(a.narrow(d, 0, n - 1))
    return out


def _convolution(kernel, volume):
    dims = (0, 1, 2) if volume else (1, 2)

    def apply(x):
        shape = [x.shape[d] for d in dims]
        return torch.fft.irfftn(torch.fft.rfftn(x, dim=dims) * kernel, s=shape, dim=dims)

    return apply, dims


def _primal_dual(field, mask, weight, D, dims, lam, step, N, tv):
    f, M = field.double(), mask.double()
    Wt = M if weight is None else weight.double()
    chi, bar, p = torch.zeros_like(f), torch.zeros_like(f), torch.zeros_like(f)
    q = [torch.zeros_like(f) for _ in dims]
    for _ in range(N):
        p = (p + step * Wt * (D(bar) - f)) / (1.0 + step / lam)
        q = [a + step * M * g for a, g in zip(q, _grad(bar, dims))]
        if tv:
            norm = torch.sqrt(sum(a * a for a in q)).clamp_min(1.0)
            q = [a / norm for a in q]
        else:
            q = [a.clamp(-1.0, 1.0) for a in q]
        new = chi - step * (D(Wt * p) + _grad_adjoint([M * a for a in q], dims))
        bar, chi = 2.0 * new - chi, new
    return chi


def _norm_of_operator(H, W, D, dims):
    """||[D; G]|| of a full mask by the power iteration, as the batch takes its step sizes."""
    gen = torch.Generator(device="cpu").manual_seed(1)
    x = (2.0 * torch.rand((1, H, W), generator=gen, dtype=torch.float64) - 1.0).to(_device())
    est = 1.0
    for _ in range(POWER_ITERS):
        x = x / x.norm()
        y = D(D(x)) + _grad_adjoint(_grad(x, dims), dims)
        est, x = float((x * y).sum()), y
    return math.sqrt(est)


def exact(case, seed):
    kind = case["kind"]
    if kind == "fieldmap":
        s0, s1 = (s.to(torch.complex128) for s in _inputs(case, seed))
        mag2 = s0.real * s0.real + s0.imag * s0.imag
        mask = mag2 >= THRESHOLD ** 2 * mag2.max()
        field = torch.where(mask, torch.angle(s1 * s0.conj()) / RAD_PER_PPM, 0.0)
        return {"field": field, "weight": torch.sqrt(mag2 / mag2.max()), "mask": None}
    dev = _device()
    if kind == "batch":
        out, steps = [], {}
        for (f, m), (H, W, _, lam) in zip(_inputs(case, seed), _volumes(case)):
            D, dims = _convolution(_dipole_2d(H, W, case["axis"], dev), False)
            if (H, W) not in steps:
                steps[H, W] = 1.0 / _norm_of_operator(H, W, D, dims)
            out.append(_primal_dual(f, m, None, D, dims, lam, steps[H, W], case["N"], case["tv"]))
        return out
    field, mask, weight = _inputs(case, seed)
    if kind == "volume3d":
        D, dims = _convolution(_dipole_3d(case["S"], case["H"], case["W"], _voxel(case), dev), True)
        chi = _primal_dual(field, mask, weight, D, dims, case["lam"], STEP_3D, case["N"], case["tv"])
    else:
        D, dims = _convolution(_dipole_2d(case["H"], case["W"], case["axis"], dev), False)
        chi = _primal_dual(field, mask, weight, D, dims, case["lam"], STEP_2D, case["N"], case["tv"])
    return chi.cpu().numpy() if kind == "host" else chi
