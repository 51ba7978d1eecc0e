"""The propagations that programs built on this library run, as measurable cases.

Every case goes through the public entry points of ``paper_1107_5578_gb300`` (``cwo.Plan`` and
``hologram.HologramProblem``) on complex64 fields that are resident on the GPU.  ``listed()`` holds
the cases that are always measured, ``draw()`` picks further ones from the same ranges, and
``exact()`` gives the same outputs in 64 bits from plain torch.
"""
from __future__ import annotations

import math

import torch

from paper_1107_5578_gb300 import cwo, hologram

DEVICE = "cuda"
TWO_PI = 2.0 * math.pi
# the largest number of field samples of one drawn pass (16 fields of 2048^2, the largest listed)
MAX_SAMPLES = 16 * 2048 * 2048


def listed():
    return [
        # one small field, the smallest size that a propagation service is asked for: latency
        {"name": "asm-256-one", "kind": "asm", "nx": 256, "ny": 256, "batch": 1, "cached": False,
         "adjoint": False, "per_item_z": False, "pitch": 10e-6, "wavelength": 633e-9, "z": 0.05},
        # many small fields at once: the frames of a video, the sub-apertures of a sensor
        {"name": "asm-512-batch64", "kind": "asm", "nx": 512, "ny": 512, "batch": 64, "cached": False,
         "adjoint": False, "per_item_z": False, "pitch": 10e-6, "wavelength": 633e-9, "z": 0.05},
        # an autofocus sweep back to the object: an odd number of fields, each with its own distance
        {"name": "asm-1024-batch7-each-z-adjoint", "kind": "asm", "nx": 1024, "ny": 1024, "batch": 7, "cached": False,
         "adjoint": True, "per_item_z": True, "pitch": 8e-6, "wavelength": 532e-9, "z": 0.1},
        # the library's benchmark: full-size fields at one distance, transfer function kept in the plan
        {"name": "asm-2048-batch16-cached", "kind": "asm", "nx": 2048, "ny": 2048, "batch": 16, "cached": True,
         "adjoint": False, "per_item_z": False, "pitch": 10e-6, "wavelength": 633e-9, "z": 0.05},
        # the largest fields the library takes (high-resolution holograms)
        {"name": "asm-4096-batch2-cached", "kind": "asm", "nx": 4096, "ny": 4096, "batch": 2, "cached": True,
         "adjoint": False, "per_item_z": False, "pitch": 3.74e-6, "wavelength": 532e-9, "z": 0.2},
        # off-axis reconstruction of a wide strip: shifted, band-limited, rectangular, an odd batch
        {"name": "shifted-asm-4096x1024-batch3", "kind": "shifted_asm", "nx": 4096, "ny": 1024, "batch": 3,
         "pitch": 6e-6, "wavelength": 532e-9, "z": 0.1, "ox": 300e-6, "oy": -150e-6, "band_limited": True},
        # paraxial propagation of full-size fields
        {"name": "fresnel-2048-batch16", "kind": "fresnel", "nx": 2048, "ny": 2048, "batch": 16, "adjoint": False,
         "pitch": 8e-6, "wavelength": 532e-9, "z": 0.2},
        # back-propagation of one field of the largest size
        {"name": "fresnel-4096-one-adjoint", "kind": "fresnel", "nx": 4096, "ny": 4096, "batch": 1, "adjoint": True,
         "pitch": 6e-6, "wavelength": 633e-9, "z": 0.3},
        # one hologram reconstructed on 16 planes
        {"name": "fresnel-stack-2048-16-planes", "kind": "stack", "nx": 2048, "ny": 2048, "planes": 16,
         "pitch": 8e-6, "wavelength": 532e-9, "z0": 0.1, "z1": 0.4},
        # one iteration of the kinoform loop and the reconstruction that its progress is judged by
        {"name": "gs-1024", "kind": "gs", "n": 1024, "iterations": 1, "pitch": 10e-6, "wavelength": 633e-9, "z": 0.1},
        # loss and gradient of a phase-only hologram for a 1920 x 1080 modulator
        {"name": "hologram-1080x1920", "kind": "hologram", "h": 1080, "w": 1920, "canvas": 2048, "pitch": 6.4e-6,
         "wavelength": 520e-9, "z": 0.15},
        # what a propagation service runs: fields of one size, each with its own method and geometry
        {"name": "items-512-batch12", "kind": "items", "nx": 512, "ny": 512, "batch": 12, "fresnel_share": 0.3},
    ]


def _side(rng, lo=16, hi=4096):
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def _geometry(rng):
    return {"pitch": round(rng.uniform(4e-6, 10e-6), 8), "wavelength": rng.choice([450e-9, 532e-9, 633e-9]),
            "z": round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 5)}


def _batch(rng, samples, most=64):
    top = max(1, min(most, MAX_SAMPLES // samples))
    return max(1, min(top, round(math.exp(rng.uniform(0.0, math.log(top))))))


def draw(rng):
    """One more case: every power-of-two side that the plans take, square and rectangular fields,
    any batch, the geometries of the library's serving mix."""
    kind = rng.choice(["asm", "asm", "asm", "fresnel", "fresnel", "stack", "items", "gs", "hologram", "shifted_asm",
                       "shifted_fresnel", "fourier"])
    g = _geometry(rng)
    nx = _side(rng, 32)
    ny = nx if rng.random() < 0.5 else _side(rng, 32)
    if kind == "asm":
        case = {"kind": kind, "nx": nx, "ny": ny, "batch": _batch(rng, nx * ny), "cached": rng.random() < 0.5,
                "adjoint": rng.random() < 0.3, "per_item_z": False, **g}
        case["per_item_z"] = not case["cached"] and rng.random() < 0.3
        return case
    if kind == "fresnel":
        return {"kind": kind, "nx": nx, "ny": ny, "batch": _batch(rng, nx * ny), "adjoint": rng.random() < 0.3, **g}
    if kind == "stack":
        return {"kind": kind, "nx": nx, "ny": ny, "planes": max(2, _batch(rng, nx * ny, 24)), "pitch": g["pitch"],
                "wavelength": g["wavelength"], "z0": 0.1, "z1": round(rng.uniform(0.2, 0.5), 4)}
    if kind == "items":
        nx, ny = _side(rng, 64, 2048), _side(rng, 64, 2048)
        return {"kind": kind, "nx": nx, "ny": ny, "batch": _batch(rng, nx * ny, 16), "fresnel_share": 0.3}
    if kind == "gs":
        return {"kind": kind, "n": _side(rng, 128, 1024), "iterations": 1, "pitch": g["pitch"], "wavelength": g["wavelength"],
                "z": g["z"]}
    if kind == "hologram":
        canvas = _side(rng, 256, 2048)
        return {"kind": kind, "h": rng.randint(canvas // 4, canvas), "w": rng.randint(canvas // 3, canvas),
                "canvas": canvas, "pitch": g["pitch"], "wavelength": g["wavelength"], "z": g["z"]}
    if kind == "shifted_asm":
        return {"kind": kind, "nx": nx, "ny": ny, "batch": _batch(rng, nx * ny, 8), "ox": round(rng.uniform(-5e-4, 5e-4), 7),
                "oy": round(rng.uniform(-5e-4, 5e-4), 7), "band_limited": rng.random() < 0.5, **g}
    if kind == "shifted_fresnel":
        return {"kind": kind, "nx": nx, "ny": ny, "batch": _batch(rng, nx * ny, 8), "pitch1": round(rng.uniform(4e-6, 10e-6), 8),
                "ox1": round(rng.uniform(-5e-4, 5e-4), 7), "oy1": round(rng.uniform(-5e-4, 5e-4), 7), **g}
    return {"kind": "fourier", "nx": nx, "ny": ny, "batch": _batch(rng, nx * ny, 8), **g}


# ---------------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _fields(case, seed, batch):
    """complex64 fields, amplitude U[0, 1), phase U[0, 2 pi): what a diffuse object sends out."""
    g = _gen(seed)
    shape = (batch, case["ny"], case["nx"])
    amp = torch.rand(shape, generator=g, device=DEVICE)
    ph = torch.rand(shape, generator=g, device=DEVICE) * TWO_PI
    return torch.polar(amp, ph)


def _distances(case):
    """the plan's z, or one distance for each field of the batch, around the plan's"""
    if not case["per_item_z"]:
        return None
    return [case["z"] * (0.8 + 0.4 * (k + 0.5) / case["batch"]) for k in range(case["batch"])]


def _plane_distances(case):
    n = case["planes"]
    return [case["z0"] + (case["z1"] - case["z0"]) * k / (n - 1) for k in range(n)]


def _items(case, seed):
    """method and geometry of each item: the library's serving mix (30% Fresnel)"""
    out = []
    for k in range(case["batch"]):
        u = [((seed * 7919 + k * 104729 + j * 1299709) % 9973) / 9973.0 for j in range(3)]
        fresnel = k >= round(case["batch"] * (1.0 - case["fresnel_share"]))   # a service orders its batch by type
        out.append({"type": cwo.FRESNEL_CONV if fresnel else cwo.ANGULAR, "z": 0.01 + 0.49 * u[0],
                    "wavelength": (450e-9, 532e-9, 633e-9)[int(3 * u[1])], "dx": 4e-6 + 6e-6 * u[2]})
    return out


def _gs_inputs(case, seed):
    """object amplitude (a smooth image of 30 spots) and the field it starts from (random phase)"""
    n, g = case["n"], _gen(seed)
    p = torch.rand((30, 4), generator=g, device=DEVICE).tolist()
    i = torch.arange(n, device=DEVICE, dtype=torch.float32)
    img = torch.full((n, n), 0.02, device=DEVICE)
    for cy, cx, s, a in p:
        sig = n / 64.0 + (n / 8.0 - n / 64.0) * s
        ey = torch.exp(-((i - cy * n) ** 2) / (2.0 * sig * sig))
        ex = torch.exp(-((i - cx * n) ** 2) / (2.0 * sig * sig))
        img += (0.3 + 0.7 * a) * ey[:, None] * ex[None, :]
    amp = torch.sqrt(img / img.max())
    ph = torch.rand((n, n), generator=g, device=DEVICE) * TWO_PI
    return amp[None].contiguous(), torch.polar(amp, ph)[None].contiguous()


def _hologram_inputs(case, seed):
    """the phase to improve (uniform) and the intensity wanted on its window (spots, mean near 1)"""
    h, w, g = case["h"], case["w"], _gen(seed)
    phi = torch.rand((h, w), generator=g, device=DEVICE) * TWO_PI
    p = torch.rand((20, 4), generator=g, device=DEVICE).tolist()
    y = torch.arange(h, device=DEVICE, dtype=torch.float32)
    x = torch.arange(w, device=DEVICE, dtype=torch.float32)
    tgt = torch.zeros((h, w), device=DEVICE)
    for cy, cx, s, a in p:
        sig = 0.02 * w + 0.06 * w * s
        ey = torch.exp(-((y - cy * h) ** 2) / (2.0 * sig * sig))
        ex = torch.exp(-((x - cx * w) ** 2) / (2.0 * sig * sig))
        tgt += (0.5 + 0.5 * a) * ey[:, None] * ex[None, :]
    return phi, tgt / tgt.mean()


# ---------------------------------------------------------------------------------- the passes
def prepare(case, seed):
    k = case["kind"]
    if k == "asm":
        flags = cwo.FLAG_CACHE_H if case["cached"] else 0
        plan = cwo.Plan(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z"], cwo.ANGULAR, flags)
        plan.reserve(case["batch"])
        x = _fields(case, seed, case["batch"])
        return {"case": case, "plan": plan, "x": x[0].contiguous() if case["batch"] == 1 else x, "z": _distances(case)}
    if k == "fresnel":
        plan = cwo.Plan(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z"], cwo.FRESNEL_CONV)
        plan.reserve(case["batch"])
        x = _fields(case, seed, case["batch"])
        return {"case": case, "plan": plan, "x": x[0].contiguous() if case["batch"] == 1 else x, "z": None}
    if k == "stack":
        plan = cwo.Plan(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z0"], cwo.FRESNEL_CONV)
        plan.reserve(case["planes"])
        return {"case": case, "plan": plan, "x": _fields(case, seed, 1)[0].contiguous(), "zs": _plane_distances(case)}
    if k == "items":
        plan = cwo.Plan(case["nx"], case["ny"])
        plan.reserve(case["batch"])
        return {"case": case, "plan": plan, "x": _fields(case, seed, case["batch"]), "items": _items(case, seed)}
    if k == "gs":
        plan = cwo.Plan(case["n"], case["n"], case["pitch"], case["pitch"], case["wavelength"], case["z"], cwo.ANGULAR, cwo.FLAG_CACHE_H)
        amp, field = _gs_inputs(case, seed)
        return {"case": case, "plan": plan, "amp": amp, "field": field}
    if k == "hologram":
        prob = hologram.HologramProblem(case["h"], case["w"], case["canvas"], case["pitch"], case["wavelength"], case["z"],
                                        seed=1, device=DEVICE)
        phi, prob.target = _hologram_inputs(case, seed)
        return {"case": case, "problem": prob, "phi": phi.requires_grad_(True)}
    if k == "shifted_asm":
        sh = cwo.band_limit(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z"]) \
            if case["band_limited"] else cwo.Shift()
        sh.ox, sh.oy = case["ox"], case["oy"]
        plan = cwo.Plan(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z"], shift=sh)
    elif k == "shifted_fresnel":
        sf = cwo.ShiftedFresnel(case["pitch1"], case["pitch1"], 0.0, 0.0, case["ox1"], case["oy1"])
        plan = cwo.Plan(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z"], shifted_fresnel=sf)
    else:
        plan = cwo.Plan(case["nx"], case["ny"], case["pitch"], case["pitch"], case["wavelength"], case["z"], cwo.FRESNEL_FOURIER)
    plan.reserve(case["batch"])
    return {"case": case, "plan": plan, "x": _fields(case, seed, case["batch"])}


def run(state):
    case, k = state["case"], state["case"]["kind"]
    if k in ("asm", "fresnel"):
        plan, x = state["plan"], state["x"]
        if x.dim() == 2 and state["z"] is None:
            return plan.adjoint(x) if case["adjoint"] else plan.propagate(x)
        return plan.propagate_batch(x, z=state["z"], adjoint=case["adjoint"])
    if k == "stack":
        return state["plan"].propagate_stack(state["x"], state["zs"])
    if k == "items":
        return state["plan"].propagate_items(state["x"], state["items"])
    if k == "gs":
        field = state["field"].clone()
        intensity = state["plan"].gs_run(state["amp"], field, case["iterations"])
        return {"kinoform": field, "intensity": intensity}
    if k == "hologram":
        phi = state["phi"]
        phi.grad = None
        loss = state["problem"].loss(phi)
        loss.backward()
        return {"loss": loss.detach(), "grad": phi.grad}
    return state["plan"].propagate_batch(state["x"])


# ---------------------------------------------------------------------------------- their work
def _fft_flops(n):
    return 5.0 * n * math.log2(n)


def work(case):
    """Each input read and each output written once; the transforms of the padded method with the
    zero rows left out, 5 n log2 n operations for one of length n, and the products between them."""
    k = case["kind"]
    nx = case.get("nx") or case.get("n") or case["canvas"]
    ny = case.get("ny") or nx
    n, px, py = nx * ny, 2 * nx, 2 * ny
    asm = 2 * ny * _fft_flops(px) + 2 * px * _fft_flops(py) + 6 * px * py
    sep = 2 * ny * _fft_flops(px) + 2 * nx * _fft_flops(py) + 6 * (ny * px + nx * py)
    if k in ("asm", "shifted_asm"):
        return {"bytes": 16.0 * n * case["batch"], "flops": asm * case["batch"]}
    if k in ("fresnel", "shifted_fresnel"):
        return {"bytes": 16.0 * n * case["batch"], "flops": sep * case["batch"]}
    if k == "fourier":
        return {"bytes": 16.0 * n * case["batch"], "flops": (ny * _fft_flops(nx) + nx * _fft_flops(ny) + 12 * n) * case["batch"]}
    if k == "stack":   # the source's rows are transformed once
        j = case["planes"]
        return {"bytes": 8.0 * n * (1 + j), "flops": sep * j - (j - 1) * ny * _fft_flops(px)}
    if k == "items":
        fr = case["batch"] - round(case["batch"] * (1.0 - case["fresnel_share"]))
        return {"bytes": 16.0 * n * case["batch"], "flops": asm * (case["batch"] - fr) + sep * fr}
    if k == "gs":      # field and amplitude in, kinoform and intensity out; 2 propagations an iteration and 2 more
        return {"bytes": 24.0 * n, "flops": asm * (2 * case["iterations"] + 2)}
    m = case["h"] * case["w"]   # phase and target in, gradient out; a propagation and its adjoint
    return {"bytes": 12.0 * m, "flops": 2 * asm}


# ---------------------------------------------------------------------------------- in 64 bits
def _cis(cycles):
    """exp(2 pi i cycles), the whole cycles taken off first"""
    ph = TWO_PI * (cycles - torch.floor(cycles))
    return torch.complex(torch.cos(ph), torch.sin(ph))


def _f64(n):
    return torch.arange(n, dtype=torch.float64, device=DEVICE)


def _freq(p, pitch):
    return torch.fft.fftfreq(p, pitch, dtype=torch.float64, device=DEVICE)


def _asm_transfer(nx, ny, pitch, wavelength, z):
    fx, fy = _freq(2 * nx, pitch), _freq(2 * ny, pitch)
    r = 1.0 / wavelength ** 2 - fx[None, :] ** 2 - fy[:, None] ** 2
    h = _cis(z * torch.sqrt(torch.clamp(r, min=0.0)))
    return torch.where(r >= 0, h, torch.zeros_like(h))


def _chirp_axis(n, s):
    """the transform of exp(i pi s d^2) on the padded axis"""
    d = _f64(2 * n)
    d = torch.where(d < n, d, d - 2 * n)
    return torch.fft.fft(_cis(0.5 * s * d * d))


def _coefficient(pitch, wavelength, z):
    ph = TWO_PI * math.fmod(z / wavelength, 1.0)
    return complex(math.cos(ph), math.sin(ph)) / (1j * wavelength * z) * pitch * pitch


def _fresnel_transfer(nx, ny, pitch, wavelength, z):
    s = pitch * pitch / (wavelength * z)
    return _coefficient(pitch, wavelength, z) * _chirp_axis(ny, s)[:, None] * _chirp_axis(nx, s)[None, :]


def _padded(u, h, adjoint=False):
    ny, nx = u.shape[-2:]
    s = torch.fft.fft2(u.to(torch.complex128), s=(2 * ny, 2 * nx))
    s *= h.conj() if adjoint else h
    return torch.fft.ifft2(s)[..., :ny, :nx].contiguous()


def _unit(w):
    a = w.abs()
    return torch.where(a > 0, w / torch.where(a > 0, a, torch.ones_like(a)), torch.ones_like(w))


def exact(case, seed):
    k = case["kind"]
    if k == "gs":
        amp, field = _gs_inputs(case, seed)
        n = case["n"]
        h = _asm_transfer(n, n, case["pitch"], case["wavelength"], case["z"])
        a, u = amp.double(), _unit(_padded(field, h))
        for _ in range(case["iterations"]):
            u = _unit(_padded(a * _unit(_padded(u, h, True)), h))
        return {"kinoform": u, "intensity": _padded(u, h, True).abs() ** 2}
    if k == "hologram":
        phi, target = _hologram_inputs(case, seed)
        phi = phi.double().requires_grad_(True)
        c, hh, ww = case["canvas"], case["h"], case["w"]
        h = _asm_transfer(c, c, case["pitch"], case["wavelength"], case["z"])
        oy, ox = (c - hh) // 2, (c - ww) // 2
        pad = torch.nn.functional.pad(torch.polar(torch.ones_like(phi), phi), (ox, c - ww - ox, oy, c - hh - oy))
        u = torch.fft.ifft2(torch.fft.fft2(pad, s=(2 * c, 2 * c)) * h)[oy:oy + hh, ox:ox + ww]
        loss = ((u.real ** 2 + u.imag ** 2 - target.double()) ** 2).mean()
        loss.backward()
        return {"loss": loss.detach(), "grad": phi.grad}
    nx, ny = case["nx"], case["ny"]
    if k == "items":
        x = _fields(case, seed, case["batch"])
        out = []
        for u, it in zip(x, _items(case, seed)):
            f = _asm_transfer if it["type"] == cwo.ANGULAR else _fresnel_transfer
            out.append(_padded(u, f(nx, ny, it["dx"], it["wavelength"], it["z"])))
        return torch.stack(out)
    g = (nx, ny, case["pitch"], case["wavelength"])
    if k == "stack":
        u = _fields(case, seed, 1)[0]
        return torch.stack([_padded(u, _fresnel_transfer(*g, z)) for z in _plane_distances(case)])
    x = _fields(case, seed, case["batch"])
    if k in ("asm", "fresnel"):
        zs = _distances(case) if k == "asm" else None
        f = _asm_transfer if k == "asm" else _fresnel_transfer
        h = None if zs else f(*g, case["z"])
        y = torch.stack([_padded(u, f(*g, zs[i]) if zs else h, case["adjoint"]) for i, u in enumerate(x)])
        return y[0] if case["batch"] == 1 and zs is None else y
    z, lam, dx = case["z"], case["wavelength"], case["pitch"]
    if k == "shifted_asm":
        fx, fy = _freq(2 * nx, dx), _freq(2 * ny, dx)
        h = _asm_transfer(*g, z) * _cis(case["ox"] * fx)[None, :] * _cis(case["oy"] * fy)[:, None]
        if case["band_limited"]:
            lx, ly = (1.0 / (lam * math.sqrt((2.0 * z / (2 * n * dx)) ** 2 + 1.0)) for n in (nx, ny))
            h = h * (fx.abs() <= lx)[None, :] * (fy.abs() <= ly)[:, None]
        return torch.stack([_padded(u, h) for u in x])
    if k == "shifted_fresnel":
        p1, lz = case["pitch1"], lam * z
        s = dx * p1 / lz

        def axis(n, o1):   # source factor, destination factor, transform of the kernel
            m = _f64(n) - n // 2
            chirp = 0.5 * s * m * m
            x0, x1 = m * dx, m * p1 + o1
            return _cis(x0 * x0 / (2 * lz) - m * dx * o1 / lz - chirp), _cis(x1 * x1 / (2 * lz) - chirp), _chirp_axis(n, s)

        fx, qx, hx = axis(nx, case["ox1"])
        fy, qy, hy = axis(ny, case["oy1"])
        c = _coefficient(dx, lam, z)
        h = hy[:, None] * hx[None, :]
        return torch.stack([c * _padded(u * fy[:, None] * fx[None, :], h) * qy[:, None] * qx[None, :] for u in x])
    # the Fourier form: one unpadded transform between two chirps, both planes centred
    lz = lam * z

    def centred(n, step):
        r = (_f64(n) - n // 2) * step
        return _cis(r * r / (2.0 * lz))

    pre = centred(ny, dx)[:, None] * centred(nx, dx)[None, :]
    post = centred(ny, lz / (ny * dx))[:, None] * centred(nx, lz / (nx * dx))[None, :] * _coefficient(dx, lam, z)
    dims = (-2, -1)
    return torch.stack([post * torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(u * pre, dim=dims)), dim=dims) for u in x])
