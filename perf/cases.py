"""Measured workloads of the propagation library, through the calls its users make.

A case is a dict of plain values. Six kinds cover the library's use:

  propagate  a batch of fields propagated by one call (optionally also back-propagated)
  train      autograd.propagate behind a phase mask: forward, and gradients of field and mask
  focal      one field propagated to several distances (focal stack, method chosen per distance)
  intensity  polychromatic detector intensity, its loss, and the backward to the fields
  stack      a diffractive network: forward, loss, gradients of every phase mask
  fourf      the polarised polychromatic 4f imaging step with a trainable pupil phase
  ragged     fields of different sizes, spacings, wavelengths and distances in one call
  coherence  mutual coherence through a trainable mask: intensity and mask gradient
"""
from __future__ import annotations

import math

import torch

from paper_2411_18591_gb300 import autograd as A
from paper_2411_18591_gb300 import binding as B
from paper_2411_18591_gb300.fourf import FourF
from paper_2411_18591_gb300.stack import MaskStack


def listed():
    return [
        # one Gaussian beam on a small grid, as a user explores a design: all latency
        dict(name="beam_64", kind="propagate", ny=64, nx=64, batch=1, pad=2.0, method="as", d=10e-6, lam=700e-9,
             z=0.1, backward=False),
        # one field at the usual camera size, as in an interactive session or an outer Python loop
        dict(name="single_1024", kind="propagate", ny=1024, nx=1024, batch=1, pad=2.0, method="as", d=5e-6,
             lam=532e-9, z=0.2, backward=False),
        # a batch of them with its adjoint: the unit of the throughput figure
        dict(name="batch_1024", kind="propagate", ny=1024, nx=1024, batch=16, pad=2.0, method="as", d=5e-6,
             lam=532e-9, z=0.2, backward=True),
        # one large hologram, forward and adjoint
        dict(name="field_4096", kind="propagate", ny=4096, nx=4096, batch=1, pad=2.0, method="as", d=4e-6,
             lam=633e-9, z=0.1, backward=True),
        # a small hologram optimised through torch.autograd: short launches, host latency counts
        dict(name="train_256", kind="train", ny=256, nx=256, batch=8, pad=2.0, method="as", d=8e-6, lam=633e-9,
             z=0.02),
        # an odd (prime) size cut from measured data: no mixed-radix plan
        dict(name="train_1021", kind="train", ny=1021, nx=1021, batch=4, pad=2.0, method="as", d=5e-6, lam=532e-9,
             z=0.1),
        # one non-square field to eight distances on both sides of the critical one (AS and DI)
        dict(name="focal_768x1024", kind="focal", ny=768, nx=1024, repeat=8, pad=2.0, d=6e-6, lam=633e-9,
             z0=0.01, z1=0.09),
        # RGB detector images without padding, Fresnel transfer function
        dict(name="rgb_512_pad1", kind="intensity", ny=512, nx=512, objects=16, waves=3, pad=1.0, method="fresnel",
             d=8e-6, z=0.05),
        # diffractive network of five trainable 512 x 512 masks, batch 64
        dict(name="stack_5x512", kind="stack", n=512, batch=64, layers=5, d=8e-6, lam=532e-9, z=0.05),
        # polarised 4f imaging: 16 objects x 3 components x 8 wavelengths at 1024 x 1024
        dict(name="fourf_1024", kind="fourf", n=1024, objects=16, comps=3, waves=8, d=5e-6, f=0.2),
        # 200 fields of six sizes (side, spacing, wavelength and distance drawn per field), forward and adjoint in one call each
        dict(name="ragged_200", kind="ragged", count=200, sizes="250,256,500,512,768,1000", layout=3),
        # Gaussian Schell-model coherence on a 64 x 64 grid through a trainable mask
        dict(name="coherence_64", kind="coherence", n=64, d=10e-6, lam=633e-9, z=0.2),
    ]


# Grid sides a user picks: powers of two, round decimals, and sides cut from measured data.
SIDES = [64, 100, 128, 200, 250, 256, 320, 384, 500, 509, 512, 640, 768, 1000, 1021, 1024, 1500, 2000, 2048, 4096]


def draw(rng):
    kind = rng.choice(["propagate", "propagate", "train", "train", "focal", "intensity", "stack", "fourf", "ragged",
                       "coherence"])
    side = lambda lo, hi: rng.choice([s for s in SIDES if lo <= s <= hi])
    logint = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    um = lambda lo, hi: round(rng.uniform(lo, hi), 2) * 1e-6
    lam = round(rng.uniform(450.0, 700.0), 1) * 1e-9
    z = round(rng.uniform(0.01, 0.3), 4)
    if kind in ("propagate", "train"):
        big = 4096 if kind == "propagate" else 1024
        ny, nx = side(64, big), side(64, big)
        if rng.random() < 0.6:
            nx = ny
        batch = max(1, min(logint(1, 128), (24 << 20) // (ny * nx)))
        case = dict(kind=kind, ny=ny, nx=nx, batch=batch, pad=2.0, d=um(4, 12), lam=lam, z=z,
                    method=rng.choice(["as", "as", "fresnel"]))
        if kind == "propagate":
            case["backward"] = rng.random() < 0.5
        return case
    if kind == "focal":
        return dict(kind=kind, ny=side(128, 1024), nx=side(128, 1024), repeat=rng.randint(2, 12), pad=2.0, d=um(4, 10),
                    lam=lam, z0=0.01, z1=round(rng.uniform(0.05, 0.2), 3))
    if kind == "intensity":
        n = rng.choice([64, 128, 256, 500, 512, 1000, 1024])
        waves = rng.choice([1, 3, 3, 5])
        return dict(kind=kind, ny=n, nx=n, objects=max(1, min(logint(1, 64), (24 << 20) // (n * n * waves))), waves=waves,
                    pad=rng.choice([1.0, 1.0, 2.0]), method=rng.choice(["as", "fresnel"]), d=um(4, 12), z=z)
    if kind == "stack":
        n = rng.choice([128, 200, 250, 256, 500, 512, 1024])
        return dict(kind=kind, n=n, batch=max(1, min(logint(4, 128), (16 << 20) // (n * n))), layers=rng.randint(2, 6),
                    d=8e-6, lam=lam, z=0.05)
    if kind == "fourf":
        n = rng.choice([256, 500, 512, 768, 1000, 1024])
        return dict(kind=kind, n=n, objects=rng.randint(1, 8), comps=rng.choice([1, 3]), waves=rng.randint(1, 8),
                    d=um(5, 8), f=0.2)
    if kind == "ragged":
        sizes = rng.sample([64, 128, 250, 256, 384, 500, 512, 640, 768, 1000, 1024], rng.randint(3, 6))
        return dict(kind=kind, count=logint(6, 200), sizes=",".join(str(s) for s in sorted(sizes)),
                    layout=rng.randint(0, 999))
    return dict(kind=kind, n=rng.choice([16, 24, 32, 48, 64]), d=10e-6, lam=lam, z=z)


# ----------------------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32) * (hi - lo) + lo


def _coords(n, d):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1) / 2) * d


def _screen(g, ny, nx, sigma=4.0):
    """A smooth random phase screen: white noise filtered by a Gaussian of sigma pixels, std 1 rad."""
    noise = torch.randn((ny, nx), generator=g, device="cuda", dtype=torch.float32)
    fy = torch.fft.fftfreq(ny, device="cuda")[:, None]
    fx = torch.fft.rfftfreq(nx, device="cuda")[None, :]
    s = torch.fft.irfft2(torch.fft.rfft2(noise) * torch.exp(-2 * (math.pi * sigma) ** 2 * (fy * fy + fx * fx)),
                         s=(ny, nx))
    return s / s.std()


def _polar(amplitude, phase):
    return torch.polar(amplitude, phase).contiguous()


def _beam(ny, nx, d, waist):
    y, x = _coords(ny, d)[:, None], _coords(nx, d)[None, :]
    return torch.exp(-(x * x + y * y) / (waist * waist)).to(torch.float32)


def _waves(k):
    return [450e-9 + 250e-9 * i / max(1, k - 1) for i in range(k)]


def _fields(g, case, batch):
    """Gaussian beams through independent smooth phase screens (a plain beam when there is one)."""
    ny, nx, d = case["ny"], case["nx"], case["d"]
    if batch == 1:
        return _beam(ny, nx, d, 0.08 * nx * d).to(torch.complex64)[None] * _polar(
            torch.ones(ny, nx, device="cuda"), 0.2 * _screen(g, ny, nx))
    amp = _beam(ny, nx, d, 0.3 * nx * d)
    return torch.stack([_polar(amp, _screen(g, ny, nx)) for _ in range(batch)])


def _zs(case):
    k = case["repeat"]
    return [case["z0"] + (case["z1"] - case["z0"]) * i / max(1, k - 1) for i in range(k)]


def _fourf(case):
    n, d = case["n"], case["d"]
    return FourF(n=n, d=d, f=case["f"], lens_radius=0.5003 * n * d, pupil_radius=0.1953 * n * d,
                 objects=case["objects"], comps=case["comps"], wavelengths=tuple(_waves(case["waves"])))


def _ragged_parameters(case):
    sizes = [int(s) for s in case["sizes"].split(",")]
    u = torch.rand((case["count"], 4), generator=torch.Generator().manual_seed(case["layout"]), dtype=torch.float64).tolist()
    ns = [sizes[min(len(sizes) - 1, int(r[0] * len(sizes)))] for r in u]
    return (ns, [(4 + 8 * r[1]) * 1e-6 for r in u], [(450 + 250 * r[2]) * 1e-9 for r in u],
            [0.01 + 0.49 * r[3] for r in u])


def _planes(flat, ns):
    return [v.view(n, n) for v, n in zip(flat.split([n * n for n in ns]), ns)]


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "propagate":
        s["x"] = _fields(g, case, case["batch"])
        if case["backward"]:
            s["g"] = torch.randn(s["x"].shape, generator=g, device="cuda", dtype=torch.complex64)
    elif kind == "train":
        s["x"] = _fields(g, case, case["batch"]).requires_grad_()
        s["phase"] = _uniform(g, (case["ny"], case["nx"]), -math.pi, math.pi).requires_grad_()
        s["g"] = torch.randn(s["x"].shape, generator=g, device="cuda", dtype=torch.complex64)
    elif kind == "focal":
        s["x"] = _fields(g, case, 1)
    elif kind == "intensity":
        shape = (case["objects"], case["ny"], case["nx"])
        s["x"] = _polar(_uniform(g, shape, 0.0, 1.0), _uniform(g, shape, -0.5, 0.5))
        s["target"] = _uniform(g, shape, 0.0, 0.5 * case["waves"])
        s["weights"] = torch.tensor([1.0 / (1 + i) for i in range(case["waves"])] * case["objects"], device="cuda")
    elif kind == "stack":
        n, b = case["n"], case["batch"]
        s["x"] = (torch.rand((b, n, n), generator=g, device="cuda") < 0.5).to(torch.complex64)
        s["phases"] = _uniform(g, (case["layers"], n, n), 0.0, 2 * math.pi)
        s["target"] = _uniform(g, (b, n, n), 0.0, 0.5)
        s["net"] = MaskStack(case["d"], case["lam"], [case["z"]] * case["layers"])
    elif kind == "fourf":
        n = case["n"]
        s["x"] = _uniform(g, (case["objects"] * case["comps"], n, n), 0.0, 1.0).to(torch.complex64)
        s["phase"] = _uniform(g, (n, n), -math.pi, math.pi)
        s["target"] = _uniform(g, (case["objects"], n, n), 0.0, 0.5)
        s["system"], s["buffers"] = _fourf(case), {}
    elif kind == "ragged":
        ns, s["d"], s["lam"], s["z"] = _ragged_parameters(case)
        s["x"] = [_polar(torch.ones(n, n, device="cuda"), _screen(g, n, n)) for n in ns]
        s["g"] = [torch.randn((n, n), generator=g, device="cuda", dtype=torch.complex64) for n in ns]
        # results go to buffers that the program keeps, one for each direction, field after field
        s["out"] = torch.zeros(sum(n * n for n in ns), device="cuda", dtype=torch.complex64)
        s["back"] = torch.zeros_like(s["out"])
        s["out_fields"], s["back_fields"] = _planes(s["out"], ns), _planes(s["back"], ns)
    else:
        n, d = case["n"], case["d"]
        w, l = 200e-6 * n / 64, 50e-6
        y = _coords(n, d)
        r2 = (y[:, None] ** 2 + y[None, :] ** 2).reshape(-1)
        diff = (y[:, None] - y[None, :]) ** 2
        sep = (diff[:, None, :, None] + diff[None, :, None, :]).reshape(n * n, n * n)
        gamma = torch.exp(-(r2[:, None] + r2[None, :]) / (w * w) - sep / (2 * l * l))
        s["x"] = gamma.to(torch.complex64).reshape(n, n, n, n)
        s["phase"] = _uniform(g, (n, n), -math.pi, math.pi)
        s["gi"] = _uniform(g, (n, n), -1.0, 1.0)
    return s


# ----------------------------------------------------------------------------- one pass

def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "propagate":
        out = B.top_propagate(state["x"], c["d"], c["d"], c["lam"], c["z"], c["pad"], c["method"])
        if not c["backward"]:
            return out
        return out, B.top_propagate_backward(state["g"], c["d"], c["d"], c["lam"], c["z"], c["pad"], c["method"])
    if kind == "train":
        out = A.propagate(state["x"], c["d"], c["d"], c["lam"], c["z"], c["pad"], c["method"], phase=state["phase"])
        gx, gp = torch.autograd.grad(out, (state["x"], state["phase"]), state["g"])
        return out.detach(), gx, gp
    if kind == "focal":
        return B.top_propagate(state["x"], c["d"], c["d"], c["lam"], _zs(c), c["pad"], "auto", input_repeat=c["repeat"])
    if kind == "intensity":
        lam = _waves(c["waves"]) * c["objects"]
        inten, field = B.top_propagate_intensity(state["x"], c["d"], c["d"], lam, c["z"], c["pad"], c["method"],
                                                 group=c["waves"], weights=state["weights"], keep_field=True,
                                                 input_repeat=c["waves"])
        loss, gi = B.top_mse_loss(inten, state["target"])
        gx = B.top_propagate_intensity_backward(field, gi, c["d"], c["d"], lam, c["z"], c["pad"], c["method"],
                                                group=c["waves"], weights=state["weights"])
        return loss, inten, field, gx
    if kind == "stack":
        net = state["net"]
        inten, kept = net.forward(state["x"], state["phases"])
        loss, gi = B.top_mse_loss(inten, state["target"])
        grads, _ = net.backward(kept, state["phases"], gi)
        return loss, inten, grads
    if kind == "fourf":
        grad = torch.empty_like(state["phase"])
        loss, inten = state["system"].step(state["x"], state["phase"], state["target"], grad, state["buffers"])
        return loss, inten, grad
    if kind == "ragged":
        B.top_propagate_ragged(state["x"], state["d"], state["lam"], state["z"], out=state["out_fields"])
        B.top_propagate_ragged(state["g"], state["d"], state["lam"], state["z"], backward=True, out=state["back_fields"])
        return state["out"], state["back"]
    mask = B.Modulation(phase=state["phase"])
    gamma = B.top_propagate_coherence(state["x"], c["d"], c["d"], c["lam"], c["z"], mask=mask)
    inten = B.top_coherence_intensity(gamma)
    g_gamma = B.top_coherence_intensity_backward(state["gi"], gamma)
    gp = torch.zeros_like(state["phase"])
    gx = B.top_propagate_coherence_backward(g_gamma, c["d"], c["d"], c["lam"], c["z"], mask=mask, saved_in=state["x"],
                                            grad_phase=gp)
    return gamma, inten, gx, gp


# ----------------------------------------------------------------------------- work

def _padded(n, pad):
    return int(math.floor(pad * n + 0.5))


def _prop_flops(ny, nx, pad):
    """One propagation: row transforms of the ny field rows and column transforms of every padded
    column, there and back, and the product with the transfer function."""
    py, px = _padded(ny, pad), _padded(nx, pad)
    return 2 * (5 * ny * px * math.log2(px) + 5 * px * py * math.log2(py)) + 6 * py * px


def work(case):
    kind = case["kind"]
    if kind in ("propagate", "train", "focal", "intensity"):
        plane, one = case["ny"] * case["nx"], _prop_flops(case["ny"], case["nx"], case["pad"])
    if kind == "propagate":
        n = 2 if case["backward"] else 1
        return {"bytes": 16 * n * case["batch"] * plane, "flops": n * case["batch"] * one}
    if kind == "train":  # field, upstream gradient, output, field gradient; mask and its gradient
        return {"bytes": 32 * case["batch"] * plane + 8 * plane, "flops": 2 * case["batch"] * one}
    if kind == "focal":
        return {"bytes": 8 * plane * (1 + case["repeat"]), "flops": case["repeat"] * one}
    if kind == "intensity":
        fields = case["objects"] * case["waves"]
        return {"bytes": plane * (case["objects"] * (8 + 4 + 4) + fields * 16), "flops": 2 * fields * one}
    if kind == "stack":
        plane, one = case["n"] ** 2, _prop_flops(case["n"], case["n"], 2.0)
        return {"bytes": plane * (case["batch"] * (8 + 4 + 4) + case["layers"] * 8),
                "flops": 2 * case["layers"] * case["batch"] * one}
    if kind == "fourf":
        plane, one = case["n"] ** 2, _prop_flops(case["n"], case["n"], 2.0)
        fields = case["objects"] * case["comps"]
        return {"bytes": plane * (fields * 8 + case["objects"] * 8 + 8), "flops": 6 * fields * case["waves"] * one}
    if kind == "ragged":
        sizes = [int(s) for s in case["sizes"].split(",")]
        mean = lambda f: sum(f(n) for n in sizes) / len(sizes)
        return {"bytes": int(32 * case["count"] * mean(lambda n: n * n)),
                "flops": 2 * case["count"] * mean(lambda n: _prop_flops(n, n, 2.0))}
    n = case["n"]
    return {"bytes": 8 * 3 * n ** 4 + 16 * n * n, "flops": 4 * n * n * _prop_flops(n, n, 2.0)}


# ----------------------------------------------------------------------------- exact results (64 bits)

def _transfer(py, px, d, lam, z, method):
    fy = torch.fft.fftfreq(py, d, dtype=torch.float64, device="cuda")[:, None]
    fx = torch.fft.fftfreq(px, d, dtype=torch.float64, device="cuda")[None, :]
    if method == "as":
        rad = 1 / (lam * lam) - fx * fx - fy * fy
        turns = z * torch.sqrt(rad.clamp(min=0))
        keep = (rad >= 0).to(torch.float64)
    else:
        turns = z / lam - 0.5 * lam * z * (fx * fx + fy * fy)
        keep = torch.ones_like(turns)
    return torch.polar(keep, 2 * math.pi * (turns - torch.round(turns)))


def _direct_transfer(py, px, d, lam, z):
    """Transform of the Rayleigh-Sommerfeld kernel sampled at the signed lags of the padded grid."""
    y = torch.fft.fftfreq(py, 1.0 / py, dtype=torch.float64, device="cuda")[:, None] * d
    x = torch.fft.fftfreq(px, 1.0 / px, dtype=torch.float64, device="cuda")[None, :] * d
    r = torch.sqrt(x * x + y * y + z * z)
    k = 2 * math.pi / lam
    turns = r / lam
    h = torch.complex(1 / r, torch.full_like(r, -k)) * torch.polar(z / (2 * math.pi * r * r),
                                                                   2 * math.pi * (turns - torch.round(turns)))
    return torch.fft.fft2(h) * (d * d)


def _prop64(x, h, ny, nx):
    """Zero-padded propagation of complex128 fields [..., ny, nx] with transfer function h [..., py, px]."""
    py, px = h.shape[-2:]
    oy, ox = (py - ny) // 2, (px - nx) // 2
    padded = torch.nn.functional.pad(x, (ox, px - nx - ox, oy, py - ny - oy))
    return torch.fft.ifft2(torch.fft.fft2(padded) * h)[..., oy:oy + ny, ox:ox + nx]


def _each(x, f):
    return torch.cat([f(x[i:i + 1]) for i in range(x.shape[0])])


def _mask64(phase):
    p = phase.to(torch.float64)
    return torch.polar(torch.ones_like(p), p)


def exact(case, seed):
    kind = case["kind"]
    s = prepare(case, seed)
    pad_h = lambda lam, z, method="as", d=None, n=None: _transfer(
        _padded(n or case["ny"], case.get("pad", 2.0)), _padded(n or case["nx"], case.get("pad", 2.0)),
        d or case["d"], lam, z, method)
    with torch.no_grad():
        if kind == "propagate":
            ny, nx = case["ny"], case["nx"]
            h = pad_h(case["lam"], case["z"], case["method"])
            fwd = _each(s["x"], lambda v: _prop64(v.to(torch.complex128), h, ny, nx))
            if not case["backward"]:
                return fwd
            return fwd, _each(s["g"], lambda v: _prop64(v.to(torch.complex128), h.conj(), ny, nx))
        if kind == "train":
            ny, nx = case["ny"], case["nx"]
            h = pad_h(case["lam"], case["z"], case["method"])
            m = _mask64(s["phase"])
            out = _each(s["x"], lambda v: _prop64(v.to(torch.complex128) * m, h, ny, nx))
            gy = _each(s["g"], lambda v: _prop64(v.to(torch.complex128), h.conj(), ny, nx))
            return out, gy * m.conj(), (gy * (m * s["x"].to(torch.complex128)).conj()).imag.sum(0)
        if kind == "focal":
            ny, nx, d, lam = case["ny"], case["nx"], case["d"], case["lam"]
            py, px = _padded(ny, case["pad"]), _padded(nx, case["pad"])
            crit = min(ny, nx) * d * d / lam
            return torch.cat([_prop64(s["x"].to(torch.complex128), _transfer(py, px, d, lam, z, "as") if z < crit
                                      else _direct_transfer(py, px, d, lam, z), ny, nx) for z in _zs(case)])
        if kind == "intensity":
            ny, nx, k = case["ny"], case["nx"], case["waves"]
            hs = torch.stack([pad_h(lam, case["z"], case["method"]) for lam in _waves(k)])
            w = s["weights"][:k].to(torch.float64)[:, None, None]
            field = torch.cat([_prop64(v.to(torch.complex128)[None], hs, ny, nx) for v in s["x"]])
            per = field.reshape(-1, k, ny, nx)
            inten = (w * per.abs() ** 2).sum(1)
            diff = inten - s["target"].to(torch.float64)
            src = 2 * w * (2 * diff / diff.numel())[:, None] * per
            return (diff ** 2).mean(), inten, field, torch.cat([_prop64(v, hs.conj(), ny, nx) for v in src])
        if kind == "ragged":
            out, back = [], []
            for x, g, d, lam, z in zip(s["x"], s["g"], s["d"], s["lam"], s["z"]):
                n = x.shape[-1]
                h = pad_h(lam, z, d=d, n=n)
                out.append(_prop64(x.to(torch.complex128), h, n, n).flatten())
                back.append(_prop64(g.to(torch.complex128), h.conj(), n, n).flatten())
            return torch.cat(out), torch.cat(back)
        if kind == "stack":
            n, K = case["n"], case["layers"]
            h = pad_h(case["lam"], case["z"], n=n)
            masks = _mask64(s["phases"])
            intens, total = [], torch.zeros((), dtype=torch.float64, device="cuda")
            grads = torch.zeros((K, n, n), dtype=torch.float64, device="cuda")
            for b in range(case["batch"]):
                modulated, x = [], s["x"][b].to(torch.complex128)
                for m in masks:
                    modulated.append(x * m)
                    x = _prop64(modulated[-1], h, n, n)
                intens.append(x.abs() ** 2)
                diff = intens[-1] - s["target"][b].to(torch.float64)
                total += (diff ** 2).sum()
                g = 4 * diff / (case["batch"] * n * n) * x
                for k in range(K - 1, -1, -1):
                    gy = _prop64(g, h.conj(), n, n)
                    grads[k] += (gy * modulated[k].conj()).imag
                    g = gy * masks[k].conj()
            return total / (case["batch"] * n * n), torch.stack(intens), grads
        if kind == "fourf":
            sy = s["system"]
            n, d, count = sy.n, sy.d, sy.objects * sy.n * sy.n
            r2 = _coords(n, d)[:, None] ** 2 + _coords(n, d)[None, :] ** 2
            lam = torch.tensor(sy.wavelengths, dtype=torch.float64, device="cuda")[:, None, None]
            turns = -r2 / (2 * lam * sy.f)
            lens = torch.polar((r2 <= sy.lens_radius ** 2).to(torch.float64).expand_as(turns),
                               2 * math.pi * (turns - torch.round(turns)))
            pupil = _mask64(s["phase"]) * (r2 <= sy.pupil_radius ** 2)
            hs = torch.stack([pad_h(l, sy.f, n=n) for l in sy.wavelengths])
            step = lambda v: _prop64(v, hs, n, n)
            back = lambda v: _prop64(v, hs.conj(), n, n)
            grad = torch.zeros((n, n), dtype=torch.float64, device="cuda")
            intens, total = [], torch.zeros((), dtype=torch.float64, device="cuda")
            for o in range(sy.objects):
                at_pupil, image = [], []
                for c in range(sy.comps):
                    x = s["x"][o * sy.comps + c].to(torch.complex128)[None]
                    at_pupil.append(step(lens * step(x)) * pupil)
                    image.append(step(lens * step(at_pupil[-1])))
                intens.append(sum((v.abs() ** 2).sum(0) for v in image))
                diff = intens[-1] - s["target"][o].to(torch.float64)
                total += (diff ** 2).sum()
                for a, v in zip(at_pupil, image):
                    gy = back(lens.conj() * back(4 * diff / count * v))
                    grad += (gy * a.conj()).imag.sum(0)
            return total / count, torch.stack(intens), grad
        n = case["n"]
        h = pad_h(case["lam"], case["z"], n=n)
        m = _mask64(s["phase"]).reshape(-1)

        def both(t, ha, hb):  # ha on the second coordinate pair of t, then hb on the first
            plane = lambda v, hh: torch.cat([_prop64(p, hh, n, n) for p in v.reshape(-1, n, n).split(1024)])
            t = plane(t, ha).reshape(n * n, n * n).T.contiguous()
            return plane(t, hb).reshape(n * n, n * n).T.contiguous()

        x = s["x"].to(torch.complex128).reshape(n * n, n * n)
        masked = m[:, None] * x * m.conj()[None, :]
        # Gamma_z = P (M Gamma M^H) P^H: P over the first pair; over the second pair each row times P^H from
        # the right is the propagation with the conjugate of the (even) transfer function
        gamma = both(masked, h.conj(), h)
        inten = gamma.diagonal().real.reshape(n, n)
        g = both(torch.diag(s["gi"].to(torch.complex128).reshape(-1)), h, h.conj())
        gx = m.conj()[:, None] * g * m[None, :]
        # dL/dphi(r) = sum_s Im(g(r, s) conj(masked(r, s))) - sum_s Im(g(s, r) conj(masked(s, r)))
        t = (g * masked.conj()).imag
        return gamma.reshape(n, n, n, n), inten, gx.reshape(n, n, n, n), (t.sum(1) - t.sum(0)).reshape(n, n)
