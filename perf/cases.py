"""Performance cases of the framework: what a shear pipeline has it do, through its public entry points.

A pipeline draws model stamps (render), fits every galaxy by HMC (fit_galaxies, FitPlan, RaggedFitPlan; with per-pixel
weights or a dense pixel covariance where the noise asks for it), looks at the chains (chain_ess), optimises or checks
single points (RenderLogPost), and infers the shear from the interim samples (ShearPlan: one pass, its gradient through
autograd, the joint estimate, the likelihood with every property free).  Stamps, priors, sampler settings and noise
levels are those of the repository's workloads (bench.py) and tests.

Inputs are drawn and rendered here in 64-bit torch, never by the library, so that they do not depend on it; the 64-bit
values of exact() come from the same plain torch formulas.
"""
import math

import numpy as np
import torch

from paper_2604_22048_gb300 import api

DEV = "cuda"
PIX = float(np.float32(0.2))
HLR_R0 = 1.6783469900166608          # half-light radius of the exponential profile over its scale length
LF, LS, SXY, SE = (-1.0, 9.0), (-2.0, 1.0), 0.5, 0.3   # interim prior
KINDS = ("render", "points", "fit", "pixel", "dense", "ess", "pass", "estimate", "full")


# --------------------------------------------------------------------------- the cases

def listed():
    return [
        # simulated images for a fit: uneven stamps, a Moffat PSF and a shear per galaxy
        {"name": "render_ragged", "kind": "render", "n": 20000, "side": 0, "moffat": True, "shear": True},
        # log posterior and gradient at one point per galaxy: an optimiser's step through autograd
        {"name": "points_53", "kind": "points", "n": 4000, "per": 1, "side": 53, "moffat": False},
        # the smallest call: ten galaxies on FP64 stamps, fixed-length trajectories
        {"name": "fit_tiny", "kind": "fit", "n": 10, "side": 25, "moffat": False, "chains": 2, "warmup": 100,
         "samples": 200, "leapfrog": 8, "random": False, "f64": True, "plan": "call", "exposures": 1, "corr": False,
         "profile": 0},
        # the plain batch: one stamp size, one Gaussian PSF, the setting that meets the convergence bar
        {"name": "fit_plain_53", "kind": "fit", "n": 10000, "side": 53, "moffat": False, "chains": 4, "warmup": 200,
         "samples": 300, "leapfrog": 14, "random": True, "f64": False, "plan": "plan", "exposures": 1, "corr": False,
         "profile": 0},
        # the survey batch: stamps of 25-101 px, a Moffat PSF per galaxy, one captured launch plan
        {"name": "fit_ragged", "kind": "fit", "n": 10000, "side": 0, "moffat": True, "chains": 4, "warmup": 200,
         "samples": 300, "leapfrog": 14, "random": True, "f64": False, "plan": "ragged", "exposures": 1,
         "corr": False, "profile": 0},
        # spatially variable noise and masked pixels
        {"name": "fit_pixel_41", "kind": "pixel", "n": 400, "side": 41, "chains": 4, "warmup": 100, "samples": 100,
         "leapfrog": 16},
        # noise that is neither stationary nor diagonal: the precisions, then the fit
        {"name": "fit_dense_21", "kind": "dense", "n": 64, "side": 21, "chains": 4, "warmup": 100, "samples": 100,
         "leapfrog": 8},
        # convergence of the plain batch's chains
        {"name": "ess_plain", "kind": "ess", "n": 10000, "chains": 4, "samples": 300},
        # a small sample's shear likelihood and gradient through autograd: one optimiser step
        {"name": "shear_small", "kind": "pass", "n": 1000, "K": 100, "b": False, "weights": False, "family": 0,
         "autograd": True},
        # the survey's shear likelihood, asynchronous on the device
        {"name": "shear_large", "kind": "pass", "n": 1000000, "K": 300, "b": False, "weights": False, "family": 1,
         "autograd": False},
        # joint posterior mean of the shear and the ellipticity dispersion
        {"name": "shear_estimate", "kind": "estimate", "n": 50000, "K": 300, "free": True, "weights": False},
        # every property's prior free: one evaluation of the shear sampler
        {"name": "shear_full", "kind": "full", "n": 100000, "K": 300, "family": 1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, lo, hi):
    return 2 * rng.randint((lo - 1) // 2, (hi - 1) // 2) + 1


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "render":
        side = rng.choice((0, _odd(rng, 15, 101)))
        return {"kind": kind, "n": _log(rng, 10, 20000 if side <= 61 else 4000), "side": side,
                "moffat": rng.random() < 0.5, "shear": rng.random() < 0.5}
    if kind == "points":
        return {"kind": kind, "n": _log(rng, 1, 1000), "per": rng.randint(1, 4), "side": rng.choice((0, _odd(rng, 15, 75))),
                "moffat": rng.random() < 0.5}
    if kind == "fit":
        plan = rng.choice(("call", "plan", "ragged"))
        plain = plan == "ragged" or rng.random() < 0.5
        J = 1 if plain else rng.randint(1, 4)
        return {"kind": kind, "n": _log(rng, 3, 2000), "side": rng.choice((0, _odd(rng, 15, 101))),
                "moffat": rng.random() < 0.5, "chains": rng.randint(1, 6), "warmup": rng.choice((0, 20, 100, 200)),
                "samples": _log(rng, 50, 300), "leapfrog": rng.randint(4, 16), "random": rng.random() < 0.7,
                "f64": rng.random() < 0.3, "plan": plan, "exposures": J, "corr": not plain and rng.random() < 0.5,
                "profile": 0 if plain else rng.choice((0, 0, 1, 2))}
    if kind == "pixel":
        return {"kind": kind, "n": _log(rng, 10, 400), "side": _odd(rng, 15, 63), "chains": rng.randint(1, 4),
                "warmup": rng.choice((20, 100)), "samples": _log(rng, 30, 100), "leapfrog": rng.randint(4, 12)}
    if kind == "dense":
        return {"kind": kind, "n": _log(rng, 4, 64), "side": _odd(rng, 7, 21), "chains": rng.randint(1, 4),
                "warmup": rng.choice((20, 100)), "samples": _log(rng, 30, 100), "leapfrog": rng.randint(4, 8)}
    if kind == "ess":
        return {"kind": kind, "n": _log(rng, 10, 10000), "chains": rng.randint(1, 8), "samples": _log(rng, 50, 600)}
    n, K = _log(rng, 50, 200000), rng.choice((24, 99, 100, 250, 300, 1000, 1200))
    n = min(n, 60000000 // K)
    if kind == "pass":
        return {"kind": kind, "n": n, "K": K, "b": rng.random() < 0.3, "weights": rng.random() < 0.3,
                "family": rng.randint(0, 1), "autograd": rng.random() < 0.5}
    if kind == "estimate":
        return {"kind": kind, "n": max(500, min(n, 15000000 // K)), "K": K, "free": rng.random() < 0.5,
                "weights": rng.random() < 0.3}
    return {"kind": kind, "n": min(n, 30000000 // K), "K": K, "family": rng.randint(0, 1)}


def work(case):
    kind, n = case["kind"], case["n"]
    if kind in ("pass", "estimate", "full"):
        m = n * case["K"]
        if kind == "full":
            return {"bytes": 16.0 * m, "flops": 150.0 * m}
        if kind == "estimate":   # the quadrature's nodes and about four Newton steps with their central differences
            return {"bytes": 8.0 * m, "flops": 60.0 * m * ((7 ** 3 + 4 * 7) if case["free"] else (7 ** 2 + 4 * 5))}
        return {"bytes": (12.0 if case["b"] else 8.0) * m + 4.0 * n * case["weights"], "flops": 60.0 * m}
    if kind == "ess":
        d = n * case["chains"] * case["samples"]
        return {"bytes": 24.0 * d, "flops": 6.0 * d * (4 + 2 * 8)}   # moments, and about eight lags
    N = case["side"] or 53
    H = (N + 1) // 2
    if kind == "render":
        return {"bytes": 4.0 * n * N * N, "flops": n * (8.0 * H * N * N + 4.0 * H * N * N + 40.0 * H * N)}
    if kind == "points":
        return {"bytes": 4.0 * n * N * N, "flops": n * (12.0 * H * N * N + 40.0 * H * N + case["per"] * 33.0 * H * N)}
    evals = n * case["chains"] * (case["warmup"] + case["samples"]) * (case["leapfrog"] + 1) / 2
    out = 24.0 * n * case["chains"] * case["samples"]
    if kind == "fit":
        return {"bytes": case["exposures"] * 4.0 * n * N * N + out, "flops": evals * (33.0 * H * N + 9.0 * H)}
    if kind == "pixel":
        return {"bytes": 8.0 * n * N * N + out, "flops": evals * (24.0 * N * N * H + 33.0 * H * N)}
    return {"bytes": 8.0 * n * N ** 4 + out, "flops": 1.0 * n * N ** 6 + evals * 2.0 * N ** 4}


# --------------------------------------------------------------------------- the model in 64 bits

def _psf64(psf, k):
    """Transform of the PSFs (kind, fwhm [n]) at |k| [H, N] -> [n, H, N]."""
    kind, fwhm = psf
    if kind == "gaussian":
        return torch.exp(-0.5 * (k[None] * (fwhm / 2.3548200450309493)[:, None, None]) ** 2)
    x = k[None] * (fwhm / (2.0 * math.sqrt(2.0 ** (1.0 / 3.0) - 1.0)))[:, None, None]
    z = x.clamp_min(1e-30)
    k2 = torch.special.modified_bessel_k0(z) + 2.0 * torch.special.modified_bessel_k1(z) / z
    return torch.where(x > 0, 0.5 * z * z * k2, torch.ones_like(x))     # beta = 3


def _grid(N):
    c = (N - 1) // 2
    f = dict(dtype=torch.float64, device=DEV)
    u, v = torch.arange(c + 1, **f), torch.arange(-c, c + 1, **f)
    return c, u, v, 2.0 * math.pi / (N * PIX)


def _transfer64(N, psf):
    c, u, v, dk = _grid(N)
    k = dk * torch.sqrt(u[:, None] ** 2 + v[None, :] ** 2)
    return _psf64(psf, k) * (torch.sinc(u / N)[:, None] * torch.sinc(v / N)[None, :])[None]


def _image64(th, N, T):
    """Model stamps [n, N, N] of th [n, 6] on the transfer T [n, H, N]."""
    c, u, v, dk = _grid(N)
    F = 10.0 ** th[:, 0]
    r02 = (10.0 ** th[:, 1] / HLR_R0) ** 2
    e1, e2 = th[:, 2], th[:, 3]
    E = e1 * e1 + e2 * e2
    s = lambda x: x[:, None, None]
    kx, ky = (u * dk)[None, :, None], (v * dk)[None, None, :]
    q = s(1 + E + 2 * e1) * kx * kx + s(1 + E - 2 * e1) * ky * ky + s(4 * e2) * kx * ky
    amp = s(F) * T * (1.0 + s(r02 / (1 - E)) * q) ** -1.5
    ph = (-2.0 * math.pi / N) * (u[None, :, None] * s(th[:, 4]) + v[None, None, :] * s(th[:, 5]))
    y = torch.arange(N, dtype=torch.float64, device=DEV) - c
    ev, eu = (2.0 * math.pi / N) * v[:, None] * y[None, :], (2.0 * math.pi / N) * u[:, None] * y[None, :]
    w = torch.where(u > 0, 2.0, 1.0)[:, None] / (N * N)
    re, im = amp * torch.cos(ph), amp * torch.sin(ph)
    gr = re @ torch.cos(ev) - im @ torch.sin(ev)          # [n, u, iy]
    gi = re @ torch.sin(ev) + im @ torch.cos(ev)
    return gr.transpose(1, 2) @ (w * torch.cos(eu)) - gi.transpose(1, 2) @ (w * torch.sin(eu))


def _sheared(e1, e2, g1, g2):
    z = (torch.complex(e1, e2) + torch.complex(g1, g2)) / (1 + torch.complex(g1, -g2) * torch.complex(e1, e2))
    return z.real, z.imag


def _sides(case, hlr):
    if case["side"]:
        return torch.full((case["n"],), case["side"], dtype=torch.int32, device=DEV)
    half = torch.ceil(4.43 * hlr / 0.2 + 1.5 * 0.8 / 0.2)
    return (2 * half + 1).clamp(25, 101).to(torch.int32)


def _groups(side):
    """(N, indices) of the galaxies of each stamp side."""
    return [(int(N), torch.nonzero(side == N).squeeze(1)) for N in torch.unique(side).tolist()]


def _galaxies(case, gen, J=1):
    """True parameters, sides and PSF widths of the workloads' galaxies.  The catalogue's sizes, and with them the stamps
    that are cut, are those of the case; everything else comes from the seed."""
    n = case["n"]
    fixed = torch.Generator(device=DEV)
    fixed.manual_seed(2604)
    hlr = torch.exp(math.log(0.8) + 0.3 * torch.randn(n, dtype=torch.float64, device=DEV, generator=fixed))
    f = dict(dtype=torch.float64, device=DEV, generator=gen)
    e1, e2 = _ellipticities(n, gen, 0.2, 0.7)
    e1, e2 = _sheared(e1, e2, torch.full_like(e1, 0.02), torch.zeros_like(e1))
    off = torch.rand((n, 2), **f) - 0.5
    if case.get("moffat"):
        kind, fwhm = "moffat", (0.6 + 0.3 * torch.rand((n, J), **f)).float().double()
        snr = torch.exp(math.log(10.0) + math.log(10.0) * torch.rand(n, **f))
    else:
        kind, fwhm = "gaussian", torch.full((n, J), float(np.float32(0.7)), dtype=torch.float64, device=DEV)
        snr = 15.0 + 35.0 * torch.rand(n, **f)
    side = _sides(case, hlr)
    hlr = hlr * torch.exp(0.03 * torch.randn(n, **f))
    th = torch.stack([torch.zeros_like(hlr), torch.log10(hlr), e1, e2, off[:, 0], off[:, 1]], 1)
    return th, side, kind, fwhm, snr


def _ellipticities(n, gen, sigma, rmax):
    """Isotropic Gaussian ellipticities of width sigma inside |e| < rmax."""
    f = dict(dtype=torch.float64, device=DEV, generator=gen)
    r = sigma * torch.sqrt(-2.0 * torch.log1p(-torch.rand(n, **f) * (1.0 - math.exp(-0.5 * (rmax / sigma) ** 2))))
    a = 2.0 * math.pi * torch.rand(n, **f)
    return r * torch.cos(a), r * torch.sin(a)


def _psf_arg(kind, fwhm):
    flat = fwhm.reshape(-1)
    if kind == "gaussian":
        flat = flat[:1]          # one shared PSF
    return api.psf_table(kind, flat.cpu().numpy().astype(np.float32), 3.0, device=DEV)


def _pack(side, J=1):
    """Offsets of J stamps per galaxy, each galaxy's start a multiple of 4, and the total."""
    size = (J * side.long() ** 2 + 3) // 4 * 4
    off = torch.cumsum(size, 0) - size
    return off, int(size.sum())


# correlation of noise smoothed by (0.3, 1, 0.3) along each axis, as a rolled filter
TAPS = (0.3, 1.0, 0.3)


def _smooth(w):
    for d in (-1, -2):
        w = sum(t * torch.roll(w, i - 1, dims=d) for i, t in enumerate(TAPS))
    return w / sum(t * t for t in TAPS)


def _lag_corr(N):
    c1 = torch.zeros(N, dtype=torch.float64, device=DEV)
    c = (N - 1) // 2
    for lag in range(-2, 3):
        c1[c + lag] = sum(TAPS[i] * TAPS[i + lag] for i in range(3) if 0 <= i + lag < 3)
    return c1[:, None] * c1[None, :] / c1[c] ** 2


def _stamps(case, gen, th, side, kind, fwhm, snr, noise):
    """Packed noisy stamps (float64) of J exposures each, and the flux set from the S/N of the first."""
    J = fwhm.shape[1]
    off, total = _pack(side, J)
    data = torch.zeros(total, dtype=torch.float64, device=DEV)
    sums = torch.zeros(len(th), dtype=torch.float64, device=DEV)
    for N, idx in _groups(side):
        for j in range(J):
            unit = _image64(th[idx] * th.new_tensor([0, 1, 1, 1, 1, 1]), N, _transfer64(N, (kind, fwhm[idx, j])))
            if j == 0:
                th[idx, 0] = torch.log10(snr[idx] / torch.sqrt((unit ** 2).sum((1, 2))))
            img = unit * (10.0 ** th[idx, 0])[:, None, None] + noise(idx, N)
            at = (off[idx] + j * N * N)[:, None] + torch.arange(N * N, device=DEV)[None]
            data[at.reshape(-1)] = img.reshape(-1)
            if j == 0:
                sums[idx] = img.sum((1, 2))
    return data, off, sums


def _starts(gen, th, sums, chains):
    """Chain starts: the flux from the pixel sum, size and shape near the truth, the centre at zero."""
    n = len(th)
    f = dict(dtype=torch.float64, device=DEV, generator=gen)
    x = torch.zeros((n, chains, 6), dtype=torch.float64, device=DEV)
    x[..., 0] = torch.log10(sums.clamp_min(1.0))[:, None]
    x[..., 1] = th[:, None, 1] + 0.03 * (torch.rand((n, chains), **f) - 0.5)
    e = th[:, None, 2:4] + 0.2 * (torch.rand((n, chains, 2), **f) - 0.5)
    r = e.norm(dim=-1, keepdim=True)
    x[..., 2:4] = e * torch.where(r >= 0.95, 0.95 / r, torch.ones_like(r))
    return x.float().contiguous()


# --------------------------------------------------------------------------- inputs

def _config(case, **kw):
    return api.FitConfig(n_chains=case["chains"], n_warmup=case["warmup"], n_samples=case["samples"],
                         n_leapfrog=case["leapfrog"], random_steps=case.get("random", True), **kw)


def _prepare_render(case, gen):
    th, side, kind, fwhm, snr = _galaxies(case, gen)
    th[:, 0] = 2.0 + torch.rand(case["n"], dtype=torch.float64, device=DEV, generator=gen)
    shear = None
    if case["shear"]:
        shear = (0.1 * (torch.rand((case["n"], 2), dtype=torch.float64, device=DEV, generator=gen) - 0.5)).float()
    return {"theta": th.float(), "side": side, "psf": _psf_arg(kind, fwhm), "shear": shear, "kind": kind, "fwhm": fwhm}


def _prepare_points(case, gen):
    th, side, kind, fwhm, snr = _galaxies(case, gen)
    data, off, _ = _stamps(case, gen, th, side, kind, fwhm, snr, lambda idx, N: torch.randn(
        (len(idx), N, N), dtype=torch.float64, device=DEV, generator=gen))
    per = case["per"]
    gi = torch.arange(case["n"], dtype=torch.int32, device=DEV).repeat_interleave(per)
    step = th.new_tensor([0.02, 0.03, 0.05, 0.05, 0.2, 0.2])
    pts = th.repeat_interleave(per, 0) + step * torch.randn((len(gi), 6), dtype=torch.float64, device=DEV, generator=gen)
    pts[:, 2:4] *= (0.9 / pts[:, 2:4].norm(dim=1, keepdim=True)).clamp_max(1.0)
    return {"data": data.float(), "offsets": off, "side": side, "psf": _psf_arg(kind, fwhm), "gal": gi,
            "sigma": torch.ones(case["n"], device=DEV), "theta": pts.float(), "kind": kind, "fwhm": fwhm}


def _prepare_fit(case, gen):
    J = case["exposures"]
    th, side, kind, fwhm, snr = _galaxies(case, gen, J)

    def noise(idx, N):
        w = torch.randn((len(idx), N, N), dtype=torch.float64, device=DEV, generator=gen)
        return _smooth(w) if case["corr"] else w

    data, off, sums = _stamps(case, gen, th, side, kind, fwhm, snr, noise)
    corr = None
    if case["corr"]:
        corr = torch.zeros(len(data), dtype=torch.float32, device=DEV)
        for N, idx in _groups(side):
            at = off[idx][:, None] + torch.arange(J * N * N, device=DEV)[None]
            corr[at.reshape(-1)] = _lag_corr(N).float().reshape(-1).repeat(len(idx) * J)
    s = {"data": data if case["f64"] else data.float(), "offsets": off, "side": side, "psf": _psf_arg(kind, fwhm),
         "noise_sigma": torch.ones(case["n"] * J, device=DEV), "init": _starts(gen, th, sums, case["chains"]),
         "cfg": _config(case, profile=case["profile"], spergel_nu=-0.3 if case["profile"] == 1 else 0.5)}
    kw = {"n_exposures": J, "noise_corr": corr}
    if case["plan"] == "call":
        return {"args": s, "kw": kw}
    cls = api.RaggedFitPlan if case["plan"] == "ragged" else api.FitPlan
    return {"plan": cls(**s, **kw)}


def _prepare_pixel(case, gen):
    th, side, kind, fwhm, snr = _galaxies(case, gen)
    N, n = case["side"], case["n"]
    i = torch.arange(N, dtype=torch.float64, device=DEV)
    sd = 1.0 + 0.6 * (i[:, None] + i[None, :]) / (2.0 * (N - 1))
    data, off, sums = _stamps(case, gen, th, side, kind, fwhm, snr, lambda idx, N: sd * torch.randn(
        (len(idx), N, N), dtype=torch.float64, device=DEV, generator=gen))
    w = torch.zeros(len(data), dtype=torch.float32, device=DEV)
    keep = torch.rand((n, N * N), device=DEV, generator=gen) >= 0.01      # 1% of the pixels are masked
    at = off[:, None] + torch.arange(N * N, device=DEV)[None]
    w[at.reshape(-1)] = (keep * (1.0 / sd ** 2).float().reshape(-1)[None]).reshape(-1)
    return {"plan": api.FitPlan(data.float(), off, side, _psf_arg(kind, fwhm), torch.ones(n, device=DEV),
                                _starts(gen, th, sums, case["chains"]), _config(case), max_side=N, pixel_weight=w)}


def _prepare_dense(case, gen):
    """A noise level rising across the stamp, smoothed noise, and a stray-light wave per galaxy."""
    n, N = case["n"], case["side"]
    f = dict(dtype=torch.float64, device=DEV, generator=gen)
    c = (N - 1) // 2
    p = torch.arange(N * N, device=DEV)
    y, x = p // N - c, p % N - c
    C = _lag_corr(N)[(y[:, None] - y[None, :] + c) % N, (x[:, None] - x[None, :] + c) % N]
    ang = 2.0 * math.pi * torch.rand((n, 1), **f)
    sd = 1.1 + 0.4 * (x * torch.cos(ang) + y * torch.sin(ang)) / max(c, 1)
    k = torch.rand((n, 2, 1), **f) - 0.5
    v = 0.4 * torch.cos(k[:, 0] * x + k[:, 1] * y + 2.0 * math.pi * torch.rand((n, 1), **f))
    cov = (sd[:, :, None] * C * sd[:, None, :] + v[:, :, None] * v[:, None, :]).float()
    th, side, kind, fwhm, snr = _galaxies(dict(case, moffat=False), gen)
    th[:, 1] -= 0.25                                                      # galaxies that fit the smaller stamps

    def noise(idx, N):
        w = _smooth(torch.randn((len(idx), N, N), **f))
        return sd[idx].reshape(-1, N, N) * w + v[idx].reshape(-1, N, N) * torch.randn((len(idx), 1, 1), **f)

    data, off, sums = _stamps(case, gen, th, side, kind, fwhm, snr + 10.0, noise)
    return {"cov": cov.reshape(-1), "cov_offsets": torch.arange(n, device=DEV) * N ** 4, "side": side,
            "fit": (data.float(), off, side, _psf_arg(kind, fwhm), torch.ones(n, device=DEV),
                    _starts(gen, th, sums, case["chains"]), _config(case)), "shape": (n, N * N)}


def _prepare_ess(case, gen):
    """Chains as HMC leaves them: short correlations of either sign, means far from zero beside the spread."""
    n, C, S = case["n"], case["chains"], case["samples"]
    f = dict(device=DEV, generator=gen)
    phi = -0.4 + 0.9 * torch.rand((6, n, 1), **f)
    z = torch.randn((S, 6, n, C), **f)
    a = torch.sqrt(1.0 - phi * phi)
    for t in range(1, S):
        z[t] = phi * z[t - 1] + a * z[t]
    mean = torch.tensor([2.8, -0.1, 0.05, 0.05, 0.0, 0.0], device=DEV).view(6, 1, 1, 1)
    sd = torch.tensor([0.02, 0.03, 0.06, 0.06, 0.1, 0.1], device=DEV).view(6, 1, 1, 1)
    return {"samples": (mean + sd * torch.randn((6, n, 1, 1), **f) + sd * z.permute(1, 2, 3, 0)).contiguous()}


def _interim(n, K, gen):
    """Interim ellipticity samples of sheared galaxies, scattered in eta = 2 atanh|e| e/|e|."""
    e1, e2 = torch.empty((n, K), device=DEV), torch.empty((n, K), device=DEV)
    for s in range(0, n, 100000):
        m = min(100000, n - s)
        a, b = _ellipticities(m, gen, 0.2, 0.62)
        a, b = _sheared(a, b, torch.full_like(a, 0.02), torch.full_like(a, -0.01))
        r = torch.hypot(a, b).clamp_min(1e-12)
        k = (2.0 * torch.atanh(r) / r)
        a, b = [(t * k + 0.1 * torch.randn(m, dtype=torch.float64, device=DEV, generator=gen)).float() for t in (a, b)]
        x = a[:, None] + 0.1 * torch.randn((m, K), device=DEV, generator=gen)
        y = b[:, None] + 0.1 * torch.randn((m, K), device=DEV, generator=gen)
        rho = torch.hypot(x, y).clamp_min(1e-12)
        k = torch.tanh(0.5 * rho) / rho
        e1[s:s + m], e2[s:s + m] = x * k, y * k
    return e1, e2


def _point(gen):
    u = torch.rand(3, dtype=torch.float64, device=DEV, generator=gen).cpu().numpy()
    return [0.01 + 0.02 * float(u[0]), -0.02 + 0.02 * float(u[1]), 0.18 + 0.04 * float(u[2])]


def _prepare_shear(case, gen):
    n, K = case["n"], case["K"]
    e1, e2 = _interim(n, K, gen)
    b = 0.1 * torch.randn((n, K), device=DEV, generator=gen) if case.get("b") else None
    w = None
    if case.get("weights"):      # the counts of a bootstrap resample
        w = torch.bincount(torch.randint(n, (n,), device=DEV, generator=gen), minlength=n).float()
    plan = api.ShearPlan(e1, e2, b, family=case.get("family", 1), trunc_r=0.7, weights=w)
    s = {"plan": plan, "e1": e1, "e2": e2, "b": b, "w": w, "x": _point(gen)}
    if case["kind"] == "full":
        f = dict(device=DEV, generator=gen)
        lf = 2.45 + 0.4 * torch.randn((n, 1), **f).abs() + 0.1 * (torch.rand((n, 1), **f) - 0.2)
        s["lf"] = (lf + 0.03 * torch.randn((n, K), **f)).contiguous()
        s["ls"] = (-0.4 + 0.06 * torch.randn((n, 1), **f) + 0.03 * torch.randn((n, K), **f)).contiguous()
        s["theta"] = s["x"] + [2.45, 0.4, 14.0, -0.4, 0.06]
    return s


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    kind = case["kind"]
    make = _prepare_shear if kind in ("pass", "estimate", "full") else {
        "render": _prepare_render, "points": _prepare_points, "fit": _prepare_fit, "pixel": _prepare_pixel,
        "dense": _prepare_dense, "ess": _prepare_ess}[kind]
    return {"case": dict(case), **make(case, gen)}


# --------------------------------------------------------------------------- one pass

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "render":
        img, off = api.render(state["theta"], state["side"], state["psf"], shear=state["shear"])
        return {"stamps": img, "offsets": off}
    if kind == "points":
        th = state["theta"].detach().requires_grad_()
        lp = api.RenderLogPost.apply(th, state["data"], state["offsets"], state["side"], state["psf"], state["sigma"],
                                     state["gal"])
        return {"logp": lp.detach(), "grad": torch.autograd.grad(lp.sum(), th)[0]}
    if kind == "fit" and case["plan"] == "call":
        return api.fit_galaxies(**state["args"], **state["kw"])
    if kind in ("fit", "pixel"):
        return state["plan"].run().result()
    if kind == "dense":
        prec, status = api.dense_precision(state["cov"], state["cov_offsets"], state["side"])
        out = api.fit_galaxies(*state["fit"], pixel_prec=prec, prec_offsets=state["cov_offsets"])
        return {"prec": prec, "prec_status": status, "fit": out}
    if kind == "ess":
        ess, rhat = api.chain_ess(state["samples"])
        return {"ess": ess, "rhat": rhat}
    plan = state["plan"]
    if kind == "estimate":
        mean, cov = plan.estimate(free_alpha=case["free"], alpha=0.21, alpha_lo=0.1, alpha_hi=0.4)
        return {"mean": mean, "cov": cov}
    if kind == "full":
        value, grad = plan.loglike_full(state["lf"], state["ls"], state["theta"])
        return {"value": float(value), "grad": grad}
    if case["autograd"]:
        x = torch.tensor(state["x"], dtype=torch.float64, requires_grad=True)
        v = api.ShearLogLike.apply(x, plan)
        return {"value": v.detach(), "grad": torch.autograd.grad(v, x)[0]}
    return {"value_grad": plan.loglike(*state["x"])}


# --------------------------------------------------------------------------- the same in 64 bits

def _log_z(family, alpha):
    if family == 1:
        return torch.log(2.0 * math.pi * alpha ** 2) + torch.log(-torch.expm1(-0.49 / (2.0 * alpha ** 2)))
    a = 1.0 / (2.0 * alpha ** 2)
    return torch.log(math.pi * (1.0 / a - 2.0 / a ** 2 - 2.0 * torch.expm1(-a) / a ** 3))


def _log_p(family, alpha, E):
    q = -E / (2.0 * alpha ** 2) - _log_z(family, alpha)
    if family == 1:
        return torch.where(E < float(np.float32(0.7) ** 2), q, torch.full_like(q, -math.inf))
    return q + 2.0 * torch.log1p(-E)


def _shear64(s, family, x, grad=True):
    """Log-likelihood and gradient at x = (g1, g2, alpha[, mu_f, sigma_f, a_f, mu_s, sigma_s])."""
    x = torch.tensor(x, dtype=torch.float64, device=DEV, requires_grad=grad)
    n, K = s["e1"].shape
    e0 = torch.tensor(float(np.float32(0.3)), dtype=torch.float64, device=DEV)
    total, g = 0.0, torch.zeros_like(x)
    rows = max(1, 6000000 // K)
    for i in range(0, n, rows):
        e1, e2 = s["e1"][i:i + rows].double(), s["e2"][i:i + rows].double()
        E = e1 * e1 + e2 * e2
        U = (1.0 - x[0] * e1 - x[1] * e2) ** 2 + (x[0] * e2 - x[1] * e1) ** 2
        Q = ((e1 - x[0]) ** 2 + (e2 - x[1]) ** 2) / U
        lw = _log_p(family, x[2], Q) + 2.0 * torch.log((1.0 - x[0] ** 2 - x[1] ** 2) / U) - _log_p(0, e0, E)
        if s["b"] is not None:
            lw = lw + s["b"][i:i + rows].double()
        if len(x) > 3:
            z = (s["lf"][i:i + rows].double() - x[3]) / x[4]
            y = (s["ls"][i:i + rows].double() - x[6]) / x[7]
            lw = lw + (math.log(2.0 * (LF[1] - LF[0]) * (LS[1] - LS[0]) / (2.0 * math.pi)) - 0.5 * (z * z + y * y)
                       + torch.special.log_ndtr(x[5] * z) - torch.log(x[4] * x[7]))
        L = torch.logsumexp(lw, 1) - math.log(K)
        v = (L * s["w"][i:i + rows].double()).sum() if s["w"] is not None else L.sum()
        if grad:
            g += torch.autograd.grad(v, x)[0]
        total = total + v.detach()
    return float(total), g.detach().cpu().numpy()


def _estimate64(s, free):
    """Posterior mean and covariance: Newton to the mode, 7-point Gauss-Hermite nodes on the Laplace grid."""
    d = 3 if free else 2
    x = np.array([0.0, 0.0, 0.21])

    def grad(y):
        return _shear64(s, 1, list(y))[1][:d]

    for _ in range(6):
        H = np.zeros((d, d))
        for j in range(d):
            h = np.zeros(3)
            h[j] = 1e-4
            H[j] = (grad(x + h) - grad(x - h)) / 2e-4
        step = np.linalg.solve(-(H + H.T) / 2, grad(x))
        x[:d] += step
        if np.abs(step).max() < 1e-9:
            break
    Lc = np.linalg.cholesky(np.linalg.inv(-(H + H.T) / 2))
    t, w = np.polynomial.hermite.hermgauss(7)
    z = np.stack(np.meshgrid(*[t] * d, indexing="ij"), -1).reshape(-1, d)
    lw = np.log(np.stack(np.meshgrid(*[w] * d, indexing="ij"), -1).reshape(-1, d)).sum(1) + (z * z).sum(1)
    pts = np.tile(x, (len(z), 1))
    pts[:, :d] += math.sqrt(2.0) * z @ Lc.T
    lw = lw + np.array([_shear64(s, 1, list(p), grad=False)[0] for p in pts])
    p = np.exp(lw - lw.max())
    p /= p.sum()
    mean = p @ pts[:, :d]
    return {"mean": mean, "cov": (pts[:, :d] - mean).T @ ((pts[:, :d] - mean) * p[:, None])}


def _ess64(samples):
    n6, n, C, S = samples.shape
    ess, rhat = [], []
    for k in range(n6):
        x = samples[k].double()
        m = x.mean(2)
        d = x - m[..., None]
        W = (d ** 2).sum(2).div(S - 1).mean(1)
        B = m.var(1) if C > 1 else torch.zeros_like(W)
        vp = (S - 1) / S * W + B
        f = torch.fft.rfft(d, 2 * S)
        ac = torch.fft.irfft(f.real ** 2 + f.imag ** 2, 2 * S)[..., :S].mean(1) / S
        rho = 1.0 - (W[:, None] - ac) / vp[:, None]
        rho[:, 0] = 1.0
        P = rho[:, :S // 2 * 2].reshape(n, -1, 2).sum(2)
        keep = torch.cumprod((P > 0).double(), 1)
        tau = -1.0 + 2.0 * (torch.cummin(P, 1).values * keep).sum(1)
        ess.append(C * S / tau.clamp_min(1.0 / math.log10(C * S)))
        rhat.append(torch.sqrt(vp / W))
    return {"ess": torch.stack(ess, 1), "rhat": torch.stack(rhat, 1)}


def _render64(state):
    th, side = state["theta"].double(), state["side"]
    if state["shear"] is not None:
        g = state["shear"].double()
        a, b = _sheared(th[:, 2], th[:, 3], g[:, 0], g[:, 1])
        th = torch.cat([th[:, :2], a[:, None], b[:, None], th[:, 4:]], 1)
    off, total = _pack(side)
    out = torch.zeros(total, dtype=torch.float64, device=DEV)
    for N, idx in _groups(side):
        for i in idx.split(2000):
            img = _image64(th[i], N, _transfer64(N, (state["kind"], state["fwhm"][i, 0])))
            at = off[i][:, None] + torch.arange(N * N, device=DEV)[None]
            out[at.reshape(-1)] = img.reshape(-1)
    return {"stamps": out, "offsets": None}


def _points64(state):
    lp = torch.zeros(len(state["gal"]), dtype=torch.float64, device=DEV)
    grad = torch.zeros((len(lp), 6), dtype=torch.float64, device=DEV)
    sxy, se = SXY, float(np.float32(SE))
    z = _log_z(0, torch.tensor(se, dtype=torch.float64))
    const = -math.log(LF[1] - LF[0]) - math.log(LS[1] - LS[0]) - math.log(2.0 * math.pi * sxy ** 2) - float(z)
    gal = state["gal"].long()
    for N, idx in _groups(state["side"][gal]):
        for i in idx.split(1000):
            th = state["theta"][i].double().requires_grad_()
            at = state["offsets"][gal[i]][:, None] + torch.arange(N * N, device=DEV)[None]
            d = state["data"][at].double().reshape(-1, N, N)
            m = _image64(th, N, _transfer64(N, (state["kind"], state["fwhm"][gal[i], 0])))
            E = th[:, 2] ** 2 + th[:, 3] ** 2
            v = (-0.5 * ((d - m) ** 2).sum((1, 2)) + const - 0.5 * (th[:, 4] ** 2 + th[:, 5] ** 2) / sxy ** 2
                 + 2.0 * torch.log1p(-E) - 0.5 * E / se ** 2)
            grad[i] = torch.autograd.grad(v.sum(), th)[0]
            lp[i] = v.detach()
    return {"logp": lp, "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "pixel"):
        return None              # whole Markov chains: no value in 64 bits to hold the draws against
    s = prepare(case, seed)
    if kind == "render":
        return _render64(s)
    if kind == "points":
        return _points64(s)
    if kind == "ess":
        return _ess64(s["samples"])
    if kind == "dense":
        n, m = s["shape"]
        return {"prec": torch.linalg.inv(s["cov"].double().reshape(n, m, m)).reshape(-1), "prec_status": None, "fit": None}
    if kind == "estimate":
        return _estimate64(s, case["free"])
    if kind == "full":
        v, g = _shear64(s, case["family"], s["theta"])
        return {"value": v, "grad": g}
    v, g = _shear64(s, case["family"], s["x"])
    return {"value": v, "grad": g} if case["autograd"] else {"value_grad": np.concatenate([[v], g])}
