"""The calls this library is measured on: one pass of each through its public entry points.

A case is one call, or the short chain of calls, that a simulation of optical
interstellar scintillation makes: a phase screen, its propagation at one
wavelength or over a passband, the disk of an extended source, light curves and
their statistics, a whole batch of screens, the gradient step of a light-curve
fit, and the screen check.  The listed sizes are those of this repository's
workloads (paper_1301_0514_gb300/workloads.py, sweeps.py, bench.py); draw() takes
others from the same ranges.  exact() restates every case in plain torch in
64 bits, without the library.
"""
from __future__ import annotations

import math
import random
from typing import Dict

import numpy as np
import torch

import paper_1301_0514_gb300 as S

KM_PER_PC = 3.0856775814913673e13
KM_PER_NM = 1.0e-12
KOLMOGOROV = 11.0 / 3.0
R_SUN_KM = 695700.0


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def listed():
    return [
        # The smallest configuration, in FP64 throughout: screen and propagation of one 256^2 grid.
        # A call of a few microseconds per kernel: launches and the FP64 pipe count.
        dict(name="plain64_256", kind="plain64", n=256, pixel=20.0, r_diff=100.0, beta=KOLMOGOROV),
        # One pattern of a screen that is in hand, at one wavelength, with its light curves: the
        # smallest FP32 call, as an interactive user or a parameter scan makes it.
        dict(name="point_1024", kind="point", n=1024, pixel=10.0, r_diff=100.0, lam=550.0, tracks=8, samples=512),
        # The synthesis alone: one Kolmogorov screen of the single-screen configuration.
        dict(name="screen_4096", kind="screen", n=4096, pixel=10.0, r_diff=100.0, beta=KOLMOGOROV),
        # The single-screen configuration: screen, point-source pattern at one wavelength, 64 curves.
        dict(name="single_4096", kind="chain", n=4096, pixel=10.0, r_diff=30.0, beta=KOLMOGOROV, disk=0.0,
             tracks=64, samples=2048),
        # One screen of the batched configuration with its screen in hand: a 32-wavelength passband,
        # an extended source, 8 curves.
        dict(name="passband_2048", kind="passband", n=2048, pixel=10.0, r_diff=100.0, lambdas=32, flat=True,
             disk=0.7, tracks=8, samples=1024),
        # The batched configuration: 48 screens of three sizes, 32 wavelengths, extended sources,
        # curves, one call.
        dict(name="batch_48", kind="batch", small=1024, mid=2048, large=4096, per_size=16, lambdas=32, lanes=8,
             tracks=8),
        # Two patterns of the modulation-index sweep: 8192^2, the 21 wavelengths of the K_s band.
        dict(name="sweep_8192", kind="sweep", n=8192, count=2, r_diff=200.0, r_s=0.75, beta=KOLMOGOROV, lambdas=21),
        # The large single screen, non-Kolmogorov, with a disk of one R_ref and 16 curves.
        dict(name="large_16384", kind="chain", n=16384, pixel=5.0, r_diff=100.0, beta=3.3, disk=1.0,
             tracks=16, samples=8192),
        # One step of a light-curve fit, forward and backward: 8 screens of 2048^2, one long track each.
        dict(name="fit_2048", kind="fit", n=2048, count=8, pixel=10.0, r_diff=100.0, lambdas=1, disk=0.0, tracks=1,
             samples=10000),
        # The paper's one-FFT propagator over a passband at critical sampling.
        dict(name="one_fft_4096", kind="one_fft", n=4096, r_diff=500.0, lambdas=8),
        # The screen check of the paper's 14000^2 screen: spectrum and structure function recomputed.
        dict(name="check_14000", kind="check", n=14000, pixel=28.85, r_diff=500.0, lags=48),
        # What is measured on a finished pattern: m, curves, their power spectra, the decorrelation of
        # two telescopes.
        dict(name="pattern_8192", kind="pattern", n=8192, tracks=64, samples=4096, pairs=16, separations=24),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid(rng: random.Random, lo: int, hi: int) -> int:
    return 1 << rng.randint(lo.bit_length() - 1, hi.bit_length() - 1)


def draw(rng: random.Random) -> Dict:
    kind = rng.choice(["plain64", "point", "screen", "chain", "passband", "batch", "sweep", "fit", "one_fft",
                       "check", "pattern"])
    beta = rng.choice([KOLMOGOROV, KOLMOGOROV, 3.1, 3.3, 3.9])
    r_diff = math.exp(rng.uniform(math.log(30.0), math.log(300.0)))
    if kind == "plain64":
        return dict(kind=kind, n=_grid(rng, 64, 1024), pixel=rng.uniform(5.0, 20.0), r_diff=rng.uniform(50.0, 300.0),
                    beta=beta)
    if kind == "point":
        return dict(kind=kind, n=_grid(rng, 128, 8192), pixel=10.0, r_diff=r_diff, lam=rng.uniform(450.0, 2200.0),
                    tracks=rng.randint(1, 70), samples=_log_int(rng, 100, 10000))
    if kind == "screen":
        return dict(kind=kind, n=_grid(rng, 128, 16384), pixel=rng.uniform(5.0, 12.0), r_diff=r_diff, beta=beta)
    if kind == "chain":
        return dict(kind=kind, n=_grid(rng, 256, 16384), pixel=rng.uniform(5.0, 10.0), r_diff=r_diff, beta=beta,
                    disk=rng.choice([0.0, rng.uniform(0.1, 2.0)]), tracks=rng.randint(1, 64),
                    samples=_log_int(rng, 100, 10000))
    if kind == "passband":
        n = _grid(rng, 256, 8192)
        return dict(kind=kind, n=n, pixel=10.0, r_diff=r_diff, lambdas=_log_int(rng, 2, 40 if n < 8192 else 16),
                    flat=rng.random() < 0.5, disk=rng.uniform(0.1, 2.0), tracks=rng.randint(1, 16),
                    samples=_log_int(rng, 100, 10000))
    if kind == "batch":
        large = _grid(rng, 1024, 4096)
        return dict(kind=kind, small=large // 4, mid=large // 2, large=large, per_size=rng.randint(2, 12),
                    lambdas=rng.randint(3, 32), lanes=rng.choice([2, 4, 8]), tracks=rng.randint(1, 12))
    if kind == "sweep":
        return dict(kind=kind, n=_grid(rng, 2048, 8192), count=rng.randint(2, 4), r_diff=rng.uniform(50.0, 500.0),
                    r_s=rng.uniform(0.25, 1.5), beta=beta, lambdas=rng.choice([11, 21]))
    if kind == "fit":
        n = _grid(rng, 256, 4096)
        return dict(kind=kind, n=n, count=rng.randint(1, 6), pixel=10.0, r_diff=r_diff, lambdas=rng.randint(1, 5),
                    disk=rng.choice([0.0, rng.uniform(0.1, 1.0)]), tracks=rng.randint(1, 4),
                    samples=_log_int(rng, 500, 10000))
    if kind == "one_fft":
        n = _grid(rng, 1024, 8192)
        return dict(kind=kind, n=n, r_diff=rng.uniform(300.0, 800.0), lambdas=_log_int(rng, 1, 24 if n < 8192 else 8))
    if kind == "check":
        return dict(kind=kind, n=2 * _log_int(rng, 500, 7000), pixel=rng.uniform(10.0, 30.0),
                    r_diff=rng.uniform(100.0, 600.0), lags=rng.randint(1, 64))
    return dict(kind=kind, n=_grid(rng, 512, 8192), tracks=rng.randint(1, 100), samples=_grid(rng, 256, 8192),
                pairs=rng.randint(1, 16), separations=rng.randint(2, 32))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _lz(lam, z=160.0):
    return lam * KM_PER_NM * z * KM_PER_PC


def _rng(seed):
    return np.random.default_rng(int(seed) % (1 << 63))


def _tracks(rng, n, count, ds=1.0):
    return np.stack([rng.uniform(0.0, n, count), rng.uniform(0.0, n, count), rng.uniform(0.0, math.pi, count),
                     np.full(count, ds)], axis=1)


def _band(count, lo=400.0, hi=700.0):
    return np.linspace(lo, hi, count) if count > 1 else np.array([0.5 * (lo + hi)])


def _weights(case, rng):
    if case.get("flat", True):
        return None
    w = rng.uniform(0.2, 1.0, case["lambdas"])
    return w / w.sum()


def _spectrum_c(r_diff, beta):
    fb = 2.0 ** (-beta) * beta * math.gamma(-beta / 2.0) / math.gamma(beta / 2.0)
    return r_diff ** 2 / (2.0 * (2.0 * math.pi) ** (beta - 1.0) * fb)


def _any_screen(n, pixel, r_diff, seed, beta=KOLMOGOROV):
    """A phase screen in hand, as a file of a user's own: Gaussian with the power-law spectrum, FP64."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
    L = n * pixel
    k = torch.fft.fftfreq(n, d=pixel, device="cuda", dtype=torch.float64)
    kx = torch.fft.rfftfreq(n, d=pixel, device="cuda", dtype=torch.float64)
    q2 = k[:, None] ** 2 + kx[None, :] ** 2
    q2[0, 0] = 1.0
    amp = math.sqrt(_spectrum_c(r_diff, beta)) * (r_diff * r_diff * q2) ** (-beta / 4.0) / L
    amp[0, 0] = 0.0
    w = torch.view_as_complex(torch.randn(n, n // 2 + 1, 2, generator=g, device="cuda", dtype=torch.float64))
    return torch.fft.irfft2(w * (amp * math.sqrt(0.5)), s=(n, n)) * float(n) * float(n)


def _any_pattern(n, seed):
    """An illumination pattern in hand: positive, mean about one, speckles of a few tens of pixels."""
    f = _any_screen(n, 10.0, 250.0, seed)
    f = f / f.std()
    return torch.exp(0.4 * f).to(torch.float32).contiguous()


def _params(case, seed):
    """Parameters of the case's screens, host track arrays and wavelengths, from the seed alone."""
    kind, rng = case["kind"], _rng(seed)
    if kind in ("plain64", "screen"):
        p = S.params(case["n"], case["pixel"], case["r_diff"], beta=case["beta"], seed=seed, screen_id=1)
        return dict(p=[p])
    if kind == "point":
        p = S.params(case["n"], case["pixel"], case["r_diff"], lambda_nm=case["lam"], lambda_ref_nm=550.0, seed=seed)
        return dict(p=[p], tracks=[_tracks(rng, case["n"], case["tracks"])])
    if kind == "chain":
        rs = case["disk"] * _lz(500.0) / case["r_diff"]
        p = S.params(case["n"], case["pixel"], case["r_diff"], beta=case["beta"], source_radius_km=rs, seed=seed,
                     screen_id=2)
        return dict(p=[p], tracks=[_tracks(rng, case["n"], case["tracks"])])
    if kind in ("passband", "fit"):
        rs = case["disk"] * _lz(550.0) / case["r_diff"]
        count = case.get("count", 1)
        p = [S.params(case["n"], case["pixel"], case["r_diff"], lambda_nm=550.0, source_radius_km=rs, seed=seed + i,
                      screen_id=i) for i in range(count)]
        ds = 1.0 if kind == "passband" else 0.2
        lams = _band(case["lambdas"])
        return dict(p=p, tracks=[_tracks(rng, case["n"], case["tracks"], ds) for _ in p], lams=lams,
                    weights=_weights(case, rng))
    if kind == "batch":
        p, tr = [], []
        for n in (case["small"], case["mid"], case["large"]):
            for _ in range(case["per_size"]):
                rd = rng.uniform(30.0, 300.0)
                rs = rng.uniform(0.1, 2.0) * _lz(550.0) / rd
                p.append(S.params(n, 10.0, rd, lambda_nm=550.0, source_radius_km=rs, seed=seed + len(p),
                                  screen_id=len(p)))
                tr.append(_tracks(rng, n, case["tracks"]))
        return dict(p=p, tracks=tr, lams=_band(case["lambdas"]))
    if kind == "sweep":
        p = []
        for i in range(case["count"]):
            rd = case["r_diff"] * (1.0 + 0.25 * i)
            p.append(S.params(case["n"], rd / 3.0, rd, beta=case["beta"], lambda_nm=2162.0,
                              source_radius_km=case["r_s"] * R_SUN_KM * 0.16, seed=seed + i, screen_id=i))
        return dict(p=p, lams=_band(case["lambdas"], 2162.0 - 82.0, 2162.0 + 118.0))
    if kind == "one_fft":
        pixel = math.sqrt(_lz(2162.0) / case["n"])
        p = S.params(case["n"], pixel, case["r_diff"], lambda_nm=2162.0, seed=seed)
        return dict(p=[p], lams=_band(case["lambdas"], 2080.0, 2280.0))
    if kind == "check":
        p = S.params(case["n"], case["pixel"], case["r_diff"], seed=seed, screen_id=3)
        return dict(p=[p], lags=np.geomspace(0.5 * case["pixel"], 0.2 * case["n"] * case["pixel"], case["lags"]))
    p = S.params(case["n"], 10.0, 100.0, seed=seed)
    tracks = _tracks(rng, case["n"], case["tracks"])
    return dict(p=[p], tracks=[tracks], pairs=_tracks(rng, case["n"], case["pairs"]),
                separations=np.concatenate([[0.0], np.geomspace(2.0, 600.0, case["separations"] - 1)]))


def prepare(case, seed):
    kind, seed = case["kind"], int(seed)
    st = dict(_params(case, seed), case=case)
    p = st["p"][0]
    n = p.n
    f32 = lambda *s: torch.empty(s, dtype=torch.float32, device="cuda")  # noqa: E731
    f64 = lambda *s: torch.empty(s, dtype=torch.float64, device="cuda")  # noqa: E731
    ws = lambda b: torch.empty(b, dtype=torch.uint8, device="cuda")  # noqa: E731
    if kind in ("plain64", "screen", "chain"):
        st["phi"], st["ws"] = f64(n, n), ws(S.workspace_bytes(p, 1))
    if kind == "plain64":
        st["out"] = f64(n, n)
    elif kind == "chain":
        st["out"], st["curves"] = f32(n, n), f32(case["tracks"], case["samples"])
    elif kind == "point":
        st["phi"] = _any_screen(n, p.pixel_km, p.r_diff_km, seed)
        st["ws"], st["out"] = ws(S.workspace_bytes(p, 1)), f32(n, n)
        st["curves"] = f32(case["tracks"], case["samples"])
    elif kind == "passband":
        st["phi"] = _any_screen(n, p.pixel_km, p.r_diff_km, seed)
        st["ws"], st["out"] = ws(S.workspace_bytes(p, case["lambdas"])), f32(n, n)
        st["curves"] = f32(case["tracks"], case["samples"])
    elif kind in ("batch", "sweep"):
        items, maps, curves = [], {}, {}
        for i, q in enumerate(st["p"]):
            k = sum(1 for r in st["p"] if r.n == q.n)
            maps.setdefault(q.n, (f32(k, q.n, q.n), []))
            j = len(maps[q.n][1])
            maps[q.n][1].append(i)
            it = dict(params=q, intensity=maps[q.n][0][j])
            if kind == "batch":
                ns = q.n // 2
                curves.setdefault(q.n, f32(k, case["tracks"], ns))
                it.update(tracks=st["tracks"][i], n_samples=ns, curves=curves[q.n][j])
            items.append(it)
        st["lanes"] = case.get("lanes", 2)
        st["items"] = S.batch_items(items)
        st["ws"] = ws(S.batch_workspace_bytes(st["items"], case["lambdas"], st["lanes"]))
        st["maps"], st["curves"] = {m: v[0] for m, v in maps.items()}, curves
    elif kind == "fit":
        g = torch.Generator(device="cuda").manual_seed(seed)
        st["phi"] = [_any_screen(n, p.pixel_km, p.r_diff_km, seed + 7 * i) for i in range(case["count"])]
        st["delta"] = [(0.05 * torch.randn(n, n, generator=g, device="cuda")).requires_grad_() for _ in st["phi"]]
        st["target"] = [1.0 + 0.3 * torch.randn(case["tracks"], case["samples"], generator=g, device="cuda")
                        for _ in st["phi"]]
        st["ws"] = ws(S.workspace_bytes(p, case["lambdas"]))
    elif kind == "one_fft":
        st["phi"] = _any_screen(n, p.pixel_km, p.r_diff_km, seed)
        st["out"] = f32(n, n)
        st["ws"] = ws(S.workspace_bytes(p, case["lambdas"]) + 4 * n * n * case["lambdas"])
    elif kind == "check":
        bins = S.max_annulus(n) + 1
        st["s"], st["c"] = f64(bins), torch.empty(bins, dtype=torch.int64, device="cuda")
        st["r"] = torch.as_tensor(st["lags"], device="cuda")
        st["d"], st["root"], st["ws"] = f64(case["lags"]), f64(1), ws(1 << 16)
    elif kind == "pattern":
        st["map"] = _any_pattern(n, seed)
        st["ws"] = ws(S.workspace_bytes(p, 1))
        st["curves"] = f32(case["tracks"], case["samples"])
    return st


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(st):
    case = st["case"]
    kind, p = case["kind"], st["p"][0]
    if kind == "screen":
        return {"phi": S.make_screen(p, out=st["phi"], workspace=st["ws"])}
    if kind == "plain64":
        phi = S.make_screen(p, out=st["phi"], workspace=st["ws"])
        return {"phi": phi, "intensity": S.propagate64(p, phi, out=st["out"], workspace=st["ws"])}
    if kind == "point":
        inten = S.propagate(p, st["phi"], out=st["out"], workspace=st["ws"])
        return {"intensity": inten,
                "curves": S.lightcurve(p, inten, st["tracks"][0], case["samples"], out=st["curves"])}
    if kind == "chain":
        phi = S.make_screen(p, out=st["phi"], workspace=st["ws"])
        inten = S.propagate(p, phi, out=st["out"], workspace=st["ws"])
        if p.source_radius_km > 0.0:
            S.smooth_source(p, inten, workspace=st["ws"])
        return {"intensity": inten,
                "curves": S.lightcurve(p, inten, st["tracks"][0], case["samples"], out=st["curves"])}
    if kind == "passband":
        inten = S.sum_passband(p, st["phi"], st["lams"], st["weights"], out=st["out"], workspace=st["ws"])
        S.smooth_source(p, inten, workspace=st["ws"])
        return {"intensity": inten,
                "curves": S.lightcurve(p, inten, st["tracks"][0], case["samples"], out=st["curves"])}
    if kind in ("batch", "sweep"):
        S.run_batch(st["items"], st["lams"], n_lanes=st["lanes"], workspace=st["ws"])
        return {"maps": [st["maps"][n] for n in sorted(st["maps"])],
                "curves": [st["curves"][n] for n in sorted(st["curves"])]}
    if kind == "fit":
        # the correction of each screen is the user's parameter, in torch's default type
        out = {"curves": [], "loss": [], "grad": []}
        for i, q in enumerate(st["p"]):
            delta = st["delta"][i]
            delta.grad = None
            curves = S.light_curves(st["phi"][i] + delta, q, st["lams"], st["tracks"][i], case["samples"],
                                    workspace=st["ws"])
            loss = ((curves - st["target"][i]) ** 2).mean()
            loss.backward()
            out["curves"].append(curves.detach())
            out["loss"].append(loss.detach())
            out["grad"].append(delta.grad)
        return out
    if kind == "one_fft":
        return {"intensity": S.sum_passband_conjugate(p, st["phi"], st["lams"], out=st["out"], workspace=st["ws"])}
    if kind == "check":
        s, c = S.spectrum_rec(p, out=(st["s"], st["c"]))
        d, root = S.structure_function_rec(p, s, st["r"], workspace=st["ws"], out=(st["d"], st["root"]))
        return {"s_rec": s, "counts": c, "d_rec": d, "r_rec": root}
    from paper_1301_0514_gb300 import timeseries
    m = S.modulation_index(p, st["map"], workspace=st["ws"])
    curves = S.lightcurve(p, st["map"], st["tracks"][0], case["samples"], out=st["curves"])
    return {"m": m, "curves": curves, "m_curves": S.curve_modulation(curves),
            "power": timeseries.power_spectra(curves),
            "decorrelation": timeseries.decorrelation(p, st["map"], st["pairs"], st["separations"], case["samples"])}


# --------------------------------------------------------------------------
# bytes and operations a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    fft2 = lambda n: 5.0 * n * n * 2.0 * math.log2(n)  # noqa: E731  (one complex 2D transform)
    if kind == "batch":
        b = f = 0.0
        for n in (case["small"], case["mid"], case["large"]):
            b += case["per_size"] * (4.0 * n * n + 2.0 * n * case["tracks"])
            f += case["per_size"] * (0.5 * fft2(n) + 2.0 * case["lambdas"] * fft2(n) + fft2(n))
        return {"bytes": b, "flops": f}
    n = case["n"]
    nn = float(n) * n
    if kind == "screen":
        return {"bytes": 8.0 * nn, "flops": 0.5 * fft2(n)}
    if kind == "plain64":
        return {"bytes": 16.0 * nn, "flops": 2.5 * fft2(n)}
    if kind == "point":
        return {"bytes": 12.0 * nn + 4.0 * case["tracks"] * case["samples"], "flops": 2.0 * fft2(n)}
    if kind == "chain":
        return {"bytes": 4.0 * nn + 4.0 * case["tracks"] * case["samples"],
                "flops": (2.5 + (1.0 if case["disk"] > 0 else 0.0)) * fft2(n)}
    if kind == "passband":
        return {"bytes": 12.0 * nn + 4.0 * case["tracks"] * case["samples"],
                "flops": (2.0 * case["lambdas"] + 1.0) * fft2(n)}
    if kind == "sweep":
        return {"bytes": 4.0 * nn * case["count"], "flops": case["count"] * (1.5 + 2.0 * case["lambdas"]) * fft2(n)}
    if kind == "fit":
        d = 2.0 if case["disk"] > 0 else 0.0
        return {"bytes": case["count"] * 16.0 * nn, "flops": case["count"] * (6.0 * case["lambdas"] + d) * fft2(n)}
    if kind == "one_fft":
        return {"bytes": 12.0 * nn, "flops": 1.0 * case["lambdas"] * fft2(n)}
    if kind == "check":
        # 10 Philox rounds of two 32 x 32 -> 64 bit products and the sum, per bin
        return {"bytes": 16.0 * 0.71 * n, "flops": 41.0 * nn}
    ns = case["samples"]
    return {"bytes": 4.0 * nn + 6.0 * case["tracks"] * ns,
            "flops": case["tracks"] * 2.5 * ns * math.log2(ns) + 3.0 * nn}


# --------------------------------------------------------------------------
# the same in 64 bits, plain torch
# --------------------------------------------------------------------------
def _philox(c0, c1, c2, seed):
    """Philox4x32-10 words of counters (c0, c1, c2, 0), as int64 tensors of 32-bit values."""
    mask = 0xFFFFFFFF
    c = [c0, c1, torch.full_like(c0, c2), torch.zeros_like(c0)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(m, x):       # 32 x 32 -> (high, low) without overflowing 63 bits
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        t = hi + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return c


def _uniform(hi, lo):
    return ((hi * 2097152 + (lo >> 11)).to(torch.float64) + 0.5) * 2.0 ** -53


def _noise_rows(p, rows):
    """F of the spectral rows (index tensor), complex128."""
    n, L = p.n, p.n * p.pixel_km
    kx = torch.arange(n, device="cuda")
    c0 = kx[None, :].expand(len(rows), n).contiguous()
    c1 = rows[:, None].expand(len(rows), n).contiguous()
    w = _philox(c0, c1, p.screen_id, p.seed)
    r = torch.sqrt(-2.0 * torch.log(_uniform(w[1], w[0])))
    th = 2.0 * math.pi * _uniform(w[3], w[2])
    f = torch.fft.fftfreq(n, d=p.pixel_km, device="cuda", dtype=torch.float64)
    q = torch.sqrt(f[rows][:, None] ** 2 + f[None, :] ** 2)
    s = torch.where(q > 0, _spectrum_c(p.r_diff_km, p.beta) * (p.r_diff_km * q) ** (-p.beta), torch.zeros_like(q))
    s = torch.sqrt(L * L * s) * math.sqrt(0.5) * r
    return torch.complex(s * torch.cos(th), s * torch.sin(th))


def _row_groups(n):
    step = max(1, (1 << 24) // n)
    for r in range(0, n, step):
        yield torch.arange(r, min(n, r + step), device="cuda")


def _screen64(p):
    F = torch.empty(p.n, p.n, dtype=torch.complex128, device="cuda")
    for rows in _row_groups(p.n):
        F[rows[0]:rows[-1] + 1] = _noise_rows(p, rows)
    L = p.n * p.pixel_km
    return torch.fft.ifft2(F).real.mul(math.sqrt(2.0) / (L * L) * float(p.n) ** 2)


def _taper64(p, lam):
    n, L = p.n, p.n * p.pixel_km
    margin = p.margin_km if p.margin_km >= 0 else min(10.0 * math.sqrt(_lz(lam, p.z_pc) / (2.0 * math.pi)), L / 4.0)
    if margin <= 0:
        return torch.ones(n, dtype=torch.float64, device="cuda")
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * p.pixel_km
    u = torch.minimum(x, L - x)
    return torch.where(u <= margin, torch.sin(math.pi * u / (2.0 * margin)) ** 2, torch.ones_like(u))


def _field64(p, phi, lam):
    t = phi * (p.lambda_ref_nm / lam)
    sf = _taper64(p, lam)
    return torch.polar(sf[:, None] * sf[None, :], t)


def _h64(p, lam):
    f = torch.fft.fftfreq(p.n, d=p.pixel_km, device="cuda", dtype=torch.float64)
    turns = 0.5 * _lz(lam, p.z_pc) * f * f
    th = -2.0 * math.pi * (turns - torch.floor(turns))
    return torch.polar(torch.ones_like(th), th)


def _intensity64(p, phi, lam):
    a = torch.fft.fft2(_field64(p, phi, lam))
    h = _h64(p, lam)
    a = torch.fft.ifft2(a * h[:, None] * h[None, :])
    return a.real ** 2 + a.imag ** 2


def _passband64(p, phi, lams, weights=None):
    w = np.full(len(lams), 1.0 / len(lams)) if weights is None else weights
    out = torch.zeros_like(phi)
    for lam, wl in zip(lams, w):
        out = out + float(wl) * _intensity64(p, phi, float(lam))
    return out


def _smooth64(p, inten):
    if p.source_radius_km <= 0:
        return inten
    n = p.n
    f = torch.fft.fftfreq(n, d=p.pixel_km, device="cuda", dtype=torch.float64)
    fx = torch.fft.rfftfreq(n, d=p.pixel_km, device="cuda", dtype=torch.float64)
    x = 2.0 * math.pi * p.source_radius_km * torch.sqrt(f[:, None] ** 2 + fx[None, :] ** 2)
    k = torch.where(x > 0, 2.0 * torch.special.bessel_j1(x) / x.clamp(min=1e-300), torch.ones_like(x))
    return torch.fft.irfft2(torch.fft.rfft2(inten) * k, s=(n, n))


def _curves64(inten, tracks, samples):
    n = inten.shape[0]
    tr = torch.as_tensor(np.asarray(tracks, dtype=np.float64), device=inten.device)
    d = torch.arange(samples, device=inten.device, dtype=torch.float64)[None, :] * tr[:, 3:4]
    x, y = tr[:, 0:1] + d * torch.cos(tr[:, 2:3]), tr[:, 1:2] + d * torch.sin(tr[:, 2:3])
    fx, fy = torch.floor(x), torch.floor(y)
    tx, ty = x - fx, y - fy
    ix, iy = torch.remainder(fx.long(), n), torch.remainder(fy.long(), n)
    jx, jy = (ix + 1) % n, (iy + 1) % n
    return ((1 - tx) * (1 - ty) * inten[iy, ix] + tx * (1 - ty) * inten[iy, jx]
            + (1 - tx) * ty * inten[jy, ix] + tx * ty * inten[jy, jx])


def _one_fft64(p, phi, lams):
    n = p.n
    i = torch.arange(n, device="cuda", dtype=torch.float64) - n // 2
    out = torch.zeros_like(phi)
    for lam in lams:
        lz = _lz(lam, p.z_pc)
        c = torch.polar(torch.ones_like(i), math.pi * (i * p.pixel_km) ** 2 / lz)
        g = _field64(p, phi, lam) * c[:, None] * c[None, :]
        a = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(g)))
        h = (a.real ** 2 + a.imag ** 2) * (p.pixel_km ** 2 / lz) ** 2
        u = i * (p.lambda_nm / lam) + n // 2
        f = torch.floor(u)
        t = u - f
        a0 = torch.remainder(f.long(), n)
        a1 = (a0 + 1) % n
        rows = (1 - t)[:, None] * h[a0] + t[:, None] * h[a1]
        out = out + ((1 - t)[None, :] * rows[:, a0] + t[None, :] * rows[:, a1]) / len(lams)
    return out


def _check64(p, lags):
    n, L = p.n, p.n * p.pixel_km
    bins = int(math.floor(math.sqrt(2.0 * (n // 2) ** 2) + 0.5)) + 1
    m = torch.round(torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) * n).long()
    sums = torch.zeros(bins, dtype=torch.float64, device="cuda")
    counts = torch.zeros(bins, dtype=torch.int64, device="cuda")
    for rows in _row_groups(n):
        F = _noise_rows(p, rows)
        j = torch.floor(torch.sqrt((m[rows][:, None] ** 2 + m[None, :] ** 2).to(torch.float64)) + 0.5).long().reshape(-1)
        sums += torch.bincount(j, weights=(F.real ** 2 + F.imag ** 2).reshape(-1), minlength=bins)
        counts += torch.bincount(j, minlength=bins)
    s = sums / counts.clamp(min=1) / (L * L)
    J = min(bins - 1, n // 2)
    q = torch.arange(1, J + 1, device="cuda", dtype=torch.float64) / L

    def d(r):
        return 4.0 * math.pi / L * (q * s[1:J + 1] * (1.0 - torch.special.bessel_j0(2.0 * math.pi * q * r))).sum()

    lo, hi = 0.0, 0.5 * L
    for _ in range(64):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float(d(mid)) < 1.0 else (lo, mid)
    return {"s_rec": s, "counts": None, "d_rec": torch.stack([d(float(r)) for r in lags]),
            "r_rec": torch.tensor([0.5 * (lo + hi)], dtype=torch.float64)}


def exact(case, seed):
    kind, seed = case["kind"], int(seed)
    st = _params(case, seed)
    p = st["p"][0]
    n = p.n
    if kind in ("screen", "plain64", "chain"):
        phi = _screen64(p)
        if kind == "screen":
            return {"phi": phi}
        inten = _intensity64(p, phi, p.lambda_nm)
        if kind == "plain64":
            return {"phi": phi, "intensity": inten}
        del phi
        inten = _smooth64(p, inten)
        return {"intensity": inten, "curves": _curves64(inten, st["tracks"][0], case["samples"])}
    if kind in ("point", "passband"):
        phi = _any_screen(n, p.pixel_km, p.r_diff_km, seed)
        lams = [p.lambda_nm] if kind == "point" else st["lams"]
        inten = _passband64(p, phi, lams, st.get("weights"))
        if kind == "passband":
            inten = _smooth64(p, inten)
        return {"intensity": inten, "curves": _curves64(inten, st["tracks"][0], case["samples"])}
    if kind in ("batch", "sweep"):
        maps, curves = {}, {}
        for i, q in enumerate(st["p"]):
            inten = _smooth64(q, _passband64(q, _screen64(q), st["lams"]))
            if kind == "batch":
                curves.setdefault(q.n, []).append(_curves64(inten, st["tracks"][i], q.n // 2))
            maps.setdefault(q.n, []).append(inten)
        return {"maps": [torch.stack(maps[m]) for m in sorted(maps)],
                "curves": [torch.stack(curves[m]) for m in sorted(curves)]}
    if kind == "fit":
        g = torch.Generator(device="cuda").manual_seed(seed)
        phis = [_any_screen(n, p.pixel_km, p.r_diff_km, seed + 7 * i) for i in range(case["count"])]
        deltas = [0.05 * torch.randn(n, n, generator=g, device="cuda") for _ in phis]
        targets = [1.0 + 0.3 * torch.randn(case["tracks"], case["samples"], generator=g, device="cuda") for _ in phis]
        out = {"curves": [], "loss": [], "grad": []}
        for i, q in enumerate(st["p"]):
            phi = (phis[i] + deltas[i]).requires_grad_()
            curves = _curves64(_smooth64(q, _passband64(q, phi, st["lams"])), st["tracks"][i], case["samples"])
            loss = ((curves - targets[i]) ** 2).mean()
            loss.backward()
            out["curves"].append(curves.detach())
            out["loss"].append(loss.detach())
            out["grad"].append(phi.grad)
        return out
    if kind == "one_fft":
        return {"intensity": _one_fft64(p, _any_screen(n, p.pixel_km, p.r_diff_km, seed), st["lams"])}
    if kind == "check":
        return _check64(p, st["lags"])
    pat = _any_pattern(n, seed).to(torch.float64)
    i0, i1 = _fiducial(p)
    zone = pat[i0:i1, i0:i1]
    mean, sd = zone.mean(), zone.std(unbiased=False)
    m = torch.stack([sd / mean, mean, sd, torch.tensor(float(zone.numel()), dtype=torch.float64, device="cuda")])
    curves = _curves64(pat, st["tracks"][0], case["samples"])
    cm, cs = curves.mean(1), curves.std(1, unbiased=False)
    power = torch.fft.rfft(curves - cm[:, None]).abs() ** 2 / case["samples"]
    x0, y0, th, ds = (st["pairs"][:, i] for i in range(4))
    sep = st["separations"]
    par = np.stack([x0[:, None] - sep[None, :] * np.sin(th)[:, None], y0[:, None] + sep[None, :] * np.cos(th)[:, None],
                    np.repeat(th[:, None], len(sep), 1), np.repeat(ds[:, None], len(sep), 1)], axis=2)
    c = _curves64(pat, par.reshape(-1, 4), case["samples"]).reshape(len(x0), len(sep), -1)
    c = c - c.mean(2, keepdim=True)
    corr = (c * c[:, :1]).sum(2) / torch.sqrt((c * c).sum(2) * (c[:, :1] ** 2).sum(2))
    return {"m": m, "curves": curves, "m_curves": torch.stack([cs / cm, cm, cs], 1), "power": power,
            "decorrelation": corr}


def _fiducial(p):
    n, L = p.n, p.n * p.pixel_km
    margin = (min(10.0 * math.sqrt(_lz(p.lambda_nm, p.z_pc) / (2.0 * math.pi)), L / 4.0)
              + 0.5 * _lz(p.lambda_nm, p.z_pc) / p.r_diff_km + p.source_radius_km)
    x = (np.arange(n) + 0.5) * p.pixel_km
    inside = np.nonzero((x >= margin) & (x <= L - margin))[0]
    return (int(inside[0]), int(inside[-1]) + 1) if inside.size else (0, n)
