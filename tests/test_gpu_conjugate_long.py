"""One-FFT patterns on 8192-point lines (two half lines per team) are as accurate as on whole lines.

Bound: the rms error of these calls, relative to the pattern's rms, when the lines were whole (sixteen values of
512 threads, twiddles of depth 3 at the most): 3.80e-7 at one wavelength and 3.30e-7 over three, the same to 0.3 %
for any screen.  With every factor of the half lines' first step rounded three times it was 3.86e-7 and 3.41e-7.
"""
import math

import numpy as np
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu

N = 8192
KM = 1.0e-12 * 160.0 * 3.0856775814913673e13    # lambda z in km^2 per nm at 160 pc


def _screen(pixel, r_diff, seed):
    """Gaussian phases with the Kolmogorov spectrum, FP64."""
    beta = 11.0 / 3.0
    g = torch.Generator(device="cuda").manual_seed(seed)
    k = torch.fft.fftfreq(N, d=pixel, device="cuda", dtype=torch.float64)
    kx = torch.fft.rfftfreq(N, d=pixel, device="cuda", dtype=torch.float64)
    q2 = k[:, None] ** 2 + kx[None, :] ** 2
    q2[0, 0] = 1.0
    fb = 2.0 ** (-beta) * beta * math.gamma(-beta / 2.0) / math.gamma(beta / 2.0)
    c = r_diff ** 2 / (2.0 * (2.0 * math.pi) ** (beta - 1.0) * fb)
    amp = math.sqrt(c) * (r_diff * r_diff * q2) ** (-beta / 4.0) / (N * pixel)
    amp[0, 0] = 0.0
    w = torch.view_as_complex(torch.randn(N, N // 2 + 1, 2, generator=g, device="cuda", dtype=torch.float64))
    return torch.fft.irfft2(w * (amp * math.sqrt(0.5)), s=(N, N)) * float(N) * float(N)


def _exact(p, phi, lams):
    i = torch.arange(N, device="cuda", dtype=torch.float64) - N // 2
    x = (i + N // 2 + 0.5) * p.pixel_km
    length = N * p.pixel_km
    out = torch.zeros_like(phi)
    for lam in lams:
        lz = lam * KM
        margin = min(10.0 * math.sqrt(lz / (2.0 * math.pi)), length / 4.0)
        u = torch.minimum(x, length - x)
        sf = torch.where(u <= margin, torch.sin(math.pi * u / (2.0 * margin)) ** 2, torch.ones_like(u))
        c = torch.polar(sf, math.pi * (i * p.pixel_km) ** 2 / lz)
        a = torch.polar(torch.ones_like(phi), phi * (p.lambda_ref_nm / lam)) * c[:, None] * c[None, :]
        a = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(a)))
        h = (a.real ** 2 + a.imag ** 2) * (p.pixel_km ** 2 / lz) ** 2
        s = i * (p.lambda_nm / lam) + N // 2
        f = torch.floor(s)
        t = s - f
        a0 = torch.remainder(f.long(), N)
        a1 = (a0 + 1) % N
        rows = (1 - t)[:, None] * h[a0] + t[:, None] * h[a1]
        out += ((1 - t)[None, :] * rows[:, a0] + t[None, :] * rows[:, a1]) / len(lams)
    return out


@pytest.mark.parametrize("count,bound", [(1, 3.80e-7), (3, 3.30e-7)])
def test_one_fft_patterns_are_as_accurate_as_on_whole_lines(count, bound):
    p = S.params(N, math.sqrt(2162.0 * KM / N), 500.0, lambda_nm=2162.0, seed=1)
    phi = _screen(p.pixel_km, p.r_diff_km, 1)
    lams = np.linspace(2080.0, 2280.0, count) if count > 1 else np.array([2180.0])
    got = S.sum_passband_conjugate(p, phi, lams).double()
    exact = _exact(p, phi, lams)
    assert ((got - exact).square().mean().sqrt() / exact.square().mean().sqrt()).item() <= bound
