"""8192-point lines (two half lines per team) on a real screen: a passband is the weighted sum of its wavelengths
one by one, with and without room for the transfer function's tables, and each is the 64-bit propagation.

Tolerances: against the sum of single calls the order of the FP32 additions differs, at most 2^-24 of the
sum so far per wavelength on either side, and the single calls round each product; against 64 bits the library's 2e-4 of the mean intensity
(a wrong factor or a swapped pair of frequencies is off by its own size).
"""
import numpy as np
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu
N = 8192


@pytest.fixture(scope="module")
def screen():
    p = S.params(N, 10.0, 100.0, lambda_nm=550.0, seed=11)
    return p, S.make_screen(p)


def _intensity64(p, phi, lam):
    lz = lam * 1.0e-12 * p.z_pc * 3.0856775814913673e13
    length = p.n * p.pixel_km
    margin = min(10.0 * np.sqrt(lz / (2.0 * np.pi)), length / 4.0)
    x = (torch.arange(p.n, device="cuda", dtype=torch.float64) + 0.5) * p.pixel_km
    u = torch.minimum(x, length - x)
    sf = torch.where(u <= margin, torch.sin(np.pi * u / (2.0 * margin)) ** 2, torch.ones_like(u))
    f = torch.fft.fftfreq(p.n, d=p.pixel_km, device="cuda", dtype=torch.float64)
    turns = 0.5 * lz * f * f
    h = torch.polar(torch.ones_like(f), -2.0 * np.pi * (turns - torch.floor(turns)))
    a = torch.polar(sf[:, None] * sf[None, :], phi * (p.lambda_ref_nm / lam))
    a = torch.fft.ifft2(torch.fft.fft2(a) * h[:, None] * h[None, :])
    return a.real ** 2 + a.imag ** 2


@pytest.mark.parametrize("count", [2, 9])
@pytest.mark.parametrize("tables", [True, False])
def test_passband_is_the_sum_of_its_wavelengths(screen, count, tables):
    p, phi = screen
    lams = np.linspace(430.0, 690.0, count)
    w = np.linspace(1.0, 2.0, count)
    w /= w.sum()
    # the fields (an even number), the tapers and the twiddles, and no room for the transfer function's tables besides
    least = 8 * N * N * ((count + 1) // 2 * 2) + 4 * N * count + 8 * N
    ws = None if tables else torch.empty(least, dtype=torch.uint8, device="cuda")
    got = S.sum_passband(p, phi, lams, w, workspace=ws)
    one = torch.zeros_like(got)
    for lam, wl in zip(lams, w):
        S.sum_passband(p, phi, [lam], [wl], out=one, accumulate=True)
    assert ((got - one).abs() <= (2 * count + 2) * 2.0 ** -24 * one).all()
    exact = sum(wl * _intensity64(p, phi, lam) for lam, wl in zip(lams, w))
    assert (got - exact).abs().max().item() <= 2e-4 * exact.mean().item()
