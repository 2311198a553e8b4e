"""The adjoint multiplies by the same transfer function as the forward passes.

Without a screen and without a taper the forward field is 1 everywhere.  Curves along every column with
dL/dcurve = sum_k cos(2 pi k y / n) then have the gradient -2 sum_k Im H_y(k) cos(2 pi k y / n) in every column
(constant along x, so that the row transforms are exact: k_x = 0 alone, where H_x = 1).  Projected on each cosine
it gives Im H_y(k) of the adjoint column pass, with the line transforms' rounding averaged over the line (the
column passes' twiddles are exactly rounded; the row passes' products of two bases bias a mode by up to 2e-7).

Tolerance per value: the forward columns evaluate H to FP32 accuracy: 6e-8 for the
rounding of the sine, as much for its evaluation in the last place, 6e-8 for the rounded angle and the products;
and 2 pi 2^-53 m^2 for the fixed-point constant of H.
The hardware sine over a whole turn, which the forward rows below 16384 use, is off by up to 4e-7.
"""
import math

import numpy as np
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu

H_TOL = 1.8e-7


@pytest.mark.parametrize("n", [16, 64, 512, 2048, 8192, 16384])
def test_adjoint_columns_take_the_forward_transfer_function(n):
    p = S.params(n, 10.0, 100.0, lambda_nm=550.0, margin_km=0.0, seed=1)
    rng = np.random.default_rng(n)
    modes = np.sort(rng.choice(np.arange(1, n // 2), size=min(64, n // 2 - 1), replace=False))
    waves = np.cos(2.0 * math.pi * (np.outer(modes, np.arange(n)) % n) / n)
    g = torch.from_numpy(waves.sum(axis=0).astype(np.float32)).cuda()[None].expand(n, n).contiguous()
    tracks = [(float(i), 0.0, 0.5 * math.pi, 1.0) for i in range(n)]
    grad = S.lightcurve_adjoint(p, torch.zeros(n, n, dtype=torch.float64, device="cuda"), [550.0], tracks, n, g)
    got = waves @ grad.mean(dim=1).cpu().numpy() * (2.0 / n) / 2.0
    # -Im H = sin(2 pi m^2 c), c = lambda z / (2 L^2), c m^2 by whole turns first
    c = 550.0e-12 * 160.0 * 3.0856775814913673e13 / (2.0 * (n * 10.0) ** 2)
    turns = c * modes.astype(np.float64) ** 2
    want = np.sin(2.0 * math.pi * (turns - np.floor(turns)))
    err = np.abs(got - want) - 2.0 * math.pi * 2.0 ** -53 * modes.astype(np.float64) ** 2
    assert err.max() <= H_TOL
