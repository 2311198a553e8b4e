"""Observables where their kernels change form: track counts around the two argument sizes, positions
around 2^19 pixels (fixed point below, FP64 above), zones and maps off the 16-byte grid, and curve
values that a bitwise widening does not cover (zeros, subnormals, infinities, NaN)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tracks", [1, 64, 65, 512, 513, 577])
def test_track_counts_and_far_positions(n_tracks):
    n, ns = 64, 37
    rng = np.random.default_rng(n_tracks)
    I = rng.uniform(0.0, 2.0, (n, n)).astype(np.float32)
    far = np.array([0.0, -0.5, 2.0 ** 19 - 3.0, -2.0 ** 19 + 3.25, 2.0 ** 19 + 0.125, -2.0 ** 20 - 7.5, 1e9 + 0.25])
    tr = np.stack([rng.choice(far, n_tracks) + rng.uniform(0.0, 4.0, n_tracks), rng.choice(far, n_tracks),
                   rng.uniform(0.0, 6.3, n_tracks), rng.uniform(0.1, 1.5, n_tracks)], axis=1)
    got = S.lightcurve(S.params(n=n, pixel_km=10.0, r_diff_km=100.0), torch.from_numpy(I).cuda(), tr, ns)
    want = O.lightcurves(I.astype(np.float64), tr, ns)
    # a few FP32 roundings of values up to 2, and of fractions (2^-24); 1e9 px positions resolve 2^-23 px
    assert np.abs(got.cpu().numpy() - want).max() <= 2e-6


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("margin_px", [0.0, 1.0, 2.5, 3.0, 30.25, 127.0])
def test_map_moments_off_the_grid(offset, margin_px):
    n = 256
    kw = dict(n=n, pixel_km=1.0, r_diff_km=1e9, lambda_nm=550.0, lambda_ref_nm=550.0, margin_km=margin_px)
    p, po = S.params(**kw), O.ScreenParams(**kw)
    buf = torch.empty(n * n + 1, device="cuda")[offset:offset + n * n].view(n, n)
    buf.copy_(torch.from_numpy(np.random.default_rng(3).uniform(0.5, 1.5, (n, n)).astype(np.float32)))
    got = S.modulation_index(p, buf).cpu().numpy()
    i0, i1, _ = O.fiducial_slice(po)
    z = buf.cpu().numpy().astype(np.float64)[i0:i1, i0:i1]
    np.testing.assert_allclose(got, [z.std() / z.mean(), z.mean(), z.std(), z.size], rtol=1e-6)


def test_correlation_of_unusual_values():
    rng = np.random.default_rng(4)
    a = rng.normal(1.0, 0.3, (1, 1000)).astype(np.float32)
    b = np.repeat(a, 5, axis=0) + rng.normal(0.0, 0.1, (5, 1000)).astype(np.float32)
    b[0, ::3] = 0.0
    b[1, ::2] = -0.0
    b[2, 5:50] = 1e-42                     # subnormal
    b[3, 7] = np.inf
    b[4, 7] = np.nan
    r = S.curve_correlation(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    np.testing.assert_allclose(r[:3], O.pearson(np.repeat(a, 3, axis=0), b[:3]), rtol=1e-12)
    assert np.isnan(r[3:]).all()
