"""A curve right behind a pass that adds to the map in place, and the FP64 passes right behind their tables: what
the kernel before wrote is what the next one reads, without a synchronisation between them."""
import numpy as np
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 256, 512, 1024])
def test_curves_behind_accumulating_passes(n):
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi, lam = S.make_screen(p), [520.0, 560.0, 600.0, 640.0]
    ws = torch.empty(S.workspace_bytes(p, 1), dtype=torch.uint8, device="cuda")
    tracks = np.stack([np.linspace(0.0, n, 8, endpoint=False), np.full(8, 1.5), np.full(8, 0.4), np.full(8, 0.9)], axis=1)
    out = torch.zeros((n, n), device="cuda")

    def chain(wait):
        curves = [torch.empty((8, n), device="cuda") for _ in lam]
        out.zero_()
        for l, c in zip(lam, curves):
            S.sum_passband(p, phi, [l], [0.25], out=out, accumulate=True, workspace=ws)
            wait()
            S.lightcurve(p, out, tracks, n, out=c)
            wait()
        return curves

    want = chain(torch.cuda.synchronize)
    for _ in range(20):
        got = chain(lambda: None)
        assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("n", [64, 256, 512])
def test_fp64_passes_behind_their_tables(n):
    ps = [S.params(n=n, pixel_km=pix, r_diff_km=100.0, seed=7) for pix in (20.0, 15.0, 10.0)]
    phi = S.make_screen(ps[0])
    ws = torch.empty(S.workspace_bytes(ps[0], 1), dtype=torch.uint8, device="cuda")
    want = []
    for p in ps:
        want.append(S.propagate64(p, phi, workspace=ws))
        torch.cuda.synchronize()
    for _ in range(20):
        got = [S.propagate64(p, phi, workspace=ws) for p in ps]
        assert all(torch.equal(a, b) for a, b in zip(got, want))
