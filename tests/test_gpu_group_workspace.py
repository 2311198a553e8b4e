"""Workspaces without room for the transfer function's tables: as many wavelengths per group as with the tables
left out of account, and the same bits (the column blocks evaluate H_x themselves)."""
import numpy as np
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


def _up(b):
    return (b + 255) // 256 * 256


def _group_bytes(n, g):
    """Twiddles, tapers and fields of a group of g wavelengths."""
    slots = g if g == 1 else (g + 1) // 2 * 2
    return _up(n * 8) + _up(g * n * 4) + _up(slots * n * n * 8) + (_up(n * n * 4) if n >= 16384 else 0)


def _row_passes(call):
    S.profile_enable(True)
    call()
    torch.cuda.synchronize()
    rows = S.profile_read()["prop_rows"]["launches"]
    S.profile_enable(False)
    return rows


@pytest.fixture(autouse=True)
def one_wavelength_plans():
    sizes = (64, 256, 512, 1024, 2048, 4096, 8192)
    old = {n: S.get_plan(n) for n in sizes}
    for n in sizes:
        S.set_plan(n, 0)
    yield
    for n, pl in old.items():
        S.set_plan(n, pl["packed"], pl["row_twiddles"], pl["col_twiddles"], pl["points"])


@pytest.mark.parametrize("n,count", [(64, 5), (256, 2), (256, 9), (512, 2), (512, 9), (1024, 2), (1024, 5), (1024, 9),
                                     (2048, 2), (2048, 5), (2048, 9), (4096, 2), (4096, 5), (4096, 9), (8192, 2)])
def test_one_group_in_a_workspace_without_tables(n, count):
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi, lam = S.make_screen(p), np.linspace(500.0, 640.0, count)
    want = S.sum_passband(p, phi, lam)
    ws, out = torch.empty(_group_bytes(n, count), dtype=torch.uint8, device="cuda"), torch.empty_like(want)
    assert _row_passes(lambda: S.sum_passband(p, phi, lam, out=out, workspace=ws)) == 1
    assert torch.equal(out, want)
    buf = torch.empty(n * n + 1, device="cuda")[1:].view(n, n)    # narrow stores
    assert torch.equal(S.sum_passband(p, phi, lam, out=buf, workspace=ws), want)
    half = torch.empty(_group_bytes(n, (count + 1) // 2), dtype=torch.uint8, device="cuda")
    assert _row_passes(lambda: S.sum_passband(p, phi, lam, out=out, workspace=half)) == 2
    # each pixel's sum rounds once more per group
    assert (out - want).abs().max().item() <= count * 2.0 ** -23 * want.max().item()


@pytest.mark.parametrize("n,count", [(256, 5), (1024, 4)])
def test_one_group_of_the_adjoint(n, count):
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi, lam = S.make_screen(p), np.linspace(500.0, 640.0, count)
    track, g = np.array([[3.0, 5.0, 0.3, 0.7]]), torch.ones((1, 300), device="cuda")
    want = S.lightcurve_adjoint(p, phi, lam, track, 300, g)
    out = torch.empty_like(want)
    ws = torch.empty(_up(n * n * 4) + _up((n // 2 + 1) * n * 8) + _group_bytes(n, count), dtype=torch.uint8, device="cuda")
    assert _row_passes(lambda: S.lightcurve_adjoint(p, phi, lam, track, 300, g, out=out, workspace=ws)) == 1
    # the scatter's atomic additions come in any order: a few roundings of the largest sums
    assert (out - want).abs().max().item() <= 64 * 2.0 ** -23 * want.abs().max().item()
