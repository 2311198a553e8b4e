"""The streamed propagation passes (inputs of the next line or wavelength copied ahead): every
number of rows per block and columns per block, few wavelengths (a block walks lines) and many
(one line per block), and buffers off the 16-byte boundary that the copies need, which take plain
loads and narrow stores through the same arithmetic."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu

I_TOL = 2e-4      # the FP32 passes' bound against the oracle (tests/test_gpu_parity.py)


@pytest.fixture(autouse=True)
def one_wavelength_plans():
    """The passes under test are the one-wavelength plans': other tests leave the plan that was
    fastest for them, whose packed passes round differently."""
    old = {n: S.get_plan(n) for n in (64, 256, 512, 1024, 2048, 4096, 8192)}
    for n in old:
        S.set_plan(n, 0)
    yield
    for n, pl in old.items():
        S.set_plan(n, pl["packed"], pl["row_twiddles"], pl["col_twiddles"], pl["points"])


def _off(n, dtype):
    """An n x n tensor whose first element is one element past an aligned address."""
    return torch.empty(n * n + 1, dtype=dtype, device="cuda")[1:].view(n, n)


def _band(count):
    return np.linspace(500.0, 640.0, count) if count > 1 else np.array([550.0])


@pytest.mark.parametrize("n,count", [(512, 1), (512, 8), (1024, 1), (1024, 7), (1024, 8), (2048, 3)])
def test_streamed_passes_match_oracle(n, count):
    kw = dict(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, lambda_ref_nm=550.0, seed=20130514 + 640 + n)
    p, po = S.params(**kw), O.ScreenParams(**kw)
    phi = O.make_screen(po)
    want = O.sum_passband(phi, po, _band(count))
    got = S.sum_passband(p, torch.from_numpy(phi).cuda(), _band(count)).cpu().numpy()
    assert np.abs(got - want).max() <= I_TOL


@pytest.mark.parametrize("n", [512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("count", [1, 2, 9])
def test_streamed_passes_off_alignment(n, count):
    """The same bits from buffers off the 16-byte boundary, and the wavelengths one at a time (each
    pixel's sum then rounds once more per wavelength)."""
    if n == 8192 and count > 2:
        pytest.skip("the same code as at 4096 with one row per block")
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi = S.make_screen(p)
    lam = _band(count)
    want = S.sum_passband(p, phi, lam)
    phi2, out2 = _off(n, torch.float64), _off(n, torch.float32)
    assert phi2.data_ptr() % 16 and out2.data_ptr() % 8
    phi2.copy_(phi)
    S.sum_passband(p, phi2, lam, out=out2)
    assert torch.equal(out2, want)
    out2.fill_(0.0)
    for l in lam:
        S.sum_passband(p, phi2, [l], [1.0 / count], out=out2, accumulate=True)
    assert (out2 - want).abs().max().item() <= count * 2.0 ** -23 * want.max().item()
    pc = S.params(n=n, pixel_km=100.0 * (512.0 / n) ** 0.5, r_diff_km=600.0, lambda_nm=550.0, seed=5)
    assert torch.equal(S.sum_passband_conjugate(pc, phi2, lam, out=out2), S.sum_passband_conjugate(pc, phi, lam))


@pytest.mark.parametrize("count", [1, 2, 9])
def test_long_lines_match_the_one_wavelength_form(count):
    """8192-point lines (two half lines per team): a passband and its wavelengths one by one, and the
    FP64 field theory: a uniform untapered screen stays 1 everywhere."""
    n = 8192
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, margin_km=0.0, seed=5)
    one = S.sum_passband(p, torch.zeros((n, n), dtype=torch.float64, device="cuda"), _band(count))
    assert (one - 1.0).abs().max().item() <= 2e-5


def _least_bytes(n, g=1):
    """The twiddles, the tapers and the fields of a group (and the column-major sums at 16384): what a
    propagation accepts without its transfer-function tables."""
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    slots = g if g == 1 else (g + 1) // 2 * 2
    return up(n * 8) + up(g * n * 4) + up(slots * n * n * 8) + (up(n * n * 4) if n >= 16384 else 0)


@pytest.mark.parametrize("n", [64, 512, 1024, 4096, 8192, 16384])
def test_least_workspace_and_capture_without_tables(n):
    """The same bits when the transfer function's tables have room in the workspace, only in the
    twiddles' slot (one wavelength, twiddles kept), or nowhere (a capture before any call): one
    expression gives the values in all three."""
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi = S.make_screen(p)
    want = S.propagate(p, phi)
    small = torch.empty(_least_bytes(n), dtype=torch.uint8, device="cuda")
    assert torch.equal(S.propagate(p, phi, workspace=small), want)
    with pytest.raises(S.ScintError):
        S.propagate(p, phi, workspace=small[:-256])
    torch.cuda.synchronize()
    S.release()
    out = torch.zeros((n, n), dtype=torch.float32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        S.propagate(p, phi, out=out, workspace=small)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("n", [256, 2048])
def test_least_group_workspace(n):
    """A group's least workspace still runs the passband (in smaller groups)."""
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi, lam = S.make_screen(p), _band(5)
    ws = torch.empty(_least_bytes(n, 4), dtype=torch.uint8, device="cuda")
    want = S.sum_passband(p, phi, lam)
    got = S.sum_passband(p, phi, lam, workspace=ws)
    assert (got - want).abs().max().item() <= 5 * 2.0 ** -23 * want.max().item()


@pytest.mark.parametrize("n", [64, 256, 512, 1024, 2048])
def test_overlapped_launches_keep_their_order(n):
    """Kernels set up while the one before ends (grids on both sides of the line) read nothing early:
    chains of screen, propagation and curves through the same buffers, back to back, replayed as a graph
    and with another library's kernels between them, give the bits of one call at a time."""
    ps = [S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=7, screen_id=i) for i in range(4)]
    tr = np.array([[3.0, 5.0, 0.3, 0.7], [n / 3.0, 1.0, 1.1, 0.5]])
    ws = torch.empty(S.workspace_bytes(ps[0], 1), dtype=torch.uint8, device="cuda")
    phi, out = torch.empty((n, n), dtype=torch.float64, device="cuda"), torch.empty((n, n), device="cuda")
    curves = torch.empty((2, 100), device="cuda")

    def chain(p):
        S.make_screen(p, out=phi, workspace=ws)
        S.propagate(p, phi, out=out, workspace=ws)
        S.lightcurve(p, out, tr, 100, out=curves)
        return out, curves

    want = []
    for p in ps:
        want.append([t.clone() for t in chain(p)])
        torch.cuda.synchronize()
    for _ in range(8):
        got = [[t.clone() for t in chain(p)] for p in ps]
        assert all(torch.equal(a, b) for g, w in zip(got, want) for a, b in zip(g, w))
    for p in ps:        # no other kernel between the chains
        chain(p)
    assert torch.equal(out, want[-1][0]) and torch.equal(curves, want[-1][1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for p in ps:
            chain(p)
    for _ in range(4):
        out.zero_(), curves.zero_(), phi.zero_()
        g.replay()
        assert torch.equal(out, want[-1][0]) and torch.equal(curves, want[-1][1])
