"""Lags of Eq. crec: one block per lag or a cluster of them (few lags, many terms), the same bits either way."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu

N, PIX = 4200, 10.0


def _spectrum(J):
    q = np.arange(J + 1) / (N * PIX)
    s = np.zeros_like(q)
    s[1:] = O.phase_spectrum(q[1:], 60.0, 11.0 / 3.0)
    return s


@pytest.mark.parametrize("J", [1, 255, 256, 257, 512, 513, 1025, 2048, 2100])
def test_lags_alone_and_among_many(J):
    s = _spectrum(J)
    sd, p = torch.from_numpy(s).cuda(), S.params(n=N, pixel_km=PIX, r_diff_km=60.0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    r = np.geomspace(1.0, 0.4 * N * PIX, 3 * sms)
    few, many = sms * 2 // 3, len(r)
    d, _ = S.structure_function_rec(p, sd, r, root=False)
    for count in (1, few, few + 1, many):
        part, _ = S.structure_function_rec(p, sd, r[:count], root=False)
        assert torch.equal(part, d[:count]), count
    want = O.structure_function_rec(s, N, PIX, r[::37])
    np.testing.assert_allclose(d.cpu().numpy()[::37], want, rtol=1e-12, atol=1e-12 * want.max())


def test_many_short_lags_take_a_block_each():
    """20000 lags of 8 terms: 0.14 ms with a block per lag, 1.07 ms with a cluster of eight."""
    p = S.params(n=16, pixel_km=PIX, r_diff_km=60.0)
    s = torch.ones(9, dtype=torch.float64, device="cuda")
    r = torch.linspace(1.0, 50.0, 20000, dtype=torch.float64, device="cuda")
    d, t = torch.empty_like(r), []
    for _ in range(10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        S.structure_function_rec(p, s, r, root=False, out=(d, None))
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b))
    assert min(t) < 0.5
