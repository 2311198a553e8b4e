"""Correlation of curves of every remainder (four samples of a thread at a time, then one by one)."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 255, 256, 257, 768, 769, 1023, 1024, 1025, 1793, 4096, 4097])
def test_lengths_match_oracle(n):
    rng = np.random.default_rng(n)
    a = (1.0 + rng.standard_normal((2, n))).astype(np.float32)
    b = (0.5 * np.repeat(a, 3, 0) + rng.standard_normal((6, n))).astype(np.float32)
    r = S.curve_correlation(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()).cpu().numpy()
    # FP64 sums of O(1) values, each rounded to 2^-53: 1e-12 absolute leaves three orders
    np.testing.assert_allclose(r, O.pearson(np.repeat(a, 3, 0).astype(np.float64), b.astype(np.float64)), rtol=0, atol=1e-12)


def test_short_curves_cost_less_than_long_ones():
    """256 samples are a quarter of 1024: with additions of zeros for the rest both took the same time."""
    def time(n):
        a, b = torch.rand((10000, n), device="cuda"), torch.rand((10000, n), device="cuda")
        r, t = torch.empty(10000, dtype=torch.float64, device="cuda"), []
        for _ in range(10):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            S.curve_correlation(a, b, out=r)
            e1.record()
            e1.synchronize()
            t.append(e0.elapsed_time(e1))
        return min(t)

    assert time(256) < 0.85 * time(1024)
