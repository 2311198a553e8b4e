"""The FP64 square of the screen check's octant, at every number of lanes per cell, against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu

S_TOL = 2e-6      # the bound of the other grids (tests/test_gpu_screen_check.py)


# the square's half side: n/2 up to 512; at 1024 and r_diff 300, 90, 20 km it is 32, 32 to 64, 128 to 256
@pytest.mark.parametrize("n,rd", [(16, 90.0), (180, 90.0), (182, 90.0), (310, 90.0), (314, 90.0), (358, 90.0), (364, 90.0),
                                  (510, 90.0), (1024, 300.0), (1024, 90.0), (1024, 20.0), (1026, 5.0)])
def test_square_cells_match_the_oracle(n, rd):
    kw = dict(n=n, pixel_km=10.0, r_diff_km=rd, seed=20130514 + 9000, screen_id=4)
    s, c = S.spectrum_rec(S.params(**kw))
    s_o, c_o = O.spectrum_rec(O.ScreenParams(**kw))
    assert torch.equal(c.cpu(), torch.from_numpy(c_o.astype(np.int64)))
    np.testing.assert_allclose(s.cpu().numpy(), s_o, rtol=S_TOL, atol=0.0)
    few, _ = S.spectrum_rec(S.params(**kw), n_bins=5)
    assert torch.equal(few, s[:5])


def test_small_spectra_do_not_wait_for_one_chain_of_logarithms():
    """16^2: 20 us with the draws of a cell over eight lanes, 68 us with four cells' draws on one lane."""
    p = S.params(n=16, pixel_km=10.0, r_diff_km=90.0)
    out = (torch.empty(12, dtype=torch.float64, device="cuda"), torch.empty(12, dtype=torch.int64, device="cuda"))
    t = []
    for _ in range(10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            S.spectrum_rec(p, out=out)
        b.record()
        b.synchronize()
        t.append(a.elapsed_time(b) / 10)
    assert min(t) < 0.045
