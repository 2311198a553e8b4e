"""The plain method in FP64 on the smallest grids (lines of 16 to 64 points, with plans of their own)
against the FP64 oracle, and under a capture that finds no kept twiddle table."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1301_0514_gb300 as S
from paper_1301_0514_gb300 import workloads as W
from conftest import gpu_params, oracle_params

pytestmark = pytest.mark.gpu

TOL64 = 1e-10      # the bound of the larger grids (tests/test_gpu_fp64.py)


@pytest.mark.parametrize("n", [16, 32, 64])
@pytest.mark.parametrize("margin", [-1.0, 0.0])
def test_smallest_grids_match_the_oracle(n, margin):
    it = W._item(n, 20.0, 60.0, margin_km=margin, seed=W.SEED_BASE + 65 + n)
    p_g, p_o = gpu_params(it), oracle_params(it)
    phi = O.make_screen(p_o)
    want = O.intensity_mono(phi, p_o)
    phi_g = torch.from_numpy(phi).cuda()
    got = S.propagate64(p_g, phi_g)
    assert np.abs(got.cpu().numpy() - want).max() <= TOL64 * max(1.0, np.abs(want).max() / 10.0)
    # twiddles in the workspace, H and the taper in the passes: the same bits
    ws = torch.empty(S.workspace_bytes(p_g, 1), dtype=torch.uint8, device="cuda")
    out = torch.zeros((n, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    S.release()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        S.propagate64(p_g, phi_g, out=out, workspace=ws)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, got)
