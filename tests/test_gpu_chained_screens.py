"""Screens one after the other take no longer than their kernels do one by one."""
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


def test_chained_screens_of_1024():
    """66.6 us per screen in a graph, 74 for the two kernels between events; 76.5 when the passes were set up
    beside one another."""
    p = S.params(n=1024, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi = S.make_screen(p)
    ws = torch.empty(S.workspace_bytes(p, 1), dtype=torch.uint8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(20):
            S.make_screen(p, out=phi, workspace=ws)
    chained, alone = [], []
    for _ in range(10):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        b.synchronize()
        chained.append(a.elapsed_time(b) / 20)
        S.profile_enable(True)
        for _ in range(20):
            S.make_screen(p, out=phi, workspace=ws)
        torch.cuda.synchronize()
        alone.append(sum(k["total_ms"] for k in S.profile_read().values()) / 20)
        S.profile_enable(False)
    assert min(chained) < min(alone)
