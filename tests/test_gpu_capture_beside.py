"""A call that makes its twiddle table while a capture is open on another stream, in the same thread or
another, leaves the capture whole (torch captures in global mode) and gives the usual bits."""
import threading

import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_thread", [False, True])
@pytest.mark.parametrize("call,dtype", [(S.propagate64, torch.float64), (S.propagate, torch.float32)])
def test_first_call_beside_an_open_capture(call, dtype, own_thread):
    n = 256
    p = S.params(n=n, pixel_km=20.0, r_diff_km=100.0, seed=7)
    phi = S.make_screen(p)
    ws = torch.empty(S.workspace_bytes(p, 1), dtype=torch.uint8, device="cuda")
    out, x = torch.zeros((n, n), dtype=dtype, device="cuda"), torch.zeros(4, device="cuda")
    side = torch.cuda.Stream()
    want = call(p, phi)
    torch.cuda.synchronize()
    S.release()
    errors = []

    def first_call():
        try:
            call(p, phi, out=out, workspace=ws, stream=side)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        x.add_(1.0)
        if own_thread:
            t = threading.Thread(target=first_call)
            t.start()
            t.join()
        else:
            first_call()
        x.add_(1.0)
    torch.cuda.synchronize()
    assert not errors
    assert torch.equal(out, want)
    x.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert x.tolist() == [2.0] * 4
