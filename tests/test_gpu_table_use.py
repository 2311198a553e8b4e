"""The transfer function's tables are made for the passes that read them: the bytes that the table launch
accounts for are the tapers' alone for the packed plans and for the adjoint below 16384."""
import numpy as np
import pytest
import torch

import paper_1301_0514_gb300 as S

pytestmark = pytest.mark.gpu


def _table_bytes(call):
    S.profile_enable(True)
    call()
    torch.cuda.synchronize()
    b = S.profile_read()["prop_tables"]["bytes"]
    S.profile_enable(False)
    return b


@pytest.mark.parametrize("n", [256, 1024, 8192])
def test_table_bytes(n):
    lam = np.linspace(500.0, 600.0, 2)
    p = S.params(n=n, pixel_km=10.0, r_diff_km=60.0, lambda_nm=550.0, seed=5)
    phi, old = S.make_screen(p), S.get_plan(n)
    tapers = 4.0 * n * len(lam)
    entries = {256: 0, 1024: 514, 8192: 8192}[n]
    try:
        S.set_plan(n, 0)
        one = S.sum_passband(p, phi, lam)
        assert _table_bytes(lambda: S.sum_passband(p, phi, lam)) == tapers + 8.0 * entries * len(lam)
        if n == 1024:
            S.set_plan(n, 1, 2, 2, 16)
            assert _table_bytes(lambda: S.sum_passband(p, phi, lam)) == tapers
            # whole-turn hardware sines, once more per axis (the FP32 passes' bound, tests/test_gpu_parity.py)
            assert (S.sum_passband(p, phi, lam) - one).abs().max().item() <= 2e-4
    finally:
        S.set_plan(n, old["packed"], old["row_twiddles"], old["col_twiddles"], old["points"])
    g = torch.ones((1, 50), device="cuda")
    assert _table_bytes(lambda: S.lightcurve_adjoint(p, phi, lam, [[1.0, 2.0, 0.3, 1.0]], 50, g)) == tapers
