"""What the decorrelation refuses, before anything is launched (no GPU)."""
import pytest
import torch

import paper_1301_0514_gb300 as S
from paper_1301_0514_gb300 import timeseries as TS

TRACK = [1.0, 2.0, 0.3, 1.0]


@pytest.mark.parametrize("tracks,separations,message", [([], [0.0, 1.0], "at least one track"),
                                                        ([TRACK], 5.0, "a list of separations"),
                                                        ([TRACK], [[0.0, 1.0]], "a list of separations"),
                                                        ([TRACK, TRACK], [[0.0, 1.0], [2.0, 3.0]], "a list of separations")])
def test_refused(tracks, separations, message):
    p = S.params(n=64, pixel_km=10.0, r_diff_km=60.0)
    with pytest.raises(ValueError, match=message):
        TS.decorrelation(p, torch.zeros((64, 64)), tracks, separations, 16)
