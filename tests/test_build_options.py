"""The sources compile one way: no macro that a compiler flag could set chooses between forms of a kernel.

(The former SCINT_ROW_TWIDDLES=1 did not compile and SCINT_COL_TWIDDLES reached only a part of the column passes.)"""
import os
import re

from paper_1301_0514_gb300 import build


def test_sources_offer_no_build_options():
    found = []
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as f:
            found += [f"{name}:{i}: {line.strip()}" for i, line in enumerate(f, 1)
                      if re.match(r"\s*#\s*(if|ifdef|ifndef|elif)\b", line) and "__CUDA" not in line]
    assert found == []
