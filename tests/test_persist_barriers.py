"""Named barriers of the persistent batch kernel, from the sizes its bodies are compiled with (no GPU): a
barrier that two groups of threads use without a block barrier between them may release early or never."""
import ctypes

import pytest

import paper_1301_0514_gb300 as S

BLOCK = 512


@pytest.mark.parametrize("n", [256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("which", [0, 1])
def test_every_barrier_of_an_item_has_one_group_of_threads(n, which):
    parts = (ctypes.c_int * 2)()
    k = S.lib().scint_testing_persist_parts(n, which, parts)
    owner = {}
    for size in parts[:k]:
        assert size % 32 == 0 and BLOCK % size == 0
        for i in range(BLOCK // size):
            threads = range(i * size, (i + 1) * size)
            assert owner.setdefault(1 + i, threads) == threads, (list(parts[:k]), 1 + i)
    assert max(owner, default=0) <= 15
