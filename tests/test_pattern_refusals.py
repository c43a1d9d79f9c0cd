"""Targets that the adapted pattern refuses cost no memory (no GPU: they are refused before it)."""

import tracemalloc

import numpy as np
import pytest


@pytest.mark.parametrize("k_target", [65, 10 ** 8, 10 ** 12])
def test_target_beyond_the_grid(k_target):
    from paper_2103_10203_gb300.build import build
    build()
    from paper_2103_10203_gb300 import rf
    tracemalloc.start()
    with pytest.raises(rf.RFError) as e:
        rf.rf_pattern_adapted(np.ones((8, 8), np.uint8), 1, k_target)
    peak = tracemalloc.get_traced_memory()[1]
    tracemalloc.stop()
    assert e.value.code == -1
    assert peak < 1 << 22
