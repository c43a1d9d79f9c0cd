"""Selection of the adapted pattern at the sizes where a digit of |k|^2 or of the linear index begins
to matter, against the oracle, exactly. One inclusion voxel: all amplitudes tie, so |k|^2 and the
index decide."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 2), (3, 3), (32, 32), (33, 32), (63, 63), (64, 64),
                                   (1, 4095), (1, 4096), (4096, 2), (1024, 1024), (1025, 1024),
                                   (16, 8, 8), (5, 11, 19), (65, 64, 64)])
@pytest.mark.parametrize("tied", [True, False])
def test_every_digit(lib, shape, tied):
    rng = np.random.default_rng(sum(shape))
    pm = np.zeros(shape, np.uint8)
    if not tied:
        pm[:] = rng.random(shape) < 0.4
    pm.flat[pm.size // 2] = 1
    for k in sorted({1, max(1, pm.size // 23), max(1, pm.size // 3)}):
        got = lib.rf_pattern_adapted(pm, 1, k)
        assert np.array_equal(got, O.pattern_adapted(pm, 1, k)), (shape, k)
