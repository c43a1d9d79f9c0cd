"""Which kernels a 3D FFT solve runs on: the updates on team FFTs wherever the three sides have a plan
and nothing is pinned, whatever the pattern."""

import numpy as np
import pytest

from synth.configs import elastic_phases, j2_phases

pytestmark = pytest.mark.gpu


def ran(lib, shape, pat, phases, **opts):
    """Updates of the z phase (stage "column_phase" is theirs alone in 3D) of a traced solve."""
    pm = np.zeros(shape, np.uint8)
    pm[:shape[0] // 2, :, :shape[2] // 2] = 1
    s = lib.Solver(pm, phases, pattern=pat, tol=0.0, max_iter=2, transform="fft", **opts)
    s.rf_set_tracing(True)
    s.rf_solve(np.array([0.01, 0, 0, 0.002, 0, 0]))
    n = s.rf_get_stage_times()["column_phase"][1]
    s.close()
    return n


WAVES = np.array([[-1, 0, 0], [0, -1, 0], [0, 0, -1], [0, 0, 0], [0, 0, 1], [0, 1, 0], [1, 0, 0]],
                 np.int32)


@pytest.mark.parametrize("shape", [(32, 48, 64), (48, 96, 32), (96, 64, 48), (32, 32, 192),
                                   (32, 32, 384), (32, 512, 32), (256, 32, 128)])
@pytest.mark.parametrize("plastic", [False, True])
def test_team_updates_run(lib, shape, plastic):
    ph = j2_phases() if plastic else elastic_phases()
    assert ran(lib, shape, WAVES, ph) == 2
    assert ran(lib, shape, WAVES[3:4], ph) == 2


def test_pinned_and_other_sides_keep_the_general_kernels(lib):
    ph = elastic_phases()
    assert ran(lib, (32, 32, 32), WAVES, ph, fft_fuse=-1) == 0
    assert ran(lib, (32, 32, 32), WAVES, ph, fft_rows=2) == 0
    assert ran(lib, (32, 32, 32), WAVES, ph, fft_cols=4) == 0
    assert ran(lib, (16, 32, 32), WAVES, ph) == 0
