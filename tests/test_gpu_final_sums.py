"""The homogenised stress of a solve is the volume average of the stress field it returns.

Both sum the same FP32 stresses in FP64, in different orders: N terms of at most the largest stress
are off by at most N 2^-53 of it each way, 2.4e-10 for 1024^2 voxels.
"""

import numpy as np
import pytest

import oracle as O
from synth import random_discs
from synth.configs import elastic_phases, j2_phases, k_target

pytestmark = pytest.mark.gpu

TOL = 1e-9


def off_average(s, out):
    """Distance of the homogenised stress from the average of the stress field, relative."""
    _, sig, _ = s.rf_get_fields()
    mean = sig.reshape(6, -1).mean(axis=1, dtype=np.float64)
    return np.abs(out - mean).max() / np.abs(sig).max()


def test_first_solve_after_the_tuner_timed_every_persistent_form(lib):
    """Default options on 1024 x 1024: the tuner launches each persistent solve before the first
    final pass, which must not take over anything that they leave behind."""
    pm = random_discs(1024, (8.0, 24.0), 0.4, seed=21)
    pat = O.pattern_adapted(pm, 1, k_target(0.01, pm.size))
    s = lib.Solver(pm, j2_phases(), pattern=pat, tol=0.0, max_iter=4, transform="fft")
    macro = np.array([0.012, -0.004, 0, 0, 0, 0.003])
    for _ in range(2):
        assert off_average(s, s.rf_solve(macro)["sigma_bar"]) <= TOL
    out = s.rf_solve_path(macro * np.array([0.5, 1.0])[:, None])
    assert off_average(s, out["sigma_bar"][-1]) <= TOL
    s.close()


@pytest.mark.parametrize("nx", [48, 64, 96, 192, 384])
@pytest.mark.parametrize("plastic", [False, True])
def test_3d_final_pass(lib, nx, plastic):
    """Rows whose teams do not fill their last warp (48, 96, 192, 384), and one that does."""
    shape = (64, 64, nx)
    pm = np.zeros(shape, np.uint8)
    pm[10:40, 5:50, 3:nx // 2] = 1
    pat = O.pattern_adapted(pm, 1, k_target(0.02, pm.size))
    s = lib.Solver(pm, j2_phases() if plastic else elastic_phases(), pattern=pat, tol=0.0,
                   max_iter=3, transform="fft")
    s.rf_set_tracing(True)
    out = s.rf_solve(np.array([0.015, -0.004, 0.002, 0.001, 0.003, -0.002]))
    assert s.rf_get_stage_times()["column_phase"][1] == 3   # the updates on team FFTs ran
    assert off_average(s, out["sigma_bar"]) <= TOL
    s.close()
