"""Which kernels a solve on team FFTs runs on. 3D: the team updates wherever the three sides have a plan
and nothing is pinned, whatever the pattern. Persistent 2D solve: each of its forms, asked for.

Tolerances as in test_gpu_parity.py: fields 1e-5, homogenised stress 1e-6.
"""

import numpy as np
import pytest

import oracle as O
from oracle.rf_oracle import VOIGT
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


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("shape,forms", [((32, 32), (0, 8, 16)), ((48, 48), (0, 8, 16)),
                                         ((64, 64), (0, 8, 16)), ((96, 96), (0, 8, 16)),
                                         ((128, 128), (0, 8, 16)), ((192, 192), (0, 16)),
                                         ((32, 192), (0, 8, 16)), ((128, 48), (0, 8, 16)),
                                         ((256, 256), (0,)), ((512, 512), (0,)), ((768, 768), (0,))])
@pytest.mark.parametrize("plastic", [False, True])
def test_forms_of_the_persistent_solve(lib, shape, forms, plastic):
    """Clusters of 8 and 16 blocks and the co-resident grid: two increments (the second one reads what
    the first committed), the form from the block count that the context reports. 0: the grid, asked
    for by a row per block."""
    rng = np.random.default_rng(sum(shape))
    pm = np.zeros(shape, np.uint8)
    for _ in range(4):
        y, x = rng.integers(0, shape[0]), rng.integers(0, shape[1])
        pm[np.ix_(np.arange(y, y + shape[0] // 3) % shape[0],
                  np.arange(x, x + shape[1] // 3) % shape[1])] = 1
    ph = j2_phases() if plastic else elastic_phases()
    pat = O.pattern_adapted(pm, 1, max(5, pm.size // 40))
    path = np.zeros((2, 6))
    path[:, 0], path[:, 1], path[:, 5] = [0.008, 0.013], [-0.002, -0.004], [0.001, 0.002]
    ref = None
    for blocks in forms:
        s = lib.Solver(pm, ph, pattern=pat, tol=1e-2, max_iter=60, transform="fft", fft_fuse=3,
                       fft_row_blocks=blocks or shape[0])
        out = s.rf_solve_path(path)
        eps, sig, _ = s.rf_get_fields()
        info = s.rf_get_info()
        s.close()
        assert info["fft_fused"] == 3
        if blocks:
            assert info["fft_row_blocks"] == blocks
        if ref is None or not np.array_equal(ref[0], out["iters"]):
            ref = (out["iters"],) + O.solve_path(pm, ph, path, pat, fixed_iters=out["iters"])
        _, sbar, _, r = ref
        for n in range(2):
            assert rel(out["sigma_bar"][n], sbar[n]) <= 1e-6
        f = np.stack([r.eps[..., i, j] for (i, j) in VOIGT]).reshape(eps.shape)
        assert rel(eps, f) <= 1e-5
