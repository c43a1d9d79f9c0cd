"""The J2 law at strains whose stress invariant overflows FP32: an elastic phase stays elastic."""

import numpy as np
import pytest

from synth.configs import j2_phases

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [32, 40, 1024])
@pytest.mark.parametrize("transform", ["fft", "dft"])
def test_elastic_phase_beside_j2_at_huge_strain(lib, side, transform):
    if transform == "fft" and side == 40 or transform == "dft" and side == 1024:
        pytest.skip("one case per kernel")
    ph = j2_phases()
    el = [i for i, p in enumerate(ph) if not p["plastic"]][0]
    pm = np.full((side, side), el, np.uint8)
    pat = np.array([[-1, 0, 0], [0, 0, 0], [1, 0, 0]], np.int32)
    s = lib.Solver(pm, ph, pattern=pat, tol=1e-3, max_iter=20, transform=transform)
    out = s.rf_solve(np.array([1e18, 0, 0, 0, 0, 0]))
    s.close()
    lam, mu = ph[el]["lam"], ph[el]["mu"]
    want = np.array([lam + 2 * mu, lam, lam, 0, 0, 0]) * 1e18
    # one FP32 law evaluation per voxel and an FP64 average
    assert np.linalg.norm(out["sigma_bar"] - want) <= 1e-5 * np.linalg.norm(want)
