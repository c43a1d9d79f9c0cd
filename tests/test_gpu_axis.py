"""Transforms along y and z of the pruned DFT: lines that come as partial sums over slices of x (the
split modes on rows of more than 128 voxels), and long sums for few results (blocks of a cluster
share them).

Tolerances as in test_gpu_parity.py: FP32 1e-5 for the strain field and 1e-6 for the homogenised
stress, split modes 3e-5 (two-term operands and FP32 accumulation along x, amplified by the
fixed-point map).
"""

import numpy as np
import pytest

import oracle as O
from oracle.rf_oracle import VOIGT
from synth.configs import elastic_phases, j2_phases

pytestmark = pytest.mark.gpu

EPS_TOL, SBAR_TOL, SPLIT_TOL = 1e-5, 1e-6, 3e-5


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def check(lib, shape, phases, K, eps_tol, sbar_tol, **opts):
    rng = np.random.default_rng(sum(shape))
    pm = (rng.random(shape) < 0.4).astype(np.uint8)
    pat = O.pattern_adapted(pm, 1, K)
    macro = np.array([0.012, -0.004, 0, 0, 0, 0.003])
    s = lib.Solver(pm, phases, pattern=pat, tol=0.0, max_iter=3, transform="dft", **opts)
    out = s.rf_solve(macro)
    eps, _, _ = s.rf_get_fields()
    s.close()
    r = O.solve(pm, phases, macro, pat, tol=0.0, max_iter=3)
    want = np.stack([r.eps[..., i, j] for (i, j) in VOIGT]).reshape(eps.shape)
    assert rel(eps, want) <= eps_tol
    assert rel(out["sigma_bar"], r.sigma_bar) <= sbar_tol


@pytest.mark.parametrize("prec", ["split_bf16", "split_tf32"])
@pytest.mark.parametrize("shape,K", [((50, 300), 900), ((3, 129), 20), ((300, 700), 40),
                                     ((20, 33, 300), 2000), ((5, 9, 1100), 300)])
def test_slices_of_x(lib, prec, shape, K):
    """Two to nine slices, few and many rows of the pattern, 2D and 3D."""
    check(lib, shape, j2_phases(), K, SPLIT_TOL, SPLIT_TOL, precision=prec)


@pytest.mark.parametrize("shape,K", [((2000, 7), 1), ((2000, 7), 30), ((1025, 5), 11), ((255, 40), 3),
                                     ((130, 5), 650), ((131, 3), 393), ((700, 3, 4), 25),
                                     ((3, 520, 2), 9)])
def test_long_sums_for_few_results(lib, shape, K):
    """Two to eight blocks per cluster, shares of unequal length, both directions (the full sets
    make the inverse's sum the long one)."""
    check(lib, shape, elastic_phases(), K, EPS_TOL, SBAR_TOL)
