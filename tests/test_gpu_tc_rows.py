"""The tensor-core row kernel that holds its twiddles (BF16 parts, at most 64 kx), at the sizes where
its tiles, slices and rounds can go wrong, against the oracle. Tolerance as the split modes' in
test_gpu_parity.py: 3e-5 relative L2 (two-term operands exact to 2^-18, sums of at most 128
products in FP32)."""

import numpy as np
import pytest

import oracle as O
from oracle.rf_oracle import VOIGT
from synth.configs import elastic_phases, j2_phases

pytestmark = pytest.mark.gpu

TOL = 3e-5
M2 = np.array([0.012, -0.004, 0, 0, 0, 0.003])
M3 = np.array([0.01, -0.004, 0.002, 0.001, 0.003, -0.002])


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def field(t, shape):
    return np.stack([t[..., i, j] for (i, j) in VOIGT]).reshape((6,) + tuple(shape))


def check(lib, shape, phases, ratio, full=False, n=3):
    from paper_2103_10203_gb300.sweep import full_pattern
    rng = np.random.default_rng(sum(shape))
    pm = (rng.random(shape) < 0.4).astype(np.uint8)
    pm.flat[0], pm.flat[-1] = 0, 1
    pat = full_pattern(shape) if full else O.pattern_adapted(pm, 1, max(1, int(ratio * pm.size)))
    macro = M2 if len(shape) == 2 else M3
    s = lib.Solver(pm, phases, pattern=pat, tol=0.0, max_iter=n, transform="dft",
                   precision="split_bf16")
    out = s.rf_solve(macro)
    eps, sig, _ = s.rf_get_fields()
    s.close()
    r = O.solve(pm, phases, macro, pat, tol=0.0, max_iter=n)
    assert rel(eps, field(r.eps, shape)) <= TOL
    assert rel(sig, field(r.sigma, shape)) <= TOL
    assert rel(out["sigma_bar"], r.sigma_bar) <= TOL


# one row to several rounds of row tiles (a device takes 608 groups), slices of x of 128 and less
@pytest.mark.parametrize("shape", [(2, 2), (1, 5), (33, 31), (16, 128), (17, 129), (40, 300),
                                   (700, 20), (4096, 6), (3, 2, 4), (5, 7, 130), (71, 70, 12)])
@pytest.mark.parametrize("plastic", [False, True])
def test_shapes(lib, shape, plastic):
    check(lib, shape, j2_phases() if plastic else elastic_phases(), 0.05)


# 64 kx are the most that it takes; one more goes to the kernel that stages its twiddles
@pytest.mark.parametrize("shape", [(9, 127), (9, 128), (3, 4, 127), (3, 4, 128)])
def test_widest_pattern(lib, shape):
    check(lib, shape, elastic_phases(), 1.0, full=True)
