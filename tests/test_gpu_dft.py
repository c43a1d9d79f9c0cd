"""The pruned-DFT kernels at the sizes where their tiles, splits and pairs can go wrong, against the
oracle. Tolerances as in test_gpu_parity.py (relative L2 1e-5, homogenised stress 1e-6): sums of at
most 1535 terms in FP32 partial sums stay two orders below."""

import numpy as np
import pytest

import oracle as O
from oracle.rf_oracle import VOIGT
from synth.configs import elastic_phases, j2_phases

pytestmark = pytest.mark.gpu

EPS_TOL = 1e-5
SBAR_TOL = 1e-6


def full_pattern(shape):
    from paper_2103_10203_gb300.sweep import full_pattern as full
    return full(shape)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def field(t, shape):
    """oracle [Nz,Ny,Nx,3,3] -> [6, *shape]"""
    return np.stack([t[..., i, j] for (i, j) in VOIGT]).reshape((6,) + tuple(shape))


def check(lib, shape, phases, ratio, macro, full=False, n=3):
    rng = np.random.default_rng(sum(shape))
    pm = (rng.random(shape) < 0.4).astype(np.uint8)
    pm.flat[0], pm.flat[-1] = 0, 1
    pat = full_pattern(shape) if full else O.pattern_adapted(pm, 1, max(1, int(ratio * pm.size)))
    s = lib.Solver(pm, phases, pattern=pat, tol=0.0, max_iter=n, transform="dft")
    out = s.rf_solve(macro)
    eps, sig, _ = s.rf_get_fields()
    co = s.rf_get_reduced_strain()
    s.close()
    r = O.solve(pm, phases, macro, pat, tol=0.0, max_iter=n)
    assert rel(eps, field(r.eps, shape)) <= EPS_TOL
    assert rel(sig, field(r.sigma, shape)) <= EPS_TOL
    assert rel(out["sigma_bar"], r.sigma_bar) <= SBAR_TOL
    want = np.stack([r.eps_hat[:, i, j] for (i, j) in VOIGT], axis=1)
    assert rel(co[..., 0] + 1j * co[..., 1], want) <= EPS_TOL


M2 = np.array([0.012, -0.004, 0, 0, 0, 0.003])
M3 = np.array([0.01, -0.004, 0.002, 0.001, 0.003, -0.002])


@pytest.mark.parametrize("shape", [(2, 1), (1, 2), (3, 3), (5, 2), (31, 33), (32, 32), (61, 97),
                                   (129, 64), (130, 767), (7, 768), (3, 1533), (2, 1534),
                                   (2, 1535), (260, 40), (40, 260)])
@pytest.mark.parametrize("plastic", [False, True])
def test_2d_sizes(lib, shape, plastic):
    check(lib, shape, j2_phases() if plastic else elastic_phases(), 0.1, M2)


@pytest.mark.parametrize("shape", [(7, 6), (33, 40), (40, 33)])
def test_2d_full_set(lib, shape):
    check(lib, shape, elastic_phases(), 1.0, M2, full=True)


@pytest.mark.parametrize("shape", [(1, 2, 3), (3, 1, 2), (9, 7, 5), (20, 31, 18), (33, 16, 25),
                                   (12, 130, 9), (70, 11, 75), (6, 5, 301)])
@pytest.mark.parametrize("plastic", [False, True])
def test_3d_sizes(lib, shape, plastic):
    check(lib, shape, j2_phases() if plastic else elastic_phases(), 0.05, M3)


def test_3d_full_set(lib):
    check(lib, (7, 10, 9), elastic_phases(), 1.0, M3, full=True)


def test_single_frequency(lib):
    check(lib, (30, 50), elastic_phases(), 0.0, M2)
