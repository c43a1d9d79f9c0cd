"""The kernels on team FFTs (several threads per transform, sizes fixed at compile time): the
persistent 2D solve and the 3D updates, at every side they take, against the oracle.

Tolerances as in test_gpu_parity.py: relative L2 error of fields and coefficients 1e-5 (FP32
transforms of at most 1024 points: some ten roundings of 2^-24 per pass, three passes per
direction and a handful of updates stay two orders below), homogenised stress 1e-6.
"""

import numpy as np
import pytest

import oracle as O
from oracle.rf_oracle import VOIGT
from synth import random_discs
from synth.configs import elastic_phases, j2_phases, k_target

pytestmark = pytest.mark.gpu

EPS_TOL = 1e-5
SBAR_TOL = 1e-6


def full_pattern(shape):
    from paper_2103_10203_gb300.sweep import full_pattern as full
    return full(shape)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def field(t):
    g = t[0] if t.shape[0] == 1 else t
    return np.stack([g[..., i, j] for (i, j) in VOIGT])


def blocks(shape, seed):
    """A two-phase cell of random boxes (any shape)."""
    rng = np.random.default_rng(seed)
    pm = np.zeros(shape, np.uint8)
    for _ in range(4):
        lo = [int(rng.integers(0, n)) for n in shape]
        idx = [np.arange(a, a + max(1, n // 3)) % n for a, n in zip(lo, shape)]
        pm[np.ix_(*idx)] = 1
    return pm


def check(lib, pm, phases, pat, macro, n=4, **opts):
    s = lib.Solver(pm, phases, pattern=pat, tol=0.0, max_iter=n, transform="fft", **opts)
    out = s.rf_solve(macro)
    eps, sig, _ = s.rf_get_fields()
    co = s.rf_get_reduced_strain()
    info = s.rf_get_info()
    s.close()
    r = O.solve(pm, phases, macro, pat, tol=0.0, max_iter=n)
    assert out["iters"] == n
    assert rel(eps, field(r.eps)) <= EPS_TOL
    assert rel(sig, field(r.sigma)) <= EPS_TOL
    assert rel(out["sigma_bar"], r.sigma_bar) <= SBAR_TOL
    want = np.stack([r.eps_hat[:, i, j] for (i, j) in VOIGT], axis=1)
    assert rel(co[..., 0] + 1j * co[..., 1], want) <= EPS_TOL
    return info


@pytest.mark.parametrize("shape", [(32, 32), (48, 48), (64, 64), (96, 96), (128, 128), (192, 192),
                                   (256, 256), (384, 384), (512, 512), (32, 512), (96, 48),
                                   (384, 64), (128, 192), (768, 768), (1024, 1024),
                                   (64, 1024), (1024, 32), (768, 48), (96, 768)])
@pytest.mark.parametrize("plastic", [False, True])
def test_persistent_solve_sides(lib, shape, plastic):
    """Every side of the plans, square and mixed; a pattern of a few per cent."""
    pm = blocks(shape, sum(shape))
    pat = O.pattern_adapted(pm, 1, k_target(0.06, pm.size))
    macro = np.array([0.012, -0.004, 0, 0, 0, 0.003])
    info = check(lib, pm, j2_phases() if plastic else elastic_phases(), pat, macro, fft_fuse=3)
    assert info["fft_fused"] == 3


@pytest.mark.parametrize("shape", [(32, 32), (48, 96), (64, 64), (192, 128)])
def test_persistent_solve_full_set(lib, shape):
    """Every frequency: self-conjugate kx, null frequencies, more kx than blocks of a cluster."""
    pm = blocks(shape, 7)
    check(lib, pm, elastic_phases(), full_pattern(shape), np.array([0.01, 0, 0, 0, 0, 0.002]),
          fft_fuse=3)


def test_persistent_solve_zero_frequency_alone(lib):
    pm = blocks((64, 48), 3)
    check(lib, pm, elastic_phases(), np.zeros((1, 3), np.int32),
          np.array([0.01, 0.002, 0, 0, 0, 0.0]), fft_fuse=3)


def test_persistent_solve_continues_after_divergence(lib):
    """A solve that diverges commits nothing and leaves the context usable."""
    pm = random_discs(64, (6.0, 10.0), 0.05, 5)
    phases = elastic_phases().copy()
    phases["lam"][1] *= 1000.0
    phases["mu"][1] *= 1000.0
    pat = full_pattern(pm.shape)
    s = lib.Solver(pm, phases, pattern=pat, tol=1e-6, max_iter=500, transform="fft", fft_fuse=3,
                   ref="volume")
    with pytest.raises(lib.RFError) as e:
        s.rf_solve(np.array([0.01, 0, 0, 0, 0, 0]))
    assert e.value.code == -4
    with pytest.raises(lib.RFError):
        s.rf_get_fields()
    s.close()


def check3(lib, pm, phases, pat, macro, n=3, **opts):
    """The 3D updates (stage "column_phase" is theirs alone in 3D), traced and untraced."""
    check(lib, pm, phases, pat, macro, n, **opts)
    s = lib.Solver(pm, phases, pattern=pat, tol=0.0, max_iter=n, transform="fft", **opts)
    s.rf_set_tracing(True)
    s.rf_solve(macro)
    ran = s.rf_get_stage_times()["column_phase"][1]
    s.close()
    return ran == n


SIDES3 = [(32, 48, 64), (48, 96, 32), (96, 64, 48), (64, 32, 96), (32, 32, 128), (32, 128, 32),
          (128, 32, 32), (192, 32, 32), (32, 192, 32), (32, 32, 192), (256, 32, 32), (32, 256, 32),
          (32, 32, 256), (384, 32, 32), (32, 384, 32), (32, 32, 384), (512, 32, 32), (32, 512, 32),
          (32, 32, 512)]


@pytest.mark.parametrize("shape", SIDES3)
def test_3d_updates_sides(lib, shape):
    """Every side along every axis; ragged groups of kx and rows included."""
    pm = blocks(shape, sum(shape))
    pat = O.pattern_adapted(pm, 1, k_target(0.03, pm.size))
    check3(lib, pm, elastic_phases(), pat, np.array([0.01, -0.004, 0.002, 0.001, 0.003, -0.002]))


@pytest.mark.parametrize("shape", [(32, 48, 64), (64, 64, 64), (96, 32, 32)])
def test_3d_updates_plastic(lib, shape):
    pm = blocks(shape, 11)
    pat = O.pattern_adapted(pm, 1, k_target(0.03, pm.size))
    check3(lib, pm, j2_phases(), pat, np.array([0.015, -0.004, 0.002, 0.001, 0.003, -0.002]))


def test_3d_updates_full_set(lib):
    pm = blocks((32, 48, 32), 2)
    check3(lib, pm, elastic_phases(), full_pattern(pm.shape), np.array([0.01, 0, 0, 0, 0.002, 0]))


def test_3d_updates_are_the_ones_that_run(lib):
    """At a size where their advantage is large the tuner takes them; pinned modes do not."""
    pm = random_discs(64, (6.0, 10.0), 0.3, 5)[None].repeat(64, 0)
    pat = O.pattern_adapted(pm, 1, k_target(0.02, pm.size))
    macro = np.array([0.01, 0, 0, 0.002, 0, 0])
    assert check3(lib, pm, elastic_phases(), pat, macro)
    assert not check3(lib, pm, elastic_phases(), pat, macro, fft_fuse=-1)


@pytest.mark.parametrize("side", [512, 768, 1024])
def test_persistent_solve_plastic_path(lib, side):
    """Two increments: the second reads committed internal variables (held in shared memory, or
    fetched from global memory on the long sides)."""
    pm = blocks((side, side), side)
    pat = O.pattern_adapted(pm, 1, k_target(0.02, pm.size))
    path = np.zeros((2, 6))
    path[:, 0] = [0.008, 0.014]
    path[:, 1] = [-0.002, -0.004]
    s = lib.Solver(pm, j2_phases(), pattern=pat, tol=1e-2, max_iter=500, transform="fft", fft_fuse=3)
    out = s.rf_solve_path(path)
    eps, _, _ = s.rf_get_fields()
    assert s.rf_get_info()["fft_fused"] == 3
    s.close()
    sbar, _, r = O.solve_path(pm, j2_phases(), path, pat, fixed_iters=out["iters"])
    for n in range(len(path)):
        assert rel(out["sigma_bar"][n], sbar[n]) <= SBAR_TOL
    assert rel(eps, field(r.eps)) <= EPS_TOL
