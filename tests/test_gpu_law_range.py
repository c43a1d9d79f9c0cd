"""The J2 law at the ends of FP32's range and on restored states, in every kernel that evaluates it."""

import numpy as np
import pytest

from synth.configs import j2_phases

pytestmark = pytest.mark.gpu

# grid, transform options: one per row kernel
KERNELS = [((32, 32), dict(transform="fft")), ((32, 32), dict(transform="fft", fft_fuse=3)),
           ((32, 32), dict(transform="fft", fft_fuse=-1)), ((40, 40), dict(transform="dft")),
           ((1024, 1024), dict(transform="fft", fft_fuse=3)),
           ((64, 64, 64), dict(transform="fft")), ((32, 32, 40), dict(transform="dft")),
           ((40, 40), dict(transform="dft", precision="split_bf16")),
           ((40, 40), dict(transform="dft", precision="split_tf32"))]


def indices():
    ph = j2_phases()
    pl = [i for i, p in enumerate(ph) if p["plastic"]][0]
    el = [i for i, p in enumerate(ph) if not p["plastic"]][0]
    return ph, pl, el


def waves(dim):
    return np.array([[-1, 0, 0], [0, 0, 0], [1, 0, 0]], np.int32)


@pytest.mark.parametrize("shape,opts", KERNELS)
def test_overflowing_invariant_of_a_yielding_phase_is_an_error(lib, shape, opts):
    """mu eps = 1e19: the squared invariant overflows, the trial stress itself does not. A J2 phase
    must not hand that trial stress back as if it had not yielded."""
    ph, pl, _ = indices()
    pm = np.full(shape, pl, np.uint8)
    s = lib.Solver(pm, ph, pattern=waves(len(shape)), tol=1e-3, max_iter=20, **opts)
    with pytest.raises(lib.RFError) as e:
        s.rf_solve(np.array([1e18, 0, 0, 0, 0, 0]))
    assert e.value.code == -3
    s.close()


@pytest.mark.parametrize("shape,opts", KERNELS)
def test_tiny_yield_stress_does_not_flow_at_rest(lib, shape, opts):
    """A yield stress below the root of the smallest normal number (1.08e-19): an unstrained cell has
    no stress, so nothing flows."""
    ph, pl, _ = indices()
    ph = ph.copy()
    ph["sigma_y0"][pl] = 1e-22
    s = lib.Solver(np.full(shape, pl, np.uint8), ph, pattern=waves(len(shape)), tol=1e-3, max_iter=5,
                   **opts)
    s.rf_solve_path(np.zeros((1, 6)))
    _, sig, alpha = s.rf_get_fields()
    s.close()
    assert not alpha.any() and not sig.any()


@pytest.mark.parametrize("shape,opts", KERNELS[:7])
def test_flow_at_tiny_stresses(lib, shape, opts):
    """A homogeneous cell in shear, its squared invariant near 1e-40 (subnormal, steps of 1.4e-45,
    1.4e-5 of it at most after four roundings), yield stress half the trial stress: the accumulated
    plastic strain is (seq - sy) / (3 mu + H), off by at most twice half that."""
    ph, pl, _ = indices()
    ph = ph.copy()
    mu, H = float(ph["mu"][pl]), float(ph["hardening"][pl])
    seq = 1.2e-20
    ph["sigma_y0"][pl] = 0.5 * seq
    e12 = seq / (np.sqrt(3.0) * 2.0 * mu)
    s = lib.Solver(np.full(shape, pl, np.uint8), ph, pattern=waves(len(shape)), tol=1e-3, max_iter=5,
                   **opts)
    s.rf_solve_path(np.array([[0, 0, 0, 0, 0, e12]]))
    alpha = s.rf_get_fields()[2]
    s.close()
    want = 0.5 * seq / (3.0 * mu + H)
    assert np.abs(alpha - want).max() <= 1e-4 * want


@pytest.mark.parametrize("shape,opts", KERNELS[:7])
def test_elastic_voxels_of_a_restored_state(lib, shape, opts):
    """A state taken on one phase map and restored on another (rf_set_state asks for the same grid,
    phases and pattern): voxels that are elastic now keep the plastic strain they were given and obey
    Hooke's law on the whole strain. One FP32 law evaluation per voxel: 1e-6 of the largest stress."""
    ph, pl, el = indices()
    pm = np.full(shape, pl, np.uint8)
    pm[..., :shape[-1] // 2] = el
    s = lib.Solver(pm, ph, pattern=waves(len(shape)), tol=1e-4, max_iter=200, **opts)
    macro = np.array([0.015, -0.01, 0, 0, 0, 0.004])
    s.rf_solve_path(macro[None])
    state, alpha = s.rf_get_state(), s.rf_get_fields()[2]
    assert alpha.max() > 1e-3
    other = np.where(pm == el, pl, el).astype(np.uint8)
    s.rf_set_phase_map(other)
    s.rf_set_state(state)
    assert s.rf_get_state() == state
    s.rf_solve(macro)
    eps, sig, after = s.rf_get_fields()
    s.close()
    at = other == el
    lam, mu = ph["lam"][el], ph["mu"][el]
    e = eps[:, at].astype(np.float64)
    want = 2.0 * mu * e
    want[:3] += lam * e[:3].sum(axis=0)
    assert np.abs(sig[:, at] - want).max() <= 1e-6 * np.abs(want).max()
    assert np.array_equal(after[at], alpha[at])
