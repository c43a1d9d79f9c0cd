"""Reading results: what a read needs, and that it leaves the next solve as it was."""

import numpy as np
import pytest

import oracle as O
from synth.configs import elastic_phases

pytestmark = pytest.mark.gpu


def full_pattern(shape):
    from paper_2103_10203_gb300.sweep import full_pattern as full
    return full(shape)


def cell(shape, seed=3):
    pm = (np.random.default_rng(seed).random(shape) < 0.4).astype(np.uint8)
    pm.flat[0], pm.flat[-1] = 0, 1
    return pm


def test_reduced_strain_needs_no_device_memory(lib):
    """The coefficients of the full set of 512 x 512 are 12.6 MB."""
    import torch
    pm = cell((512, 512))
    s = lib.Solver(pm, elastic_phases(), pattern=full_pattern(pm.shape), tol=0.0, max_iter=2,
                   transform="fft")
    s.rf_solve(np.array([0.01, 0, 0, 0, 0, 0.002]))
    s.rf_get_fields()
    before = torch.cuda.mem_get_info()[0]
    s.rf_get_reduced_strain()
    assert before - torch.cuda.mem_get_info()[0] < 4 << 20
    s.close()


@pytest.mark.parametrize("shape,full,opts", [
    ((1, 1), True, dict(transform="dft")), ((9, 7), True, dict(transform="dft")),
    ((9, 7), False, dict(transform="dft")), ((64, 48), True, dict(transform="fft")),
    ((64, 48), False, dict(transform="fft", fft_fuse=-1)),
    ((64, 48), False, dict(transform="fft", fft_fuse=1)),
    ((64, 48), False, dict(transform="fft", fft_fuse=2)),
    ((64, 48), False, dict(transform="fft", fft_fuse=3)),
    ((24, 16), True, dict(transform="fft", fft_fuse=3)),
    ((1024, 1024), False, dict(transform="fft", fft_fuse=4)),
    ((1024, 1024), False, dict(transform="fft", fft_fuse=5)),
    ((32, 32, 32), False, dict(transform="fft")), ((32, 32, 32), True, dict(transform="fft")),
    ((32, 32, 20), False, dict(transform="dft")), ((5, 6, 7), True, dict(transform="dft")),
    ((20, 200), False, dict(transform="dft", precision="split_bf16"))])
def test_reading_coefficients_between_solves(lib, shape, full, opts):
    """The coefficients (FP32 values of sums that the oracle has in FP64) and, bit for bit, a second
    solve after they were read; patterns of one entry to the whole grid."""
    pm = cell(shape)
    pat = full_pattern(shape) if full else O.pattern_adapted(pm, 1, max(1, pm.size // 50))
    macro = np.array([0.01, -0.004, 0, 0, 0, 0.002])
    s = lib.Solver(pm, elastic_phases(), pattern=pat, tol=0.0, max_iter=2, **opts)
    first = s.rf_solve(macro)["sigma_bar"]
    co = s.rf_get_reduced_strain()
    second = s.rf_solve(macro)["sigma_bar"]
    assert np.array_equal(first, second)
    assert np.array_equal(co, s.rf_get_reduced_strain())
    s.close()
    r = O.solve(pm, elastic_phases(), macro, pat, tol=0.0, max_iter=2)
    want = np.stack([r.eps_hat[:, i, j] for (i, j) in O.rf_oracle.VOIGT], axis=1)
    tol = 3e-5 if "precision" in opts else 1e-5   # as in test_gpu_parity.py
    assert np.linalg.norm(co[..., 0] + 1j * co[..., 1] - want) <= tol * np.linalg.norm(want)


def test_network_reads_need_no_device_memory_and_share_nothing(lib):
    """Parameters and gradients of 1024 hidden units (5.4 MB), read by two threads at once."""
    import threading

    import torch
    net = lib.WarmStartNet(1024, 8)
    flat = np.random.default_rng(1).standard_normal(net.dims["n_params"]).astype(np.float32)
    net.rf_mlp_set_params(flat)
    before = torch.cuda.mem_get_info()[0]
    assert np.array_equal(net.rf_mlp_get_params(), flat)
    assert before - torch.cuda.mem_get_info()[0] < 2 << 20
    bad = []

    def read(f, want):
        for _ in range(20):
            if not np.array_equal(f(), want):
                bad.append(f.__name__)

    ts = [threading.Thread(target=read, args=(net.rf_mlp_get_params, flat)),
          threading.Thread(target=read, args=(net.rf_mlp_get_grads, np.zeros_like(flat)))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    net.close()
    assert not bad


@pytest.mark.parametrize("H", [16, 48, 512])
def test_network_parameters_round_trip(lib, H):
    net = lib.WarmStartNet(H, 8)
    flat = np.arange(net.dims["n_params"], dtype=np.float32)
    net.rf_mlp_set_params(flat)
    assert np.array_equal(net.rf_mlp_get_params(), flat)
    net.close()
