"""The cell-resident batched solve (a block runs an RVE of any sides in its shared memory) and the
network's products with K split over a cluster, at the sizes where they can go wrong.

Tolerances: as in test_gpu_batch.py for solves (coefficients 1e-5, homogenised stress 1e-6) and
test_gpu_mlp.py for the network (TF32 4e-3, BF16 3e-2).
"""

import numpy as np
import pytest

import oracle as O
from oracle import mlp as M
from synth.configs import elastic_phases

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def cells(shapes, seed, ratio=0.08):
    rng = np.random.default_rng(seed)
    pms, pats, macros = [], [], []
    for sh in shapes:
        pm = (rng.random(sh) < 0.4).astype(np.uint8)
        pm.flat[0], pm.flat[-1] = 0, 1
        pms.append(pm)
        pats.append(O.pattern_adapted(pm, 1, max(2, int(ratio * pm.size))))
        macros.append([*rng.uniform(-0.01, 0.01, 2), 0, 0, 0, rng.uniform(-0.01, 0.01)])
    return pms, pats, np.array(macros)


def check(lib, shapes, n=4, **opts):
    ph = elastic_phases()
    pms, pats, macros = cells(shapes, len(shapes))
    b = lib.BatchSolver(pms, ph, pats, tol=0.0, max_iter=n, transform="dft", **opts)
    out = b.rf_batch_solve(macros)
    again = b.rf_batch_solve(macros)
    coeffs = b.rf_batch_reduced_strain().cpu().numpy()
    _, off = b.rf_batch_slots()
    b.close()
    assert np.all(out["iters"] == n)
    assert np.array_equal(out["sigma_bar"], again["sigma_bar"])
    for i, (pm, pat) in enumerate(zip(pms, pats)):
        r = O.solve(pm, ph, macros[i], pat, tol=0.0, max_iter=n)
        at = {(int(k[0]), int(k[1])): p for p, k in enumerate(pat)}
        hs = sorted((int(k[0]), int(k[1])) for k in pat if k[0] >= 0)
        want = np.array([[r.eps_hat[at[k], 0, 0], r.eps_hat[at[k], 1, 1], r.eps_hat[at[k], 0, 1]]
                         for k in hs])
        got = coeffs[off[i]:off[i + 1], :, 0] + 1j * coeffs[off[i]:off[i + 1], :, 1]
        assert rel(got, want) <= 1e-5, (pm.shape, rel(got, want))
        assert rel(out["sigma_bar"][i], r.sigma_bar) <= 1e-6, pm.shape


@pytest.mark.parametrize("shapes", [[(2, 2)], [(3, 2), (2, 3), (5, 7)], [(64, 64), (33, 120)],
                                    [(121, 50), (50, 121), (97, 97)], [(9, 300), (300, 9)]])
@pytest.mark.parametrize("many", [1, 40])
def test_cells_match_oracle(lib, shapes, many):
    """Few and many RVEs (the queue wraps and a block takes RVEs of different layouts in turn)."""
    check(lib, shapes * many, n=3)


def test_cells_beyond_shared_memory(lib):
    """An RVE that does not fit sends the whole batch to the sweeps."""
    check(lib, [(260, 256), (40, 41)], n=3)


def test_cells_reach_the_sweeps_answer(lib):
    pms, pats, macros = cells([(70, 61), (50, 55), (90, 43)] * 12, 5, 0.05)
    ph = elastic_phases()
    res = []
    for opt in (-1, 0):
        b = lib.BatchSolver(pms, ph, pats, tol=1e-6, max_iter=500, transform="dft",
                            batch_resident=opt)
        res.append(b.rf_batch_solve(macros))
        b.close()
    assert res[0]["converged"] and res[1]["converged"]
    assert np.max(np.abs(res[0]["iters"] - res[1]["iters"])) <= 1
    assert rel(res[1]["sigma_bar"], res[0]["sigma_bar"]) <= 2e-6


@pytest.mark.parametrize("B", [1, 5, 64, 127, 128, 129, 260])
@pytest.mark.parametrize("H", [16, 48, 512])
def test_network_products_of_few_rows(lib, B, H):
    """Row tiles of one row to three, K from one chunk (no split) to eight shares."""
    import torch
    net = lib.WarmStartNet(H, 300)
    rng = np.random.default_rng(B + H)
    parts = [rng.standard_normal(sh) / np.sqrt(sh[0] if len(sh) == 2 else 4.0)
             for sh in net.shapes()]
    flat = np.concatenate([p.ravel() for p in parts]).astype(np.float32)
    net.rf_mlp_set_params(flat)
    assert np.array_equal(net.rf_mlp_get_params(), flat)
    params = [p.astype(np.float64) for p in net.split(flat)]
    X = rng.standard_normal((B, M.N_DESC)).astype(np.float32)
    want, _ = M.forward(params, X.astype(np.float64))
    with torch.cuda.stream(net.stream):
        dx = torch.as_tensor(X, device="cuda")
        for prec, tol in (("tf32", 4e-3), ("bf16", 3e-2)):
            got = net.rf_mlp_forward(dx, prec).cpu().numpy()
            assert rel(got, want) <= tol, (prec, rel(got, want))
    net.close()
