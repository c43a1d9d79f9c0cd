"""options.batch_resident = 1 runs the cell-resident solve wherever a batch qualifies, -1 never. A
cell-resident solve is two kernels (start and solve), sweeps are several per update.

Tolerances as in test_gpu_batch.py: coefficients 1e-5, homogenised stress 1e-6.
"""

import numpy as np
import pytest

import oracle as O
from synth.configs import elastic_phases

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - b) / max(np.linalg.norm(b), 1e-300))


def disc(shape, share=0.08):
    """The shortest wave vectors, about that share of them (at least the first three): few distinct kx
    and ky, so that what an update needs stays small."""
    ny, nx = shape
    k = [(x, y) for y in range(-((ny - 1) // 2), ny // 2 + 1)
         for x in range(-((nx - 1) // 2), nx // 2 + 1)]
    k.sort(key=lambda v: v[0] ** 2 + v[1] ** 2)
    rho = sum(v * v for v in k[min(len(k) - 1, max(2, int(share * len(k))))])
    held = {v for v in k if v[0] ** 2 + v[1] ** 2 <= rho}

    def conj(i, n):
        i = -i % n
        return i if i <= n // 2 else i - n

    held |= {(conj(x, nx), conj(y, ny)) for x, y in held}
    return np.array([(x, y, 0) for x, y in sorted(held)], np.int32)


def solve(lib, shapes, resident, n=3, **opts):
    rng = np.random.default_rng(len(shapes))
    cells = {}
    for sh in shapes:
        if sh not in cells:
            pm = (rng.random(sh) < 0.4).astype(np.uint8)
            pm.flat[0], pm.flat[-1] = 0, 1
            cells[sh] = (pm, disc(sh))
    macros = np.zeros((len(shapes), 6))
    macros[:, [0, 1, 5]] = rng.uniform(-0.01, 0.01, (len(shapes), 3))
    b = lib.BatchSolver([cells[s][0] for s in shapes], elastic_phases(), [cells[s][1] for s in shapes],
                        tol=0.0, max_iter=n, batch_resident=resident, **opts)
    before = b.rf_batch_info()["kernel_launches"]
    out = b.rf_batch_solve(macros)
    launches = b.rf_batch_info()["kernel_launches"] - before
    coeffs = b.rf_batch_reduced_strain().cpu().numpy()
    _, off = b.rf_batch_slots()
    b.close()
    for i in range(0, len(shapes), max(1, len(shapes) // 12)):
        pm, pat = cells[shapes[i]]
        r = O.solve(pm, elastic_phases(), macros[i], pat, tol=0.0, max_iter=n)
        at = {(int(k[0]), int(k[1])): p for p, k in enumerate(pat)}
        hs = sorted((int(k[0]), int(k[1])) for k in pat if k[0] >= 0)
        want = np.array([[r.eps_hat[at[k], 0, 0], r.eps_hat[at[k], 1, 1], r.eps_hat[at[k], 0, 1]]
                         for k in hs])
        got = coeffs[off[i]:off[i + 1], :, 0] + 1j * coeffs[off[i]:off[i + 1], :, 1]
        assert rel(got, want) <= 1e-5, (pm.shape, rel(got, want))
        assert rel(out["sigma_bar"][i], r.sigma_bar) <= 1e-6, pm.shape
    return launches


# one RVE, layouts of very different shapes, more RVEs than SMs (where sweeps can be faster)
QUALIFY = [[(2, 2)], [(3, 2), (2, 3), (5, 7)], [(64, 64), (33, 120)],
           [(121, 50), (50, 121), (97, 97)], [(9, 300), (300, 9)], [(9, 12), (20, 17), (5, 7)] * 234,
           [(61, 75), (40, 41)] * 100]


@pytest.mark.parametrize("shapes", QUALIFY)
def test_cells_asked_for(lib, shapes):
    assert solve(lib, shapes, 1, transform="dft") == 2


@pytest.mark.parametrize("shapes", QUALIFY[1:4])
def test_cells_refused(lib, shapes):
    assert solve(lib, shapes, -1, transform="dft") > 6


def test_odd_cells_of_a_batch_with_ffts(lib):
    assert solve(lib, [(61, 75), (25, 85)], 1, transform="fft") == 2
    assert solve(lib, [(61, 75), (25, 64)], 1, transform="fft") > 6


def test_cells_that_do_not_fit(lib):
    assert solve(lib, [(260, 256), (40, 41)], 1, transform="dft") > 6
