"""Performance cases of the reduced-frequency solver: the work its users have it do, each through
the package's public entry points.

Kinds of work
  solve    one microstructure and one macroscopic strain (rf.Solver, rf_solve): the homogenised
           stress and the reduced strain coefficients.
  path     an elastoplastic load path in increments (rf_reset_path, rf_solve_path): the stress
           history, the reduced strain coefficients of the last increment and the voxel fields
           (strain, stress, accumulated plastic strain).
  study    reduced solve, compatibility step and the voxel fields, as in the accuracy studies of
           Sec. 5 of the paper.
  batch    many RVEs at once, as the Gauss points of an FE-FFT model (rf.BatchSolver,
           rf_batch_solve): a few microstructures, every point with a macroscopic strain of its
           own; the coefficients in a buffer that has room for every set of microstructures.
  pattern  the geometrically adapted set of frequencies of a microstructure (rf_pattern_adapted).
  train    loss and gradients of the warm-start network over one minibatch of RVEs
           (rf.WarmStartNet, rf_mlp_loss_grad, rf_mlp_get_grads).

Every solve runs to the convergence measure 1e-6. Homogenised stresses and the loss are averages
of single-precision fields that the binding hands over in 64-bit containers; they are returned in
the precision that they are computed in. The number of updates and the final measure are
diagnostics of where the iteration stopped, and no result.

Microstructures, macroscopic strains, patterns and network inputs are made here from the seed, with
torch and numpy only, so that the 64-bit results of exact() need nothing of the package.
"""

from __future__ import annotations

import math

import numpy as np
import torch

TOL = 1e-6
MAX_ITER = 2000
VOIGT = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))
FFT_SIDES = (32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024)
BATCH_SIDES = (64, 96, 128, 192, 256)
N_IN, N_BASIS, N_OUT = 48, 27, 243

# (lambda, mu, sigma_y0, H, plastic) of matrix and inclusion, GPa
_GLASS = ((70 * 0.3 / (1.3 * 0.4), 70 / 2.6), (400 * 0.2 / (1.2 * 0.6), 400 / 2.4))
LAWS = {
    # E 70 / nu 0.3 matrix with E 400 / nu 0.2 fibres, elastic and with a J2 matrix
    "fibre": ((*_GLASS[0], 0.0, 0.0, 0), (*_GLASS[1], 0.0, 0.0, 0)),
    "fibre_j2": ((*_GLASS[0], 0.25, 1.0, 1), (*_GLASS[1], 0.0, 0.0, 0)),
    # moduli of the paper's examples (Sec. 5), elastic and with its J2 matrix
    "paper": ((1.0, 1.0, 0.0, 0.0, 0), (2.0, 2.0, 0.0, 0.0, 0)),
    "paper_j2": ((1.0, 1.0, 0.01, 0.01, 1), (2.0, 2.0, 0.0, 0.0, 0)),
}


def listed():
    return [
        # the smallest call: one 64^2 fibre cell, as at one Gauss point solved by itself
        dict(name="point_64", kind="solve", nx=64, ny=64, nz=1, law="fibre", ratio=0.05, vf=0.3,
             r_lo=8.0, r_hi=24.0, transform="fft", precision="fp32"),
        # the paper's 256^2 several-inclusion cell: reduced solve, compatibility step, fields
        dict(name="study_256", kind="study", nx=256, ny=256, nz=1, law="paper", ratio=0.0154,
             vf=0.3, r_lo=16.0, r_hi=32.0, transform="fft", precision="fp32"),
        # the paper's elastoplastic example: load path of a 256^2 cell with its fields at the end
        dict(name="path_256", kind="path", nx=256, ny=256, nz=1, law="paper_j2", ratio=0.0154,
             vf=0.3, r_lo=16.0, r_hi=32.0, steps=25),
        # the large elastoplastic composite: 20 uniaxial increments on 1024^2
        dict(name="path_1024", kind="path", nx=1024, ny=1024, nz=1, law="fibre_j2", ratio=0.05,
             vf=0.4, r_lo=8.0, r_hi=24.0, steps=20),
        # 3D particle composite, 128^3, with FFTs
        dict(name="spheres_128", kind="solve", nx=128, ny=128, nz=128, law="fibre", ratio=0.02,
             vf=0.25, r_lo=6.0, r_hi=12.0, transform="fft", precision="fp32"),
        # the same composite with split-precision transforms on the tensor cores
        dict(name="spheres_128_split", kind="solve", nx=128, ny=128, nz=128, law="fibre",
             ratio=0.02, vf=0.25, r_lo=6.0, r_hi=12.0, transform="dft", precision="split_bf16"),
        # a micrograph cropped to no particular size (the default transform takes any side)
        dict(name="image_2d", kind="solve", nx=375, ny=250, nz=1, law="fibre", ratio=0.05, vf=0.35,
             r_lo=8.0, r_hi=24.0, transform="dft", precision="fp32"),
        # a cropped tomography volume
        dict(name="image_3d", kind="solve", nx=75, ny=90, nz=66, law="fibre", ratio=0.02, vf=0.25,
             r_lo=6.0, r_hi=12.0, transform="dft", precision="fp32"),
        # FE-FFT: 1024 Gauss points over 40 fibre microstructures of uneven size
        dict(name="gauss_fft", kind="batch", points=1024, micros=40, lo=64, hi=256, odd=False,
             law="fibre", ratio=0.05, transform="fft"),
        # FE-FFT on cells of arbitrary sides
        dict(name="gauss_odd", kind="batch", points=128, micros=16, lo=50, hi=120, odd=True,
             law="fibre", ratio=0.05, transform="dft"),
        # the reduced set of the large composite
        dict(name="pattern_1024", kind="pattern", nx=1024, ny=1024, nz=1, ratio=0.05, vf=0.4,
             r_lo=8.0, r_hi=24.0),
        # one gradient of the warm-start network over 64 cells of 128^2
        dict(name="train_64", kind="train", cells=64, side=128, ratio=0.05, hidden=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("solve2", "solve3", "split", "odd2", "odd3", "path", "study", "batch",
                       "batch_odd", "pattern", "train"))
    ratio = round(math.exp(rng.uniform(math.log(0.0154), math.log(0.1))), 4)
    if kind == "solve2":
        return dict(kind="solve", nx=rng.choice(FFT_SIDES), ny=rng.choice(FFT_SIDES), nz=1,
                    law=rng.choice(("fibre", "paper")), ratio=ratio, vf=round(rng.uniform(0.2, 0.4), 3),
                    r_lo=4.0, r_hi=round(rng.uniform(6.0, 10.0), 2), transform="fft",
                    precision="fp32")
    if kind in ("solve3", "split"):
        sides = (32, 48, 64, 96, 128)
        fft = kind == "solve3"
        return dict(kind="solve", nx=rng.choice(sides), ny=rng.choice(sides), nz=rng.choice(sides),
                    law=rng.choice(("fibre", "paper")), ratio=round(rng.uniform(0.0154, 0.03), 4),
                    vf=round(rng.uniform(0.15, 0.25), 3), r_lo=4.0, r_hi=round(rng.uniform(6.0, 9.0), 2),
                    transform="fft" if fft else "dft",
                    precision="fp32" if fft else rng.choice(("split_bf16", "split_tf32")))
    if kind == "odd2":
        return dict(kind="solve", nx=_log(rng, 40, 500), ny=_log(rng, 40, 400), nz=1,
                    law=rng.choice(("fibre", "paper")), ratio=ratio, vf=round(rng.uniform(0.2, 0.4), 3),
                    r_lo=4.0, r_hi=round(rng.uniform(6.0, 10.0), 2), transform="dft",
                    precision="fp32")
    if kind == "odd3":
        return dict(kind="solve", nx=_log(rng, 24, 96), ny=_log(rng, 24, 96), nz=_log(rng, 24, 96),
                    law=rng.choice(("fibre", "paper")), ratio=round(rng.uniform(0.0154, 0.03), 4),
                    vf=round(rng.uniform(0.15, 0.25), 3), r_lo=4.0, r_hi=round(rng.uniform(6.0, 9.0), 2),
                    transform="dft", precision="fp32")
    if kind == "path":
        law = rng.choice(("fibre_j2", "paper_j2"))
        # the paper's nearly ideal plasticity takes twice the updates: smaller cells, fewer steps
        side = rng.choice(FFT_SIDES[2:] if law == "fibre_j2" else FFT_SIDES[2:8])
        return dict(kind="path", nx=side, ny=side, nz=1, law=law,
                    ratio=round(rng.uniform(0.0154, 0.05), 4), vf=round(rng.uniform(0.2, 0.4), 3),
                    r_lo=6.0, r_hi=round(rng.uniform(8.0, 16.0), 2), steps=rng.randint(5, 20 if law == "fibre_j2" else 12))
    if kind == "study":
        return dict(kind="study", nx=rng.choice(FFT_SIDES[2:9]), ny=rng.choice(FFT_SIDES[2:9]),
                    nz=1, law="paper", ratio=ratio, vf=round(rng.uniform(0.2, 0.4), 3), r_lo=6.0,
                    r_hi=round(rng.uniform(8.0, 16.0), 2), transform="fft", precision="fp32")
    if kind == "batch":
        points = _log(rng, 32, 1024)
        return dict(kind="batch", points=points, micros=min(points, rng.randint(8, 40)), lo=64,
                    hi=256, odd=False, law="fibre", ratio=0.05, transform="fft")
    if kind == "batch_odd":
        points = _log(rng, 16, 128)
        return dict(kind="batch", points=points, micros=min(points, rng.randint(4, 16)),
                    lo=rng.randint(40, 60), hi=rng.randint(80, 120), odd=True, law="fibre",
                    ratio=0.05, transform="dft")
    if kind == "pattern":
        three = rng.random() < 0.4
        if three:
            return dict(kind="pattern", nx=_log(rng, 24, 96), ny=_log(rng, 24, 96),
                        nz=_log(rng, 24, 96), ratio=ratio, vf=0.25, r_lo=4.0,
                        r_hi=round(rng.uniform(6.0, 9.0), 2))
        return dict(kind="pattern", nx=rng.choice(FFT_SIDES), ny=rng.choice(FFT_SIDES), nz=1,
                    ratio=ratio, vf=0.35, r_lo=4.0, r_hi=round(rng.uniform(6.0, 10.0), 2))
    return dict(kind="train", cells=rng.choice((16, 32, 64, 96, 128)), side=rng.choice((64, 96, 128)),
                ratio=0.05, hidden=512)


# --------------------------------------------------------------------------- inputs
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _k_target(ratio, n):
    return int(math.ceil(ratio * n - 1e-9))


def _shape(case):
    s = (case["ny"], case["nx"])
    return s if case["nz"] == 1 else (case["nz"],) + s


def _micro(rng, shape, r_lo, r_hi, vf):
    """Non-overlapping periodic discs or spheres of random radii, uint8, at least one voxel of
    each phase."""
    n = np.array(shape, float)
    d = len(shape)
    top = 0.35 * n.min()
    r_hi = min(r_hi, top)
    r_lo = min(r_lo, r_hi)
    pm = np.zeros(shape, np.uint8)
    cs, rs, filled = np.zeros((0, d)), np.zeros(0), 0.0
    target = vf * n.prod()
    for _ in range(6000):
        if filled >= target:
            break
        c, r = rng.uniform(0.0, n), rng.uniform(r_lo, r_hi)
        if len(rs):
            q = np.abs(cs - c)
            q = np.minimum(q, n - q)
            if np.any((q * q).sum(1) < (rs + r + 1.0) ** 2):
                continue
        cs, rs = np.vstack([cs, c]), np.append(rs, r)
        ax = [np.arange(int(np.floor(c[i] - r)), int(np.ceil(c[i] + r)) + 1) for i in range(d)]
        g = np.meshgrid(*ax, indexing="ij")
        inside = sum((g[i] - c[i]) ** 2 for i in range(d)) <= r * r
        pm[tuple(g[i][inside] % shape[i] for i in range(d))] = 1
        filled += (np.pi * r * r) if d == 2 else (4.0 / 3.0 * np.pi * r ** 3)
    return pm


def _phases(name):
    return [dict(lam=p[0], mu=p[1], sigma_y0=p[2], hardening=p[3], plastic=p[4])
            for p in LAWS[name]]


def _signed(n, dev):
    i = torch.arange(n, device=dev)
    return torch.where(i <= n // 2, i, i - n)


def _adapted(pm, k_target):
    """Geometrically adapted pattern (Sec. 4.2), int32 [K, 3] (kx, ky, kz) sorted by signed linear
    index: pairs (k, -k) by larger quantised amplitude of the inclusion's indicator, smaller
    |k|^2, smaller signed linear index, added whole until k_target frequencies are held."""
    dev = _dev()
    g = torch.as_tensor(pm, device=dev).double()
    g = g if g.dim() == 3 else g[None]
    nz, ny, nx = g.shape
    amp = torch.fft.fftn(g).abs()
    amp = torch.round(amp / amp[0, 0, 0] * 2.0 ** 30).long()
    # the pair (k, -k) has one amplitude
    neg = torch.roll(torch.flip(amp, (0, 1, 2)), (1, 1, 1), (0, 1, 2))
    amp = torch.maximum(amp, neg).flatten()
    kz, ky, kx = torch.meshgrid(_signed(nz, dev), _signed(ny, dev), _signed(nx, dev), indexing="ij")
    k2 = (kz * kz + ky * ky + kx * kx).flatten()

    def lin(z, y, x):
        return ((z + (nz - 1) // 2) * ny + y + (ny - 1) // 2) * nx + x + (nx - 1) // 2

    def neg_of(k, n):
        return torch.where(2 * k == n, k, -k)

    idx = lin(kz, ky, kx).flatten()
    cidx = lin(neg_of(kz, nz), neg_of(ky, ny), neg_of(kx, nx)).flatten()
    rep = torch.nonzero(idx <= cidx)[:, 0]
    o = rep[torch.argsort(idx[rep], stable=True)]
    o = o[torch.argsort(k2[o], stable=True)]
    o = o[torch.argsort(-amp[o], stable=True)]
    size = 2 - (idx[o] == cidx[o]).long()
    held = torch.cumsum(size, 0)
    m = int(torch.searchsorted(held, torch.tensor(k_target, device=dev))) + 1
    keep = o[:m]
    every = torch.unique(torch.cat([idx[keep], cidx[keep]]))
    every = every.cpu().numpy()
    x = every % nx - (nx - 1) // 2
    y = every // nx % ny - (ny - 1) // 2
    z = every // (nx * ny) - (nz - 1) // 2
    return np.stack([x, y, z], 1).astype(np.int32)


def _macro(rng, dim):
    v = rng.uniform(-0.01, 0.01, 6)
    if dim == 2:
        v[2:5] = 0.0
    return v


def _single(case, seed):
    """Phase map, pattern and macroscopic strain (or path [T, 6]) of one microstructure."""
    rng = np.random.default_rng(seed)
    shape = _shape(case)
    pm = _micro(rng, shape, case["r_lo"], case["r_hi"], case["vf"])
    pat = _adapted(pm, _k_target(case["ratio"], pm.size))
    if case["kind"] == "path":
        last = np.array([0.01, -0.01, 0, 0, 0, 0.002] if case["law"].startswith("paper")
                        else [0.02, 0, 0, 0, 0, 0], float)
        last = last * rng.uniform(0.9, 1.0)
        return pm, pat, last * (np.arange(1, case["steps"] + 1) / case["steps"])[:, None]
    return pm, pat, _macro(rng, len(shape))


def _points(case, seed):
    """Phase maps and patterns of the batch's microstructures, the points' microstructures and
    macroscopic strains."""
    rng = np.random.default_rng(seed)
    pms = []
    for i in range(case["micros"]):
        if case["odd"]:
            shape = tuple(int(v) for v in rng.integers(case["lo"], case["hi"] + 1, 2))
        else:
            sides = [s for s in BATCH_SIDES if case["lo"] <= s <= case["hi"]]
            shape = (sides[i % len(sides)],) * 2
        pms.append(_micro(rng, shape, 8.0, 24.0, rng.uniform(0.2, 0.5)))
    pats = [_adapted(pm, _k_target(case["ratio"], pm.size)) for pm in pms]
    which = np.arange(case["points"]) % case["micros"]
    return pms, pats, which, np.array([_macro(rng, 2) for _ in which])


def _room(case):
    """Slots that a batch of this case can have at most: half of each pattern and its kx = 0."""
    n = case["points"] * case["hi"] ** 2
    return int(case["ratio"] * n / 2) + case["points"] * (case["hi"] + 2)


def _harmonics(a, b):
    r2 = a * a + b * b
    c2, s2 = (a * a - b * b) / r2, 2.0 * a * b / r2
    c4, s4 = c2 * c2 - s2 * s2, 2.0 * s2 * c2
    c6, s6 = c4 * c2 - s4 * s2, s4 * c2 + c4 * s2
    c8, s8 = c4 * c4 - s4 * s4, 2.0 * s4 * c4
    return torch.stack([torch.ones_like(a), c2, s2, c4, s4, c6, s6, c8, s8], -1)


def _training(case, seed):
    """Network inputs of a minibatch in 64 bits: descriptors, unit strains, slot table, offsets,
    targets (a few updates of the scheme), parameters."""
    rng = np.random.default_rng(seed)
    dev, side, B = _dev(), case["side"], case["cells"]
    pms = np.stack([_micro(rng, (side, side), 8.0, 24.0, rng.uniform(0.2, 0.5)) for _ in range(B)])
    pats = [_adapted(pm, _k_target(case["ratio"], pm.size)) for pm in pms]
    macros = np.array([_macro(rng, 2) for _ in range(B)])
    _, hat, _, _ = _reference(pms, "fibre", pats, macros[None], TOL, 12)
    N = float(side * side)
    e6 = torch.as_tensor(macros, device=dev)
    en = torch.sqrt(e6[:, 0] ** 2 + e6[:, 1] ** 2 + 2 * e6[:, 5] ** 2)
    e = torch.stack([e6[:, 0], e6[:, 1], e6[:, 5]], 1) / en[:, None]
    gam = torch.fft.fftn(torch.as_tensor(pms, device=dev).double(), dim=(1, 2)) / N
    x = torch.zeros((B, N_IN), dtype=torch.float64, device=dev)
    slots, targets, offsets = [], [], [0]
    for r in range(B):
        p = torch.as_tensor(pats[r], device=dev).long()
        p = p[p[:, 0] >= 0]
        p = p[torch.argsort(p[:, 0] * 4096 + p[:, 1])]
        zero = (p[:, 0] == 0) & (p[:, 1] == 0)
        null = (p[:, 0] * 2 == side) & (p[:, 1] * 2 == side)
        self_ = (p[:, 0] == 0) | (p[:, 0] * 2 == side)
        w = torch.where(zero | null, 0.0, torch.where(self_, 1.0, 2.0)).double()
        g = gam[r][p[:, 1] % side, p[:, 0] % side]
        a, b = p[:, 0] / side, p[:, 1] / side
        a, b = a.double(), b.double()
        pw = (g.abs() ** 2) * torch.where(zero, 0.0, torch.where(self_, 1.0, 2.0))
        bins = torch.clamp(torch.floor(96.0 * torch.sqrt(a * a + b * b)), max=23).long()
        h = _harmonics(torch.where(zero, torch.ones_like(a), a), b)
        rad = torch.zeros(24, dtype=torch.float64, device=dev).index_add_(0, bins, pw)
        x[r, 0] = g[zero][0].real
        x[r, 1:25] = torch.sqrt(rad)
        for j in range(4):
            sel = pw * (bins // 6 == j)
            x[r, 25 + 4 * j:29 + 4 * j] = (sel[:, None] * h[:, 1:5]).sum(0) / (sel.sum() + 1e-12)
        x[r, 41] = torch.sqrt(pw.sum())
        kind = torch.where(zero, 1, torch.where(null, 2, 0))
        slots.append((g, a, b, w, kind))
        c = hat[r][:, p[:, 1] % side, p[:, 0] % side] / (N * en[r])
        c = torch.where(w > 0, c, torch.zeros_like(c))
        targets.append(torch.view_as_real(c.T.contiguous()).reshape(-1, 6))
        offsets.append(offsets[-1] + len(p))
    cat = [torch.cat([s[i] for s in slots]) for i in range(5)]
    rve = torch.repeat_interleave(torch.arange(B, device=dev),
                                  torch.tensor(np.diff(offsets), device=dev))
    H = case["hidden"]
    sh = [(N_IN, H), (H,), (H, H), (H,), (H, N_OUT), (N_OUT,)]
    par = [rng.standard_normal(s) / math.sqrt(s[0]) * (0.1 if i == 4 else 1.0) if len(s) == 2
           else 0.01 * rng.standard_normal(s) for i, s in enumerate(sh)]
    f32 = torch.float32
    return dict(x=x.to(f32), e=e.to(f32), g=cat[0].to(torch.complex64), a=cat[1].to(f32),
                b=cat[2].to(f32), w=cat[3].to(f32), kind=cat[4], rve=rve, inv_n=1.0 / N,
                t=torch.cat(targets).to(f32), offsets=np.array(offsets, np.int64),
                params=[p.astype(np.float32) for p in par])


def _slot_table(d):
    """The [slots, 8] float32 view of the slot records (two int32 words at the end)."""
    n = d["a"].shape[0]
    tab = torch.empty((n, 8), dtype=torch.float32, device=d["a"].device)
    tab[:, 0], tab[:, 1] = d["g"].real, d["g"].imag
    tab[:, 2], tab[:, 3], tab[:, 4], tab[:, 5] = d["a"], d["b"], d["w"], d["inv_n"]
    ints = torch.stack([d["rve"], d["kind"]], 1).to(torch.int32).contiguous()
    tab.view(torch.int32)[:, 6:8] = ints
    return tab


# --------------------------------------------------------------------------- preparation, passes
def prepare(case, seed):
    from paper_2103_10203_gb300 import rf
    kind = case["kind"]
    if kind == "pattern":
        rng = np.random.default_rng(seed)
        pm = _micro(rng, _shape(case), case["r_lo"], case["r_hi"], case["vf"])
        return dict(kind=kind, rf=rf, pm=pm, k=_k_target(case["ratio"], pm.size))
    if kind == "batch":
        pms, pats, which, macros = _points(case, seed)
        stream = torch.cuda.Stream()
        b = rf.BatchSolver([pms[i] for i in which], _phases(case["law"]), [pats[i] for i in which],
                           stream=stream.cuda_stream, tol=TOL, max_iter=MAX_ITER,
                           transform=case["transform"])
        return dict(kind=kind, b=b, macros=macros, stream=stream,
                    room=torch.zeros((_room(case), 3, 2), device="cuda"))
    if kind == "train":
        d = _training(case, seed)
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        net = rf.WarmStartNet(n_hidden=case["hidden"], max_batch=case["cells"], stream=stream)
        net.rf_mlp_set_params(np.concatenate([p.ravel() for p in d["params"]]))
        return dict(kind=kind, net=net, x=d["x"].contiguous(), e=d["e"].contiguous(),
                    slots=_slot_table(d), t=d["t"].contiguous(), stream=stream,
                    offsets=torch.as_tensor(d["offsets"], device="cuda"))
    pm, pat, load = _single(case, seed)
    s = rf.Solver(pm, _phases(case["law"]), pattern=pat, tol=TOL, max_iter=MAX_ITER,
                  transform=case.get("transform", "fft"), precision=case.get("precision", "fp32"))
    if kind == "study":   # the full-set context of the compatibility step, kept by the solver
        s.rf_solve(load)
        s.rf_compat()
    return dict(kind=kind, s=s, load=load)


def run(state):
    kind = state["kind"]
    if kind == "solve":
        out = state["s"].rf_solve(state["load"])
        return dict(stress=out["sigma_bar"].astype(np.float32),
                    strain=state["s"].rf_get_reduced_strain())
    if kind == "path":
        s = state["s"]
        s.rf_reset_path()
        out = s.rf_solve_path(state["load"])
        return dict(stress=out["sigma_bar"].astype(np.float32), strain=s.rf_get_reduced_strain(),
                    fields=s.rf_get_fields())
    if kind == "study":
        s = state["s"]
        out = s.rf_solve(state["load"])
        comp = s.rf_compat()
        return dict(stress=out["sigma_bar"].astype(np.float32), compat=comp.astype(np.float32),
                    fields=s.rf_get_fields())
    if kind == "batch":
        with torch.cuda.stream(state["stream"]):
            out = state["b"].rf_batch_solve(state["macros"])
            strain = state["b"].rf_batch_reduced_strain()
            state["room"][:len(strain)] = strain
            return dict(stress=out["sigma_bar"].astype(np.float32), strain=state["room"])
    if kind == "pattern":
        return state["rf"].rf_pattern_adapted(state["pm"], 1, state["k"])
    with torch.cuda.stream(state["stream"]):
        net = state["net"]
        loss = net.rf_mlp_loss_grad(state["x"], state["e"], state["slots"], state["offsets"],
                                    state["t"])
        return dict(loss=np.float32(loss), grads=net.rf_mlp_get_grads())


# --------------------------------------------------------------------------- work
# updates of the scheme to 1e-6 that the laws' stiffness contrasts need (typical counts; the J2
# laws' per increment of a path into the plastic range)
_UPDATES = {"fibre": 30, "paper": 10, "fibre_j2": 165, "paper_j2": 270}


def _update_flops(n, sides, nc, ratio, plastic):
    """One update: the law at every voxel, real transforms along x of every line and complex ones
    along the other axes of the lines that the pattern keeps, both ways."""
    keep = 1.0
    f = nc * 2.5 * math.log2(max(2, sides[0])) * n
    for d, m in enumerate(sides[1:]):
        keep *= min(1.0, 0.5 * ratio ** (1.0 / len(sides)) * 1.5 if d == 0 else
                    ratio ** (1.0 / len(sides)) * 1.5)
        f += nc * 5.0 * math.log2(max(2, m)) * n * keep
    return 2.0 * f + n * ((40 if nc == 3 else 80) + (60 if plastic else 0)) + 60.0 * ratio * n


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sides = ([s for s in BATCH_SIDES if case["lo"] <= s <= case["hi"]] if not case["odd"]
                 else [(case["lo"] + case["hi"]) // 2])
        n = case["points"] * sum(s * s for s in sides) / len(sides)
        fl = _update_flops(n, (sides[len(sides) // 2],) * 2, 3, case["ratio"], False)
        return dict(bytes=n + n * case["ratio"] * 0.5 * (24 + 8), flops=_UPDATES["fibre"] * fl)
    if kind == "train":
        B, H = case["cells"], case["hidden"]
        par = N_IN * H + H + H * H + H + H * N_OUT + N_OUT
        slots = B * case["side"] ** 2 * case["ratio"] * 0.5
        return dict(bytes=8.0 * par + slots * 56 + B * 4 * (N_IN + 3),
                    flops=6.0 * B * par + slots * (4 * N_OUT + 40))
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "pattern":
        return dict(bytes=n + 12.0 * case["ratio"] * n, flops=2.5 * n * math.log2(n))
    nc = 3 if case["nz"] == 1 else 6
    sides = (case["nx"], case["ny"]) + ((case["nz"],) if nc == 6 else ())
    plastic = case["law"].endswith("_j2")
    steps = case.get("steps", 1)
    fl = _update_flops(n, sides, nc, case["ratio"], plastic) * _UPDATES[case["law"]] * steps
    by = n * (1 + (32 * steps if plastic else 0)) + case["ratio"] * n * (8 + 48)
    if kind == "study":
        fl += _update_flops(n, sides, nc, 1.0, False)
    if kind in ("study", "path"):
        by += 52.0 * n
    return dict(bytes=by, flops=fl)


# --------------------------------------------------------------------------- 64-bit results
def _reference(pms, law, pats, path, tol, max_iter, compat=False):
    """The scheme in 64 bits for B cells of one shape: pms [B, ...], a pattern for each, path
    [T][B, 6]. Returns (stress [T, B, 6], coefficients [B, nc, ...] of the last increment,
    strain and stress fields [B, 6, N], alpha [B, N]) (the fields after the compatibility step
    with `compat`; its average stress is then appended to the first)."""
    dev = _dev()
    pm = torch.as_tensor(np.asarray(pms), device=dev).long()
    B, sh = pm.shape[0], tuple(pm.shape[1:])
    d = len(sh)
    N = math.prod(sh)
    comps = (0, 1, 5) if d == 2 else tuple(range(6))
    tab = torch.tensor(LAWS[law], dtype=torch.float64, device=dev)
    lam, mu, sy, H = (tab[:, i][pm] for i in range(4))
    plastic = tab[:, 4][pm] != 0
    lam0, mu0 = (0.5 * (float(tab[:, i].min()) + float(tab[:, i].max())) for i in (0, 1))
    # unit wave vectors of the rotated finite differences
    t = [math.pi * _signed(n, dev).double() / n for n in sh]
    t = list(torch.meshgrid(*t, indexing="ij"))[::-1]   # x first
    q = []
    for j in range(d):
        v = 2.0 * torch.sin(t[j])
        for m in range(d):
            if m != j:
                v = v * torch.cos(t[m])
        q.append(v)
    nq = torch.sqrt(sum(v * v for v in q))
    null = nq < 1e-9
    n3 = [v / torch.where(null, torch.ones_like(nq), nq) for v in q]
    n3 = n3 + [torch.zeros_like(nq)] * (3 - d)
    mask = torch.zeros((B,) + sh, dtype=torch.bool, device=dev)
    for b in range(B):
        p = torch.as_tensor(pats[b], device=dev).long()
        ix = tuple(p[:, d - 1 - i] % sh[i] for i in range(d))
        mask[(b,) + ix] = True
    mask &= ~null
    cg = (lam0 + mu0) / (mu0 * (lam0 + 2.0 * mu0))
    axes = tuple(range(2, 2 + d))
    zero = (slice(None), slice(None)) + (0,) * d

    def full6(f):
        if d == 3:
            return [f[:, i] for i in range(6)]
        z = torch.zeros_like(f[:, 0])
        return [f[:, 0], f[:, 1], z, z, z, f[:, 2]]

    def stress(eps, ep, al):
        e = full6(eps)
        ee = [e[i] - ep[i] for i in range(6)] if ep is not None else e
        tr = ee[0] + ee[1] + ee[2]
        s = [2 * mu * ee[i] + (lam * tr if i < 3 else 0.0) for i in range(6)]
        if ep is None:
            return s, None, None
        p = (s[0] + s[1] + s[2]) / 3.0
        dv = [s[i] - p if i < 3 else s[i] for i in range(6)]
        seq = torch.sqrt(1.5 * (dv[0] ** 2 + dv[1] ** 2 + dv[2] ** 2 +
                                2 * (dv[3] ** 2 + dv[4] ** 2 + dv[5] ** 2)))
        phi = seq - (sy + H * al)
        y = plastic & (phi > 0)
        dg = torch.where(y, phi / (3 * mu + H), torch.zeros_like(phi))
        fl = 1.5 * dg / torch.where(y, seq, torch.ones_like(seq))
        return ([s[i] - 2 * mu * fl * dv[i] for i in range(6)],
                [ep[i] + fl * dv[i] for i in range(6)], al + dg)

    def update(eps, ep, al, ebar, keep):
        s, _, _ = stress(eps, ep, al)
        e = full6(eps)
        tr = e[0] + e[1] + e[2]
        tau = torch.stack([s[i] - 2 * mu0 * e[i] - (lam0 * tr if i < 3 else 0.0) for i in comps], 1)
        del s, e, tr
        th = full6(torch.fft.fftn(tau, dim=axes))
        v = [th[0] * n3[0] + th[5] * n3[1] + th[4] * n3[2],
             th[5] * n3[0] + th[1] * n3[1] + th[3] * n3[2],
             th[4] * n3[0] + th[3] * n3[1] + th[2] * n3[2]]
        del th
        nvn = n3[0] * v[0] + n3[1] * v[1] + n3[2] * v[2]
        out = []
        for c in comps:
            i, j = VOIGT[c]
            g = (n3[i] * v[j] + n3[j] * v[i]) / (2 * mu0) - cg * n3[i] * n3[j] * nvn
            out.append(torch.where(keep, -g, torch.zeros_like(g)))
        hat = torch.stack(out, 1)
        hat[zero] = (N * ebar[:, list(comps)]).to(hat.dtype)
        return hat, torch.fft.ifftn(hat, dim=axes).real

    weight = torch.tensor([1.0 if c < 3 else 2.0 for c in comps], dtype=torch.float64, device=dev)
    weight = weight.reshape((1, -1) + (1,) * d)
    path = torch.as_tensor(np.asarray(path), dtype=torch.float64, device=dev)
    any_plastic = bool((tab[:, 4] != 0).any())
    zf = torch.zeros((B,) + sh, dtype=torch.float64, device=dev)
    ep = [zf.clone() for _ in range(6)] if any_plastic else None
    al = zf.clone() if any_plastic else None
    eps = torch.zeros((B, len(comps)) + sh, dtype=torch.float64, device=dev)
    prev = torch.zeros((B, 6), dtype=torch.float64, device=dev)
    hat, sbar = None, []
    col = (slice(None), slice(None)) + (None,) * d
    for ebar in path:
        eps = eps + (ebar - prev)[:, list(comps)][col]
        prev = ebar
        en = torch.sqrt((ebar ** 2 * torch.tensor([1., 1, 1, 2, 2, 2], device=dev)).sum(1))
        live = torch.ones(B, dtype=torch.bool, device=dev)
        for _ in range(max_iter):
            h, new = update(eps, ep, al, ebar, mask)
            r = torch.sqrt((weight * (new - eps) ** 2).flatten(1).sum(1) / N) / en
            sel = live.reshape((B, 1) + (1,) * d)
            eps = torch.where(sel, new, eps)
            hat = h if hat is None or bool(live.all()) else torch.where(sel, h, hat)
            live = live & (r >= tol)
            if not bool(live.any()):
                break
        s, epn, aln = stress(eps, ep, al)
        if any_plastic:
            ep, al = epn, aln
        sbar.append(torch.stack([v.flatten(1).mean(1) for v in s], 1))
    if compat:
        _, eps = update(eps, ep, al, prev, (~null).expand_as(mask))
        s, _, _ = stress(eps, ep, al)
        sbar.append(torch.stack([v.flatten(1).mean(1) for v in s], 1))
    fields = (torch.stack([v.expand_as(zf) for v in full6(eps)], 1), torch.stack(s, 1),
              al if al is not None else zf)
    return torch.stack(sbar), hat, fields, mask


def _coefficients(hat, pat, sh):
    """[K, 6, 2] of one cell's coefficients in the pattern's order."""
    p = torch.as_tensor(pat, device=hat.device).long()
    d = len(sh)
    v = hat[(slice(None),) + tuple(p[:, d - 1 - i] % sh[i] for i in range(d))].T
    out = torch.zeros((len(p), 6, 2), dtype=torch.float64, device=hat.device)
    out[:, list((0, 1, 5) if d == 2 else range(6))] = torch.view_as_real(v.contiguous())
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "pattern":
        return None   # whole numbers
    if kind == "batch":
        pms, pats, which, macros = _points(case, seed)
        stress = torch.zeros((len(which), 6), dtype=torch.float64, device=_dev())
        parts = [None] * len(which)
        for shape in sorted({pm.shape for pm in pms}):
            ids = [i for i, w in enumerate(which) if pms[w].shape == shape]
            for c in range(0, len(ids), 128):
                part = ids[c:c + 128]
                sb, hat, _, _ = _reference([pms[which[i]] for i in part], case["law"],
                                           [pats[which[i]] for i in part], macros[part][None],
                                           TOL, MAX_ITER)
                for k, i in enumerate(part):
                    p = pats[which[i]]
                    p = p[p[:, 0] >= 0]
                    p = p[np.lexsort((p[:, 1], p[:, 0]))]
                    stress[i] = sb[0, k]
                    parts[i] = _coefficients(hat[k], p, shape)[:, [0, 1, 5]]
        strain = torch.cat(parts)
        room = torch.zeros((_room(case), 3, 2), dtype=strain.dtype, device=strain.device)
        room[:len(strain)] = strain
        return dict(stress=stress, strain=room)
    if kind == "train":
        d = _training(case, seed)
        par = [torch.tensor(p, device=d["x"].device).double().requires_grad_() for p in d["params"]]
        gelu = torch.nn.functional.gelu
        h = gelu(d["x"].double() @ par[0] + par[1])
        h = gelu(h @ par[2] + par[3])
        o = (h @ par[4] + par[5]).reshape(-1, 9, N_BASIS)
        a, b, w, rve = d["a"].double(), d["b"].double(), d["w"].double(), d["rve"]
        reg = d["kind"] == 0
        a1 = torch.where(reg, a, torch.ones_like(a))
        rho = (torch.sqrt(a1 * a1 + b * b) / 0.25)[:, None]
        hm = _harmonics(a1, b)
        phi = torch.cat([hm, hm * rho, hm * rho * rho], 1)
        T = torch.einsum("sin,sn->si", o[rve], phi).reshape(-1, 3, 3)
        amp = torch.einsum("scd,sd->sc", T, d["e"].double()[rve])
        g = d["g"].to(torch.complex128)
        t = d["t"].double().reshape(-1, 3, 2)
        res = (amp * g.real[:, None] - t[..., 0]) ** 2 + (amp * g.imag[:, None] - t[..., 1]) ** 2
        loss = (res * w[:, None]).sum() / (6.0 * w.sum())
        grads = torch.autograd.grad(loss, par)
        return dict(loss=loss.detach(), grads=torch.cat([v.flatten() for v in grads]))
    pm, pat, load = _single(case, seed)
    path = load[:, None] if kind == "path" else load[None, None]
    sb, hat, fields, _ = _reference(pm[None], case["law"], [pat], path, TOL, MAX_ITER,
                                    compat=kind == "study")
    sh = pm.shape
    vox = (fields[0][0].reshape((6,) + sh), fields[1][0].reshape((6,) + sh), fields[2][0].reshape(sh))
    if kind == "study":
        return dict(stress=sb[0, 0], compat=sb[1, 0], fields=vox)
    out = dict(stress=sb[:, 0] if kind == "path" else sb[0, 0],
               strain=_coefficients(hat[0], pat, sh))
    if kind == "path":
        out["fields"] = vox
    return out
