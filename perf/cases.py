"""What is timed: the calls a user of this framework makes, over the range of sizes in real use.

Four kinds of case:

* ``rad``: a kept radiation context takes a batch of leapfrog states and returns the spectra
  (reset, accumulate_steps, finalize): one window of a simulation, one run of a data set, one
  shard of a population;
* ``pic``: the live two-stream PIC from the caller's particles for some steps, fields and
  particles read back;
* ``insitu``: the same PIC handing its tracked electrons to a radiation context every step;
* ``train`` / ``predict``: the surrogate network's training steps and predictions.

Trajectories are closed-form magnetic deflections: |u| constant per particle, the direction a
sum of slow oscillations of the size a B_rms = 0.1 field gives (angular rate 0.1 / gamma), two
beams along +-x, positions the exact leapfrog sum of dt u / gamma wrapped into the periodic box
of side 40.  dt is 0.05 as in the workloads.

Spectra of the FP32 path are returned as float32 (what the surrogate's data set stores: its
arithmetic is 32-bit), those of the FP64 path as float64.
"""
import math

import numpy as np
import torch

L_BOX = 40.0
DT = 0.05
MASS_RATIO = 64.0            # the PIC's partner species


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _rad(name, precision, electrons, ions, gamma, samples, dirs, omegas, lo, hi, spacing="log",
         coherent=False, windows="one", selectors=False, host=False):
    return {"name": name, "kind": "rad", "precision": precision, "electrons": electrons,
            "ions": ions, "gamma": gamma, "samples": samples, "dirs": dirs, "omegas": omegas,
            "lo": lo, "hi": hi, "spacing": spacing, "coherent": coherent, "windows": windows,
            "selectors": selectors, "host": host}


def listed():
    return [
        # the smallest call: a quick look at a few dozen particles (launch latency)
        _rad("smoke_window", "fp32", 37, 0, 3.0, 200, 3, 96, 0.1, 300.0, windows="nested"),
        # the exact sparse subset the surrogate starts from: 12 directions x 64 omega per run
        _rad("sparse_subset", "fp32", 1024, 0, 4.0, 2000, 12, 64, 0.1, 1000.0),
        # one dense map of the surrogate's data set: 192 directions x 2048 omega per run
        _rad("dense_map", "fp32", 1024, 0, 4.0, 2000, 192, 2048, 0.1, 1000.0),
        # a shard of the headline population: gamma 10 beams, 4096 samples, 8 directions, 1024
        # omega; a ragged count (8195 = 1024 tiles of 8 and 3 particles)
        _rad("precision_shard", "fp32", 8195, 0, 10.0, 4096, 8, 1024, 0.1, 1000.0),
        # batched run of electrons and ions, phase-coherent, uneven windows with direction
        # subsets on two grids, regions and pitch cones; odd sizes throughout
        _rad("coherent_batch", "fp32", 1501, 171, 3.0, 1100, 24, 330, 0.1, 300.0, coherent=True,
             windows="uneven", selectors=True),
        # states arriving in pinned host memory, linear frequency bins
        _rad("host_batches", "fp32", 6007, 0, 3.0, 1536, 6, 512, 0.5, 60.0, spacing="lin",
             host=True),
        # the plain FP64 spectrum: 1024 electrons, one observer, 256 omega
        _rad("fp64_observer", "fp64", 1024, 0, 3.0, 2000, 1, 256, 0.1, 300.0),
        # FP64, phase-coherent, two species, uneven windows and selectors at ragged sizes
        _rad("fp64_coherent", "fp64", 301, 47, 3.0, 500, 8, 150, 0.1, 300.0, coherent=True,
             windows="uneven", selectors=True),
        # the live PIC alone at the in-situ application's size (1,048,576 particles)
        {"name": "pic_run", "kind": "pic", "n": 256, "ppc": 4, "gamma": 3.0, "steps": 16},
        # the PIC driving the diagnostic every step (launch-bound: 65,536 particles, 4096 tracked)
        {"name": "insitu_run", "kind": "insitu", "n": 64, "ppc": 4, "gamma": 3.0, "steps": 96,
         "tracked": 4096, "omegas": 256},
        # the surrogate at full width: four Adam steps, updated weights read back
        {"name": "train_steps", "kind": "train", "width_in": 768, "hidden": 512,
         "width_out": 393216, "batch": 128, "steps": 4},
        # its prediction for a ragged batch of raw sparse spectra
        {"name": "predict_batch", "kind": "predict", "width_in": 768, "hidden": 512,
         "width_out": 393216, "batch": 100},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp32", "fp32", "fp32", "fp32", "fp64", "fp64", "pic", "insitu", "train",
                       "predict"])
    if kind in ("fp32", "fp64"):
        cap = 1.2e11 if kind == "fp32" else 1.2e9
        while True:
            c = _rad("", kind, _log_int(rng, 8, 9000), rng.choice([0, 0, _log_int(rng, 1, 400)]),
                     rng.choice([2.0, 3.0, 5.0, 10.0]), _log_int(rng, 33, 4096),
                     _log_int(rng, 1, 192), _log_int(rng, 16, 2048), rng.choice([0.01, 0.1, 0.5]),
                     rng.choice([30.0, 300.0, 1000.0]), rng.choice(["log", "log", "log", "lin"]),
                     rng.random() < 0.3, rng.choice(["one", "one", "nested", "uneven"]),
                     rng.random() < 0.2, rng.random() < 0.2)
            del c["name"]
            if 1e5 <= _updates(c) <= cap and _out_len(c) <= 500000:
                return c
    if kind == "pic":
        return {"kind": "pic", "n": rng.randrange(24, 257), "ppc": rng.choice([1, 2, 4]),
                "gamma": rng.choice([2.0, 3.0, 10.0]), "steps": rng.randrange(2, 17)}
    if kind == "insitu":
        n, ppc = rng.randrange(24, 129), rng.choice([1, 2, 4])
        return {"kind": "insitu", "n": n, "ppc": ppc, "gamma": 3.0,
                "steps": rng.randrange(8, 97), "tracked": _log_int(rng, 32, 2 * ppc * n * n),
                "omegas": _log_int(rng, 16, 512)}
    c = {"kind": kind, "width_in": 128 * rng.randrange(1, 9), "hidden": 128 * rng.randrange(1, 5),
         "width_out": 128 * _log_int(rng, 4, 3072), "batch": _log_int(rng, 1, 256)}
    if kind == "train":
        c["steps"] = rng.randrange(1, 5)
    return c


# ---------------------------------------------------------------------------
# geometry shared by the cases
# ---------------------------------------------------------------------------
def _dirs(count):
    """x, y, an oblique one and -x first, then an even cover of the sphere."""
    base = [(1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (1.0, 1.0, 1.0), (-1.0, 0.0, 0.0)]
    i = np.arange(max(0, count - 4)) + 0.5
    z = 1.0 - 2.0 * i / max(1, count - 4)
    phi = math.pi * (1.0 + math.sqrt(5.0)) * i
    s = np.sqrt(1.0 - z * z)
    cover = np.stack([s * np.cos(phi), s * np.sin(phi), z], 1)
    d = np.concatenate([np.array(base), cover])[:count]
    return d / np.linalg.norm(d, axis=1, keepdims=True)


def _grids(c):
    n = c["omegas"]
    full = (np.exp(np.linspace(math.log(c["lo"]), math.log(c["hi"]), n)) if c["spacing"] == "log"
            else np.linspace(c["lo"], c["hi"], n))
    return [full] if c["windows"] != "uneven" else [full, full[: max(1, n // 2)].copy()]


def _windows(c):
    """(s0, s1, species mask, grid, direction subset or None)."""
    S, D = c["samples"], c["dirs"]
    both = 3 if c["ions"] else 1
    if c["windows"] == "one":
        return [(0, S, both, 0, None)]
    if c["windows"] == "nested":
        return [(0, S, both, 0, None), (S // 15, 3 * S // 4, 1, 0, None)]
    half = list(range(0, D, 2))
    return [(0, S, both, 0, None), (S // 3, S // 3 + S // 2, 1, 1, half),
            (S // 4 + 1, S // 2 + 3, both, 1, None)]


def _selectors(c):
    """A spatial region for the first window, a pitch cone for the second."""
    sel = [{"kind": "box", "lo": [0.0, 5.0, 0.0], "hi": [40.0, 40.0, 33.0]},
           {"kind": "cone", "axis": [1.0, 0.0, 0.0], "theta_c": 0.0, "dtheta": 0.6}]
    w = [-1] * len(_windows(c))
    w[0] = 0
    if len(w) > 1:
        w[1] = 1
    return sel, w


def _counts(c):
    return [c["electrons"], c["ions"]] if c["ions"] else [c["electrons"]]


def _species(c):
    return [(c["electrons"], -1.0, 1.0)] + ([(c["ions"], 1.0, 16.0)] if c["ions"] else [])


def _masked(c, mask):
    return sum(n for i, n in enumerate(_counts(c)) if (mask >> i) & 1)


def _updates(c):
    g = [len(x) for x in _grids(c)]
    return sum(_masked(c, m) * (s1 - s0) * (len(ds) if ds else c["dirs"]) * g[gi]
               for s0, s1, m, gi, ds in _windows(c))


def _out_len(c):
    g = [len(x) for x in _grids(c)]
    return sum((len(ds) if ds else c["dirs"]) * g[gi] for _, _, _, gi, ds in _windows(c))


def _rng(seed, device="cuda"):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return g


def _trajectory(counts, gamma, calls, seed):
    """X, U [calls][3][N] FP64 on the GPU: call s holds x_s and u_{s-1/2}."""
    g = _rng(seed)
    N = sum(counts)
    u = lambda *shape: torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    rate = torch.full((N,), 0.1 / gamma, dtype=torch.float64, device="cuda")
    rate[counts[0]:] /= 16.0                            # ions are 16 times heavier
    umag = math.sqrt(gamma * gamma - 1.0) * (1.0 + 0.05 * (2.0 * u(N) - 1.0))
    gam = torch.sqrt(1.0 + umag * umag)
    sign = torch.ones(N, dtype=torch.float64, device="cuda")
    sign[1::2] = -1.0                                   # two beams, alternating
    t = (torch.arange(calls, dtype=torch.float64, device="cuda") - 0.5)[:, None] * DT
    ang = []
    for _ in range(2):
        a = torch.zeros((calls, N), dtype=torch.float64, device="cuda")
        a += 0.1 * (2.0 * u(N) - 1.0)
        for _ in range(3):
            w = 0.2 + 1.8 * u(N)
            a += (rate / w) * torch.sin(w * t + 2.0 * math.pi * u(N))
        ang.append(a)
    X = torch.empty((calls, 3, N), dtype=torch.float64, device="cuda")
    U = torch.empty_like(X)
    U[:, 0] = sign * umag * torch.cos(ang[0]) * torch.cos(ang[1])
    U[:, 1] = umag * torch.sin(ang[0]) * torch.cos(ang[1])
    U[:, 2] = umag * torch.sin(ang[1])
    X[0] = L_BOX * u(3, N)
    X[1:] = U[1:] * (DT / gam)
    torch.cumsum(X, 0, out=X)
    X -= L_BOX * torch.floor(X / L_BOX)
    return X, U


# ---------------------------------------------------------------------------
# the radiation context
# ---------------------------------------------------------------------------
def _prepare_rad(c, seed):
    from paper_1003_1140_gb300 import rad as R
    X, U = _trajectory(_counts(c), c["gamma"], c["samples"] + 1, seed)
    if c["host"]:
        X, U = X.cpu().pin_memory(), U.cpu().pin_memory()
    fp64 = c["precision"] == "fp64"
    ctx = R.Radiation(_dirs(c["dirs"]), _grids(c), DT, _species(c), _windows(c),
                      mode=R.RAD_COHERENT if c["coherent"] else R.RAD_INCOHERENT,
                      precision=R.RAD_FP64 if fp64 else R.RAD_FP32_SPLIT, box_L=L_BOX)
    if c["selectors"]:
        ctx.set_selectors(*_selectors(c))
    return {"case": c, "ctx": ctx, "X": X, "U": U,
            "out": torch.empty(ctx.spectrum_size(), dtype=torch.float64, device="cuda")}


def _split(c, spec):
    """Per window: the spectra of the directions exact() covers, then the others."""
    res, off, q = [], 0, _exact_dirs(c)
    g = [len(x) for x in _grids(c)]
    for _, _, _, gi, ds in _windows(c):
        nd = len(ds) if ds else c["dirs"]
        S = spec[off:off + nd * g[gi]].view(nd, g[gi])
        off += nd * g[gi]
        k = min(q, nd)
        res.append([S[:k], S[k:]] if k < nd else [S])
    return res


def _run_rad(s):
    c, ctx = s["case"], s["ctx"]
    ctx.reset()
    ctx.accumulate_steps(0, s["X"], s["U"])
    out = ctx.finalize(s["out"])
    return _split(c, out if c["precision"] == "fp64" else out.float())


def _exact_dirs(c):
    """Leading directions of every window that exact() evaluates within a few seconds."""
    return max(0, min(c["dirs"], int(3.5e10 // (_updates(c) / c["dirs"]))))


def _exact_spectra(X, U, dt, L, dirs, omegas, windows, counts, charges, coherent, sel=None, q=None):
    """The definition in FP64: S = |sum_m q V e^{i w phi} dt|^2 / 4 pi^2 per particle
    (incoherent) or of the sum over particles (coherent)."""
    n = torch.zeros_like(X)
    n[1:] = -torch.cumsum(torch.round((X[1:] - X[:-1]) / L), 0)
    r = (X + L * n)[:-1]
    ub = 0.5 * (U[:-1] + U[1:])
    beta = ub / torch.sqrt(1.0 + (ub * ub).sum(1, keepdim=True))
    bh = U / torch.sqrt(1.0 + (U * U).sum(1, keepdim=True))
    bdot = (bh[1:] - bh[:-1]) / dt
    chg = torch.cat([torch.full((k,), z, dtype=torch.float64, device="cuda")
                     for k, z in zip(counts, charges)])
    first = np.concatenate([[0], np.cumsum(counts)])
    res = []
    for wi, (s0, s1, mask, gi, ds) in enumerate(windows):
        w = torch.as_tensor(omegas[gi], dtype=torch.float64, device="cuda")
        rows = list(ds) if ds else list(range(len(dirs)))
        k = len(rows) if q is None else min(q, len(rows))
        S = torch.zeros((k, len(w)), dtype=torch.float64, device="cuda")
        parts = [slice(int(first[i]), int(first[i + 1])) for i in range(len(counts))
                 if (mask >> i) & 1]
        keep = None
        if sel is not None and sel[1][wi] >= 0:
            d = sel[0][sel[1][wi]]
            if d["kind"] == "box":
                x = X[s0:s1]
                keep = torch.ones_like(x[:, 0], dtype=torch.bool)
                for a in range(3):
                    keep &= (x[:, a] >= d["lo"][a]) & (x[:, a] < d["hi"][a])
            else:
                ax = torch.tensor(d["axis"], dtype=torch.float64, device="cuda")
                cs = torch.einsum("mcj,c->mj", ub[s0:s1], ax) / ub[s0:s1].norm(dim=1)
                keep = ((cs >= math.cos(min(math.pi, d["theta_c"] + d["dtheta"]))) &
                        (cs <= math.cos(max(0.0, d["theta_c"] - d["dtheta"]))))
        for row in range(k):
            nv = torch.as_tensor(dirs[rows[row]], dtype=torch.float64, device="cuda")
            tot = torch.zeros((2, 3, len(w)), dtype=torch.float64, device="cuda")
            for sl in parts:
                b, bd = beta[s0:s1, :, sl], bdot[s0:s1, :, sl]
                nb = torch.einsum("mcj,c->mj", b, nv)
                nbd = torch.einsum("mcj,c->mj", bd, nv)
                kap = 1.0 - nb
                V = ((nv[None, :, None] - b) * nbd[:, None] - bd * kap[:, None]) / (kap * kap)[:, None]
                V *= (chg[sl] * dt)
                if keep is not None:
                    V *= keep[:, None, sl]
                m = torch.arange(s0, s1, dtype=torch.float64, device="cuda")
                phi = m[:, None] * dt - torch.einsum("mcj,c->mj", r[s0:s1, :, sl], nv)
                J = phi.shape[1]
                jb = max(1, min(J, int(2 ** 25 // max(1, phi.shape[0]))))
                fb = max(1, min(len(w), int(2 ** 26 // (phi.shape[0] * jb))))
                for j0 in range(0, J, jb):
                    ph, Vj = phi[:, j0:j0 + jb], V[:, :, j0:j0 + jb]
                    for f0 in range(0, len(w), fb):
                        th = w[f0:f0 + fb, None, None] * ph
                        cs, sn = torch.cos(th), torch.sin_(th)
                        A = torch.stack([torch.stack([(t * Vj[:, a]).sum(1) for a in range(3)])
                                         for t in (cs, sn)])             # [2][3][f][j]
                        if coherent:
                            tot[:, :, f0:f0 + fb] += A.sum(-1)
                        else:
                            S[row, f0:f0 + fb] += (A * A).sum((0, 1, 3))
                        del th, cs, sn, A
            if coherent:
                S[row] = (tot * tot).sum((0, 1))
        res.append(S / (4.0 * math.pi ** 2))
    return res


def _exact_rad(c, seed):
    q = _exact_dirs(c)
    if q < 1:
        return None
    X, U = _trajectory(_counts(c), c["gamma"], c["samples"] + 1, seed)
    charges = [-1.0, 1.0][: len(_counts(c))]
    S = _exact_spectra(X, U, DT, L_BOX, _dirs(c["dirs"]), _grids(c), _windows(c), _counts(c),
                       charges, c["coherent"], _selectors(c) if c["selectors"] else None, q)
    res = []
    for (_, _, _, _, ds), s in zip(_windows(c), S):
        nd = len(ds) if ds else c["dirs"]
        res.append([s, None] if s.shape[0] < nd else [s])
    return res


# ---------------------------------------------------------------------------
# the live PIC
# ---------------------------------------------------------------------------
PIC_D = 0.1


def _pic_species(c):
    ne = 2 * c["ppc"] * c["n"] ** 2
    w = c["gamma"] * PIC_D * PIC_D / (2 * c["ppc"])     # (n_e / gamma)^(1/2) = 1
    return [(ne, -1.0, 1.0, w), (ne, 1.0, MASS_RATIO, w)]


def _pic_particles(c, seed):
    """Electrons at random positions, each with a partner on top of it; two beams along x."""
    g = _rng(seed)
    ne = 2 * c["ppc"] * c["n"] ** 2
    x = torch.rand((3, ne), generator=g, device="cuda", dtype=torch.float64) * (c["n"] * PIC_D)
    th = 0.01 * torch.randn((2, 3, ne), generator=g, device="cuda", dtype=torch.float64)
    th[1] *= math.sqrt(MASS_RATIO)
    th[:, 0, 0::2] += math.sqrt(c["gamma"] ** 2 - 1.0)
    th[:, 0, 1::2] -= math.sqrt(c["gamma"] ** 2 - 1.0)
    return torch.cat([x, x], 1).contiguous(), torch.cat([th[0], th[1]], 1).contiguous()


def _run_pic(s):
    from paper_1003_1140_gb300.pic import Pic
    c = s["case"]
    with Pic(c["n"], PIC_D, DT, _pic_species(c), s["x"], s["u"]) as p:
        p.step(c["steps"])
        E, B = p.fields()
        x, u = torch.empty_like(s["x"]), torch.empty_like(s["u"])
        p.tracked(0, p.N, x, u)
    return {"E": E, "B": B, "x": x, "u": u}


def _observers():
    th = np.arange(6) * (math.pi / 10)
    return np.stack([np.cos(th), np.zeros(6), np.sin(th)], 1)


def _insitu_windows(c):
    S = c["steps"]
    return [(0, S // 2, 1, 0, None), (S // 2, S, 1, 0, None)]


def _insitu_grid(c):
    return np.exp(np.linspace(math.log(0.1), math.log(1000.0), c["omegas"]))


def _prepare_insitu(c, seed):
    from paper_1003_1140_gb300 import rad as R
    x, u = _pic_particles(c, seed)
    ctx = R.Radiation(_observers(), [_insitu_grid(c)], DT, [(c["tracked"], -1.0, 1.0)],
                      _insitu_windows(c), precision=R.RAD_FP32_SPLIT, box_L=c["n"] * PIC_D)
    return {"case": c, "x": x, "u": u, "ctx": ctx,
            "out": torch.empty(ctx.spectrum_size(), dtype=torch.float64, device="cuda")}


def _run_insitu(s):
    from paper_1003_1140_gb300.pic import Pic
    c, ctx = s["case"], s["ctx"]
    ctx.reset()
    with Pic(c["n"], PIC_D, DT, _pic_species(c), s["x"], s["u"]) as p:
        p.run_coupled(ctx, 0, c["tracked"], c["steps"])
        E, B = p.fields()
        S = ctx.finalize(s["out"])
    return {"E": E, "B": B, "spectra": S.float()}


def _cic(s):
    i = torch.floor(s)
    return i.long(), s - i


def _exact_pic(c, seed, tracked=0):
    """The PIC's scheme (Yee fields, CIC gather, Boris push, Esirkepov current) in FP64."""
    n, d, dt, L = c["n"], PIC_D, DT, c["n"] * PIC_D
    x, u = _pic_particles(c, seed)
    sp = _pic_species(c)
    rep = lambda k: torch.cat([torch.full((s[0],), v, dtype=torch.float64, device="cuda")  # noqa: E731
                               for s, v in zip(sp, k)])
    qm, qw = rep([s[1] / s[2] for s in sp]), rep([s[1] * s[3] for s in sp])
    E = torch.zeros((3, n, n), dtype=torch.float64, device="cuda")
    B = torch.zeros_like(E)
    hist = []

    def interp(F, jf, kf):
        (j, fy), (k, fz) = jf, kf
        j0, j1, k0, k1 = j % n, (j + 1) % n, k % n, (k + 1) % n
        return ((1 - fy) * (1 - fz) * F[j0, k0] + fy * (1 - fz) * F[j1, k0] +
                (1 - fy) * fz * F[j0, k1] + fy * fz * F[j1, k1])

    def curl(F, fwd):                       # forward or backward differences, d/dx = 0
        if fwd:
            dy = lambda a: (torch.roll(a, -1, 0) - a) / d  # noqa: E731
            dz = lambda a: (torch.roll(a, -1, 1) - a) / d  # noqa: E731
        else:
            dy = lambda a: (a - torch.roll(a, 1, 0)) / d  # noqa: E731
            dz = lambda a: (a - torch.roll(a, 1, 1)) / d  # noqa: E731
        return torch.stack([dy(F[2]) - dz(F[1]), dz(F[0]), -dy(F[0])])

    def weights(s, base):
        i, f = _cic(s)
        a = torch.arange(4, device="cuda")[:, None]
        return torch.where(a == i - base, 1 - f, 0.0) + torch.where(a == i - base + 1, f, 0.0)

    for _ in range(c["steps"]):
        if tracked:
            hist.append((x[:, :tracked].clone(), u[:, :tracked].clone()))
        sy, sz = x[1] / d, x[2] / d
        jn, jh, kn, kh = _cic(sy), _cic(sy - 0.5), _cic(sz), _cic(sz - 0.5)
        Ep = torch.stack([interp(E[0], jn, kn), interp(E[1], jh, kn), interp(E[2], jn, kh)])
        Bp = torch.stack([interp(B[0], jh, kh), interp(B[1], jn, kh), interp(B[2], jh, kn)])
        h = 0.5 * qm * dt
        um = u + h * Ep
        t = h / torch.sqrt(1.0 + (um * um).sum(0)) * Bp
        up = um + torch.linalg.cross(um, t, dim=0)
        u = um + torch.linalg.cross(up, 2.0 * t / (1.0 + (t * t).sum(0)), dim=0) + h * Ep
        v = u / torch.sqrt(1.0 + (u * u).sum(0))
        x1 = x + dt * v
        by, bz = torch.floor(sy).long() - 1, torch.floor(sz).long() - 1
        S0y, S1y = weights(sy, by), weights(x1[1] / d, by)
        S0z, S1z = weights(sz, bz), weights(x1[2] / d, bz)
        dy, dz = S1y - S0y, S1z - S0z
        Wx = (S0y[:, None] * S0z[None] + 0.5 * dy[:, None] * S0z[None] +
              0.5 * S0y[:, None] * dz[None] + dy[:, None] * dz[None] / 3.0)
        Wy = torch.cumsum(dy[:, None] * (S0z + S1z)[None] * 0.5, 0)
        Wz = torch.cumsum((S0y + S1y)[:, None] * dz[None] * 0.5, 1)
        at = (((by + torch.arange(4, device="cuda")[:, None]) % n)[:, None] * n +
              ((bz + torch.arange(4, device="cuda")[:, None]) % n)[None]).reshape(-1)
        J = torch.zeros((3, n * n), dtype=torch.float64, device="cuda")
        for a, val in enumerate((qw * v[0] / d ** 2 * Wx, -qw / (d * dt) * Wy, -qw / (d * dt) * Wz)):
            J[a].index_add_(0, at, val.reshape(-1))
        x = torch.where(x1 < 0.0, x1 + L, torch.where(x1 >= L, x1 - L, x1))
        B = B - 0.5 * dt * curl(E, True)
        E = E + dt * (curl(B, False) - J.view(3, n, n))
        B = B - 0.5 * dt * curl(E, True)
    if tracked:
        hist.append((x[:, :tracked].clone(), u[:, :tracked].clone()))
    return E, B, x, u, hist


def _exact_insitu(c, seed):
    E, B, _, _, hist = _exact_pic(c, seed, c["tracked"])
    X, U = torch.stack([h[0] for h in hist]), torch.stack([h[1] for h in hist])
    upd = c["tracked"] * c["steps"] * 6 * c["omegas"]
    if upd > 4e10:
        return {"E": E, "B": B, "spectra": None}
    S = _exact_spectra(X, U, DT, c["n"] * PIC_D, _observers(), [_insitu_grid(c)],
                       _insitu_windows(c), [c["tracked"]], [-1.0], False)
    return {"E": E, "B": B, "spectra": torch.cat([s.reshape(-1) for s in S])}


# ---------------------------------------------------------------------------
# the surrogate network
# ---------------------------------------------------------------------------
FLOOR = 1e-30
LR = 1e-3


def _widths(c):
    return [c["width_in"], c["hidden"], c["hidden"], c["hidden"], c["width_out"]]


def _net_weights(c, seed):
    """He-initialised layers with small biases, the same for both users of a seed."""
    g = _rng(seed)
    w = _widths(c)
    for l in range(len(w) - 1):
        W = torch.randn((w[l + 1], w[l]), generator=g, device="cuda") * math.sqrt(2.0 / w[l])
        yield W, 0.01 * torch.randn(w[l + 1], generator=g, device="cuda")


def _net_data(c, seed):
    """Standardised log spectra: inputs of unit spread, targets a smooth function of them."""
    g = _rng(seed + 1_000_003)
    x = torch.randn((c["batch"], c["width_in"]), generator=g, device="cuda")
    lin = torch.randn((16, c["width_out"]), generator=g, device="cuda") / 4.0
    return x, (torch.tanh(x[:, :16] @ lin) + 0.1 * torch.randn((c["batch"], c["width_out"]),
                                                               generator=g, device="cuda"))


def _net_transform(c, seed):
    r = np.random.default_rng(seed)
    f = lambda lo, hi, n: r.uniform(lo, hi, n).astype(np.float32)  # noqa: E731
    return (f(-4, 0, c["width_in"]), f(0.5, 2, c["width_in"]), f(-4, 0, c["width_out"]),
            f(0.1, 0.5, c["width_out"]))


def _raw_spectra(c, seed):
    x, _ = _net_data(c | {"width_out": 128}, seed)
    mu, sd = (torch.as_tensor(a, device="cuda") for a in _net_transform(c, seed)[:2])
    return torch.pow(10.0, x * sd + mu)


def _prepare_net(c, seed):
    from paper_1003_1140_gb300.mlp import MLP
    w = _widths(c)
    net = MLP(w, c["batch"])
    for l, (W, b) in enumerate(_net_weights(c, seed)):
        net.set_layer(l, W, b)
        del W, b
    s = {"case": c, "net": net}
    if c["kind"] == "train":
        s["x"], s["t"] = _net_data(c, seed)
        s["W"] = [torch.empty((w[l + 1], w[l]), device="cuda") for l in range(len(w) - 1)]
        s["b"] = [torch.empty(w[l + 1], device="cuda") for l in range(len(w) - 1)]
    else:
        net.set_transform(*_net_transform(c, seed), FLOOR)
        s["x"] = _raw_spectra(c, seed)
        s["y"] = torch.empty((c["batch"], w[-1]), device="cuda")
    return s


def _run_train(s):
    net = s["net"]
    losses = [net.train_step(s["x"], s["t"], LR) for _ in range(s["case"]["steps"])]
    for l, (W, b) in enumerate(zip(s["W"], s["b"])):     # rad_mlp_get_layer into device memory
        rc = net._lib.rad_mlp_get_layer(net.h, l, W.data_ptr(), b.data_ptr(), None, None)
        if rc != 0:
            raise RuntimeError("rad_mlp_get_layer failed (%d)" % rc)
    return {"loss": losses, "W": s["W"], "b": s["b"]}


def _run_predict(s):
    return s["net"].predict(s["x"], s["y"])


def _exact_net(c, seed):
    Ws, bs = zip(*[(W.double(), b.double()) for W, b in _net_weights(c, seed)])
    Ws, bs = list(Ws), list(bs)
    L = len(Ws)

    def forward(x):
        h = [x]
        for l in range(L):
            z = h[-1] @ Ws[l].T + bs[l]
            h.append(torch.relu(z) if l < L - 1 else z)
        return h

    if c["kind"] == "predict":
        mu_i, sd_i, mu_o, sd_o = (torch.as_tensor(a, device="cuda").double()
                                  for a in _net_transform(c, seed))
        x = (torch.log10(torch.clamp(_raw_spectra(c, seed).double(), min=FLOOR)) - mu_i) / sd_i
        return torch.pow(10.0, forward(x)[-1] * sd_o + mu_o)
    x, t = (a.double() for a in _net_data(c, seed))
    m = [[torch.zeros_like(a) for a in Ws + bs], [torch.zeros_like(a) for a in Ws + bs]]
    losses = []
    for step in range(1, c["steps"] + 1):
        h = forward(x)
        e = h[-1] - t
        losses.append(float((e * e).mean()))
        g = 2.0 * e / e.numel()
        grads = [None] * (2 * L)
        for l in range(L - 1, -1, -1):
            grads[l], grads[L + l] = g.T @ h[l], g.sum(0)
            if l:
                g = (g @ Ws[l]) * (h[l] > 0)
        del h, e, g
        for i, p in enumerate(Ws + bs):
            m[0][i].mul_(0.9).add_(grads[i], alpha=0.1)
            m[1][i].mul_(0.999).addcmul_(grads[i], grads[i], value=0.001)
            den = torch.sqrt(m[1][i] / (1.0 - 0.999 ** step)).add_(1e-8)
            p.sub_(m[0][i] / (1.0 - 0.9 ** step) / den, alpha=LR)
            del den
        del grads
    return {"loss": losses, "W": Ws, "b": bs}


# ---------------------------------------------------------------------------
# the interface
# ---------------------------------------------------------------------------
def prepare(case, seed):
    k = case["kind"]
    if k == "rad":
        return _prepare_rad(case, seed)
    if k == "pic":
        x, u = _pic_particles(case, seed)
        return {"case": case, "x": x, "u": u}
    if k == "insitu":
        return _prepare_insitu(case, seed)
    return _prepare_net(case, seed)


def run(state):
    return {"rad": _run_rad, "pic": _run_pic, "insitu": _run_insitu, "train": _run_train,
            "predict": _run_predict}[state["case"]["kind"]](state)


def exact(case, seed):
    k = case["kind"]
    if k == "rad":
        return _exact_rad(case, seed)
    if k == "pic":
        E, B, x, u, _ = _exact_pic(case, seed)
        return {"E": E, "B": B, "x": x, "u": u}
    if k == "insitu":
        return _exact_insitu(case, seed)
    return _exact_net(case, seed)


def _pic_work(c):
    """Per particle and step: x and u read and written; gather, push and deposit of about 300
    operations.  Per cell and step: E, B, J read and written."""
    N, nn = 4 * c["ppc"] * c["n"] ** 2, c["n"] ** 2
    return c["steps"] * (96.0 * N + 15 * 8.0 * nn), c["steps"] * 300.0 * N


def work(case):
    """The direct sum takes 8 multiply-adds and one sine/cosine pair per particle, sample,
    direction and frequency: counted as 16 operations."""
    c, k = case, case["kind"]
    if k == "rad":
        states = 48.0 * sum(_counts(c)) * (c["samples"] + 1)
        return {"bytes": states + 8.0 * _out_len(c), "flops": 16.0 * _updates(c)}
    if k == "pic":
        b, f = _pic_work(c)
        return {"bytes": b, "flops": f}
    if k == "insitu":
        b, f = _pic_work(c)
        upd = 6.0 * c["tracked"] * c["steps"] * c["omegas"]
        return {"bytes": b + 48.0 * c["tracked"] * (c["steps"] + 1), "flops": f + 16.0 * upd}
    w, B = _widths(c), c["batch"]
    par = float(sum(w[l] * w[l + 1] for l in range(len(w) - 1)))
    io = 4.0 * B * (w[0] + w[-1])
    if k == "predict":                      # BF16 weights read once, inputs and outputs
        return {"bytes": 2.0 * par + io, "flops": 2.0 * B * par}
    # per step: BF16 weights twice, FP32 weights and both moments read and written, the BF16
    # copy and the stored gradients written
    return {"bytes": c["steps"] * ((2 * 2 + 6 * 4 + 2 + 4) * par + io),
            "flops": c["steps"] * 6.0 * B * par}
