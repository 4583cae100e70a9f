"""The FP32 ring's two chunk layouts: chunks that single calls and short batches fill are
slot-major until a window closes, those of long batches (and of host blocks) particle-major.
Every change between them, in the middle of a chunk and at its edges, against the oracle.

Tolerances as in test_gpu_moments.py (frequencies up to 20, dt 0.05).
"""
import numpy as np
import pytest

import oracle
import trajgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {0: 1e-10, 1: 2.2e-5}


def _traj(n, calls, ions=0):
    species = [(n, -1.0, 1.0, 5.0)] + ([(ions, 1.0, 16.0, 3.0)] if ions else [])
    w = trajgen.Workload("layout", species, calls, 0.05,
                         np.array([[0.0, 1.0, 0.0], [-0.8, 0.0, 0.6]]), [], [], b_rms=0.4)
    X, U = w.trajectory_numpy()
    return w, X - 3.0 * np.floor(X / 3.0), U


def _close(got, ref, tol, factor=1.0):
    for g, e in zip(got, ref):
        for d in range(e.shape[0]):
            assert np.linalg.norm(g[d] - factor * e[d]) <= tol * factor * np.linalg.norm(e[d])


# (number of calls, 'h' from host memory / 'd' from device memory), repeated
MIXES = {
    "singles": [(1, "d")],
    "short": [(3, "d"), (1, "d"), (7, "d")],
    "singles and batches": [(1, "d")] * 5 + [(9, "d")] + [(1, "d")] * 40 + [(40, "d"), (3, "d")],
    "edges": [(33, "d")] + [(1, "d")] * 31 + [(32, "d")] + [(1, "d")] * 33,
    "host blocks": [(1, "d")] * 20 + [(70, "h")] + [(1, "d")] * 10 + [(64, "h"), (20, "d")],
}
WINS = [(0, 230, 3, 0), (5, 37, 1, 0), (31, 64, 1, 0), (32, 96, 3, 0), (70, 71, 1, 0),
        (90, 161, 2, 0), (100, 229, 1, 0)]


@pytest.fixture(scope="module")
def mixed():
    w, X, U = _traj(2050, 231, ions=30)
    grid = trajgen.log_grid(0.05, 20.0, 12)
    sp = [(s[0], s[1]) for s in w.species]
    refs = {n: oracle.spectra(X, U, w.dt, w.dirs, [grid], WINS, sp, box_L=3.0,
                              **({"subcycle": n} if n > 1 else {})) for n in (1, 3)}
    return w, X, U, grid, refs


@pytest.mark.parametrize("mix", sorted(MIXES))
@pytest.mark.parametrize("opts", [{}, {"use_graph": 1}, {"subcycle": 3, "use_graph": 1}, {"variant": 3},
                                  {"variant": 1, "anchor_K": 8, "use_graph": 1}, {"defer": 1}])
def test_layouts_in_every_order(mixed, mix, opts):
    import paper_1003_1140_gb300 as R
    w, X, U, grid, refs = mixed
    Xd, Ud = torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda")
    ref = refs[opts.get("subcycle", 1)]

    def hand_over(r, steps):
        s = k = 0
        while s < len(X):
            n, where = steps[k % len(steps)]
            n, k = min(n, len(X) - s), k + 1
            a, b = (X, U) if where == "h" else (Xd, Ud)
            if n == 1:
                r.accumulate(s, a[s], b[s])
            else:
                r.accumulate_steps(s, a[s:s + n], b[s:s + n])
            s += n

    with R.Radiation(w.dirs, [grid], w.dt, [s[:3] for s in w.species], WINS, box_L=3.0,
                     options=opts or None) as r:
        hand_over(r, MIXES[mix])
        _close(r.finalize(), ref, TOL[1])
        r.next_shard()                            # the same particles once more
        hand_over(r, [(50, "d"), (1, "d")])
        _close(r.finalize(), ref, TOL[1], 2.0)
        r.reset()
        hand_over(r, MIXES[mix][::-1])
        _close(r.finalize(), ref, TOL[1])


@pytest.mark.parametrize("n,batch", [(33000, 70), (33000, 9), (9000, 16), (9000, 30)])
@pytest.mark.parametrize("precision", [0, 1])
def test_batches_of_large_populations(n, batch, precision):
    """Both sides of the rule that chooses the ingest kernel."""
    import paper_1003_1140_gb300 as R
    w, X, U = _traj(n, 70)
    grid = trajgen.log_grid(0.5, 20.0, 5)
    wins = [(0, 69, 1, 0), (20, 41, 1, 0)]
    ref = oracle.spectra(X, U, w.dt, w.dirs, [grid], wins, [(n, -1.0)], box_L=3.0)
    Xd, Ud = torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda")
    with R.Radiation(w.dirs, [grid], w.dt, [(n, -1.0, 1.0)], wins, box_L=3.0,
                     precision=precision) as r:
        for s in range(0, 70, batch):
            r.accumulate_steps(s, Xd[s:s + batch], Ud[s:s + batch])
        _close(r.finalize(), ref, TOL[precision])
