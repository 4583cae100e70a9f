"""The block-moment accumulation (the default FP32 kernel) and the batched ingest at the
edges of their tilings, against the FP64 oracle.

Tolerance of the spectra: an update's phase error is at most 1.3e-7 |theta| + 5e-7 rad
(special-function unit) plus the FP32 roundings of w, dphi and theta (2^-24 |theta| each);
with w <= 20 and a chunk half-range of 0.775 (1 - n.beta) <= 1.55 that is |theta| <= 31 + pi
and 1.1e-5 rad, so a power is within 2.2e-5 of its scale (the moments' own error, below
1e-6, is far less).
"""
import math

import numpy as np
import pytest

import oracle
import trajgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = 2.2e-5


@pytest.fixture(scope="module")
def traj():
    """17 electrons (gamma 5) and 3 ions, 231 calls, in a small box so that particles cross
    its boundary every few dozen calls."""
    w = trajgen.Workload("edges", [(17, -1.0, 1.0, 5.0), (3, 1.0, 16.0, 3.0)], 231, 0.05,
                         np.array([[0.0, 1.0, 0.0], [1.0, 0, 0], [-0.8, 0.0, 0.6]]), [], [],
                         b_rms=0.4)
    X, U = w.trajectory_numpy()
    return w, X - 3.0 * np.floor(X / 3.0), U


def _close(got, ref, tol):
    for g, e in zip(got, ref):
        for d in range(e.shape[0]):
            scale = np.linalg.norm(e[d])
            assert np.linalg.norm(g[d] - e[d]) <= tol * scale, (d, np.linalg.norm(g[d] - e[d]) / scale)


@pytest.mark.parametrize("nw", [1, 31, 33, 64, 65, 129, 256, 257, 300])
@pytest.mark.parametrize("coherent", [False, True])
def test_frequency_slots_and_orders(traj, nw, coherent):
    """Frequencies around the 32-slot, pair and tile edges: sorted over four decades (moments,
    sub-blocks and direct sums in one tile), shuffled with zero and negative values among
    them, and a second grid that starts in the middle of the frequency arrays."""
    import paper_1003_1140_gb300 as R
    w, X, U = traj
    a = trajgen.log_grid(0.002, 20.0, nw)
    b = np.random.default_rng(nw).permutation(np.concatenate([a, -a, [0.0]]))
    wins = [(0, 230, 3, 0), (13, 77, 1, 1), (96, 97, 3, 1), (31, 33, 2, 0)]
    sp = [(s[0], s[1]) for s in w.species]
    ref = oracle.spectra(X, U, w.dt, w.dirs, [a, b], wins, sp, coherent=coherent, box_L=3.0)
    with R.Radiation(w.dirs, [a, b], w.dt, [s[:3] for s in w.species], wins,
                     mode=R.RAD_COHERENT if coherent else R.RAD_INCOHERENT, box_L=3.0) as r:
        r.accumulate_steps(0, torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda"))
        got = r.finalize()
        assert r.options()["variant"] == R.RAD_VARIANT_AUTO
    _close(got, ref, TOL)


@pytest.mark.parametrize("ndir,nw", [(3, 33), (3, 130), (40, 300), (100, 70), (100, 300)])
@pytest.mark.parametrize("coherent", [False, True])
def test_fp64_tile_widths(traj, ndir, nw, coherent):
    """The FP64 kernel's three tile widths (chosen by the number of units), frequencies from
    moments to direct sums, shuffled and signed: within 1e-10 of the oracle."""
    import paper_1003_1140_gb300 as R
    w, X, U = traj
    rng = np.random.default_rng(ndir + nw)
    dirs = rng.normal(size=(ndir, 3))        # the library normalises, the oracle takes unit vectors
    unit = dirs / np.linalg.norm(dirs, axis=1, keepdims=True)
    a = trajgen.log_grid(0.002, 200.0, nw)
    grids = [a, rng.permutation(a) * rng.choice([-1.0, 1.0], nw)]
    wins = [(0, 230, 3, 0), (13, 77, 1, 1)]
    sp = [(s[0], s[1]) for s in w.species]
    ref = oracle.spectra(X, U, w.dt, unit, grids, wins, sp, coherent=coherent, box_L=3.0)
    with R.Radiation(dirs, grids, w.dt, [s[:3] for s in w.species], wins, precision=R.RAD_FP64,
                     mode=R.RAD_COHERENT if coherent else R.RAD_INCOHERENT, box_L=3.0) as r:
        r.accumulate_steps(0, torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda"))
        got = r.finalize()
    _close(got, ref, 1e-10)


@pytest.mark.parametrize("cuts", [[0, 231], [0, 8, 17, 49, 81, 231], [0, 1, 33, 65, 66, 230, 231],
                                  [0, 32, 64, 128, 200, 231], [0, 7, 20, 31, 47, 160, 231]])
@pytest.mark.parametrize("opts", ["fp64", None, {"variant": 1, "anchor_K": 8}, {"variant": 3}])
def test_batches_of_any_length_give_the_same_ring(traj, cuts, opts):
    """Batches that start and end anywhere in a chunk (one call, under eight, whole chunks)
    and box crossings inside and between them."""
    import paper_1003_1140_gb300 as R
    w, X, U = traj
    grid = trajgen.log_grid(0.05, 20.0, 40)
    wins = [(0, 230, 3, 0), (37, 158, 1, 0)]
    sp = [(s[0], s[1]) for s in w.species]
    ref = oracle.spectra(X, U, w.dt, w.dirs, [grid], wins, sp, box_L=3.0)
    fp64 = opts == "fp64"
    Xd, Ud = torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda")
    with R.Radiation(w.dirs, [grid], w.dt, [s[:3] for s in w.species], wins, box_L=3.0,
                     precision=R.RAD_FP64 if fp64 else R.RAD_FP32_SPLIT,
                     options=None if fp64 else opts) as r:
        for s0, s1 in zip(cuts, cuts[1:]):
            r.accumulate_steps(s0, Xd[s0:s1], Ud[s0:s1])
        got = r.finalize()
    _close(got, ref, 1e-10 if fp64 else TOL)
