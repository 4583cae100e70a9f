"""A position that is not finite (check_inputs off): the particle's unwrapped position is lost
from that call on, however the calls are batched -- a later window must not come out finite
with an image count that missed the crossings meanwhile.  Windows before it, and species
without such a particle, are not touched."""
import numpy as np
import pytest

import oracle
import trajgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {0: 1e-10, 1: 2.2e-5}          # as in test_gpu_moments.py


@pytest.fixture(scope="module")
def traj():
    w = trajgen.Workload("edges", [(17, -1.0, 1.0, 5.0), (3, 1.0, 16.0, 3.0)], 231, 0.05,
                         np.array([[0.0, 1.0, 0.0], [-0.8, 0.0, 0.6]]), [], [], b_rms=0.4)
    X, U = w.trajectory_numpy()
    X = X - 3.0 * np.floor(X / 3.0)
    grid = trajgen.log_grid(0.05, 20.0, 40)
    wins = [(0, 49, 3, 0), (90, 200, 1, 0), (90, 200, 2, 0), (201, 230, 1, 0)]
    refs = {n: oracle.spectra(X, U, w.dt, w.dirs, [grid], wins, [(s[0], s[1]) for s in w.species],
                              box_L=3.0, **({"subcycle": n} if n > 1 else {})) for n in (1, 3)}
    return w, X, U, grid, wins, refs


@pytest.mark.parametrize("cuts", [[0, 231], list(range(232)), [0, 8, 17, 53, 81, 231],
                                  [0, 60, 61, 130, 231], [0, 7, 50, 51, 57, 231]])
@pytest.mark.parametrize("opts", ["fp64", None, {"variant": 1, "anchor_K": 8}, {"subcycle": 3}])
@pytest.mark.parametrize("value", [np.nan, -np.inf, 1e300])
def test_lost_positions_stay_lost(traj, cuts, opts, value):
    import paper_1003_1140_gb300 as R
    w, X, U, grid, wins, refs = traj
    X = X.copy()
    X[52, 1, 4] = value
    precision = 0 if opts == "fp64" else 1
    Xd, Ud = torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda")
    with R.Radiation(w.dirs, [grid], w.dt, [s[:3] for s in w.species], wins, box_L=3.0,
                     precision=precision, options=opts if precision else None) as r:
        for s0, s1 in zip(cuts, cuts[1:]):
            r.accumulate_steps(s0, Xd[s0:s1], Ud[s0:s1])
        got = r.finalize()
    ref = refs[3 if opts == {"subcycle": 3} else 1]
    for k in (0, 2):
        for d in range(2):
            assert np.linalg.norm(got[k][d] - ref[k][d]) <= TOL[precision] * np.linalg.norm(ref[k][d])
    for k in (1, 3):
        assert np.isnan(got[k]).all()
