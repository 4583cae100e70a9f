"""Windows that start late or end early: the ring is as long as the windows' span, and calls
outside it are handed over too.  Samples that no window needs must not reach the ring, where
they would share slots with samples that one does.

Tolerances as in test_gpu_moments.py (frequencies up to 20, dt 0.05).
"""
import numpy as np
import pytest

import oracle
import trajgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
TOL = {0: 1e-10, 1: 2.2e-5}


@pytest.fixture(scope="module")
def late():
    """17 electrons and 3 ions, 1301 calls, crossing a small box all the time."""
    w = trajgen.Workload("late", [(17, -1.0, 1.0, 5.0), (3, 1.0, 16.0, 3.0)], 1301, 0.05,
                         np.array([[0.0, 1.0, 0.0], [1.0, 0, 0], [-0.8, 0.0, 0.6]]), [], [],
                         b_rms=0.4)
    X, U = w.trajectory_numpy()
    return w, X - 3.0 * np.floor(X / 3.0), U


@pytest.mark.parametrize("opts", [{}, {"subcycle": 3}, {"variant": 1, "anchor_K": 8}, {"variant": 3},
                                  {"defer": 1}])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("wins,batch", [([(1000, 1100, 3, 0)], 1301), ([(1000, 1100, 3, 0)], 7),
                                        ([(1015, 1047, 1, 0), (1040, 1063, 3, 0)], 400),
                                        ([(640, 641, 3, 0)], 1301)])
def test_calls_before_and_after_the_windows(late, opts, precision, wins, batch):
    import paper_1003_1140_gb300 as R
    if precision == 0 and "variant" in opts:
        pytest.skip("an FP32 option")
    w, X, U = late
    grid = trajgen.log_grid(0.05, 20.0, 40)
    sp = [(s[0], s[1]) for s in w.species]
    ref = oracle.spectra(X, U, w.dt, w.dirs, [grid], wins, sp, box_L=3.0,
                         **({"subcycle": 3} if "subcycle" in opts else {}))
    Xd, Ud = torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda")
    with R.Radiation(w.dirs, [grid], w.dt, [s[:3] for s in w.species], wins, box_L=3.0,
                     precision=precision, options=opts or None) as r:
        for s in range(0, len(X), batch):
            r.accumulate_steps(s, Xd[s:s + batch], Ud[s:s + batch])
        got = r.finalize()
    for g, e in zip(got, ref):
        for d in range(e.shape[0]):
            assert np.linalg.norm(g[d] - e[d]) <= TOL[precision] * np.linalg.norm(e[d])
