"""The PIC's particle kernel where particles change cells all the time and wrap, and the
coupled run on one and on two streams."""
import numpy as np
import pytest

import trajgen
from oracle import pic as ref

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("axis,n", [(1, 4), (1, 16), (2, 17)])
def test_in_plane_streaming_matches_reference(axis, n):
    """Streaming in the simulation plane (about 0.47 cells per step, both ways) with a
    thermal spread across it: every particle crosses nodes and the boundary in both axes
    within 20 steps.  Same bounds as the out-of-plane comparison: the two sides differ by
    FP64 rounding and the order of the current's sums."""
    from paper_1003_1140_gb300 import pic
    ts = trajgen.TwoStream(n=n, ppc=2, gamma=3.0, u_th=0.5, axis=axis, seed=27)
    X, U, q, m, w = ts.particles()
    g = ref.Grid(ts.n, ts.d, ts.dt)
    E = np.zeros((3, n, n))
    B = np.zeros((3, n, n))
    with pic.Pic.two_stream(ts) as p:
        for _ in range(20):
            X, U, E, B, _ = ref.step(X, U, E, B, q, m, w, g)
        p.step(20)
        Eg, Bg = p.fields()
        xg, ug = p.particles()
    d = xg - X
    d -= ts.L * np.round(d / ts.L)
    assert np.abs(d).max() <= 1e-10 * ts.L
    assert np.abs(ug - U).max() <= 1e-10 * np.abs(U).max()
    assert np.abs(Eg - E).max() <= 1e-9 * np.abs(E).max()
    assert np.abs(Bg - B).max() <= 1e-9 * np.abs(B).max()
    rho = ref.charge_density(xg[1], xg[2], q * w, g)
    rho0 = np.abs(q * w).sum() / ts.L ** 2
    assert np.abs(ref.div_E(Eg, g.d) - rho).max() <= 1e-10 * rho0


@pytest.mark.parametrize("graph", [0, 1])
def test_coupled_run_on_one_and_two_streams(graph):
    """The tracked particles are read in place on one stream and through the staging
    buffers on two; a range in the middle of the particle arrays."""
    from paper_1003_1140_gb300 import pic
    from paper_1003_1140_gb300 import rad as R
    ts = trajgen.TwoStream(n=16, ppc=2, gamma=3.0, u_th=0.05, seed=28)
    grid = trajgen.log_grid(0.1, 50.0, 70)
    got = []
    for st in (None, torch.cuda.Stream()):
        with pic.Pic.two_stream(ts) as p, \
                R.Radiation(trajgen.paper_observers(), [grid], ts.dt, [(61, -1.0, 1.0)],
                            [(0, 40, 1, 0), (11, 33, 1, 0)], box_L=ts.L, stream=st,
                            options={"use_graph": graph}) as r:
            p.run_coupled(r, 37, 61, 40)
            got.append(r.finalize())
    for a, b in zip(*got):
        # the PIC's current sums (and so its particles) repeat to the last bits only
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)
        assert np.linalg.norm(b) > 0
