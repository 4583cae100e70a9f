"""The FP64 path in other units of length and time: a power of two times all positions, steps
and the box, frequencies divided by it, is the same problem (V dt has no unit), also where the
lengths are outside the FP32 range."""
import numpy as np
import pytest

import oracle
import trajgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("exponent", [-140, -20, 20, 140])
@pytest.mark.parametrize("batch", [231, 40, 1])
def test_scaled_units(exponent, batch):
    """Within the FP64 path's 1e-10 of the oracle in the original units."""
    import paper_1003_1140_gb300 as R
    w = trajgen.Workload("edges", [(17, -1.0, 1.0, 5.0), (3, 1.0, 16.0, 3.0)], 231, 0.05,
                         np.array([[0.0, 1.0, 0.0], [-0.8, 0.0, 0.6]]), [], [], b_rms=0.4)
    X, U = w.trajectory_numpy()
    X = X - 3.0 * np.floor(X / 3.0)
    grid = trajgen.log_grid(0.05, 20.0, 40)
    wins = [(0, 230, 3, 0)]
    ref = oracle.spectra(X, U, w.dt, w.dirs, [grid], wins, [(s[0], s[1]) for s in w.species],
                         box_L=3.0)[0]
    f = np.ldexp(1.0, exponent)
    Xd, Ud = torch.as_tensor(X * f, device="cuda"), torch.as_tensor(U, device="cuda")
    with R.Radiation(w.dirs, [grid / f], w.dt * f, [s[:3] for s in w.species], wins, box_L=3.0 * f,
                     precision=R.RAD_FP64) as r:
        for s in range(0, 231, batch):
            r.accumulate_steps(s, Xd[s:s + batch], Ud[s:s + batch])
        got = r.finalize()[0]
    for d in range(2):
        assert np.linalg.norm(got[d] - ref[d]) <= 1e-10 * np.linalg.norm(ref[d])
