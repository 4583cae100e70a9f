"""PIC steps captured in a CUDA graph: replays go on from the state that the last step left,
whether that was a replay, a direct step or fields set from outside."""
import numpy as np
import pytest

import trajgen

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("per_graph", [1, 2])
def test_captured_steps_replay(per_graph):
    """Bounds as in test_gpu_pic_moves.py: two runs differ by the order of the current's sums."""
    from paper_1003_1140_gb300 import pic
    ts = trajgen.TwoStream(n=16, ppc=2, gamma=3.0, u_th=0.3, seed=31)
    st = torch.cuda.Stream()
    rng = np.random.default_rng(5)
    E0, B0 = 0.01 * rng.normal(size=(2, 3, ts.n, ts.n))
    with pic.Pic.two_stream(ts, stream=st) as a, pic.Pic.two_stream(ts) as b:
        a.set_fields(E0, B0)
        b.set_fields(E0, B0)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            a.step(per_graph)
        done = 0

        def replay(k):
            nonlocal done
            with torch.cuda.stream(st):
                for _ in range(k):
                    g.replay()
            done += k * per_graph

        replay(3)
        st.synchronize()
        a.step(1)
        replay(2)
        b.step(done + 1)
        a.set_fields(B=1.5 * B0)
        b.set_fields(B=1.5 * B0)
        replay(1)
        a.step(2)
        b.step(per_graph + 2)
        Ea, Ba = a.fields()
        Eb, Bb = b.fields()
        xa, ua = a.particles()
        xb, ub = b.particles()
    d = xa - xb
    d -= ts.L * np.round(d / ts.L)
    assert np.abs(d).max() <= 1e-10 * ts.L
    assert np.abs(ua - ub).max() <= 1e-10 * np.abs(ub).max()
    assert np.abs(Ea - Eb).max() <= 1e-9 * np.abs(Eb).max()
    assert np.abs(Ba - Bb).max() <= 1e-9 * np.abs(Bb).max()
