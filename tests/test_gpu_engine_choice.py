"""Which FP32 engine the options select, and that the report selects it again."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
AUTO, SFU, MIX, PRECISE = 0, 1, 2, 3


def _run(options, w_max=50.0):
    import paper_1003_1140_gb300 as R
    rng = np.random.default_rng(1)
    U = np.ascontiguousarray(np.broadcast_to(rng.normal(size=(3, 9)), (40, 3, 9)))
    U = U + 0.01 * rng.normal(size=U.shape)
    X = np.cumsum(0.05 * U / np.sqrt(1.0 + (U * U).sum(1, keepdims=True)), axis=0)
    with R.Radiation([[0.0, 0.0, 1.0]], [np.linspace(1.0, w_max, 70)], 0.05, [(9, -1.0, 1.0)],
                     [(0, 39, 1, 0)], options=options) as r:
        r.accumulate_steps(0, torch.as_tensor(X, device="cuda"), torch.as_tensor(U, device="cuda"))
        return r.finalize()[0], r.options()


@pytest.mark.parametrize("options,variant,K,ft,mb", [
    ({}, AUTO, 32, 8, 4), ({"anchor_K": 32}, AUTO, 32, 8, 4),
    ({"blocks_per_sm": 2}, SFU, 32, 8, 2), ({"blocks_per_sm": 3}, SFU, 32, 8, 3),
    ({"freq_per_lane": 8}, SFU, 32, 8, 2), ({"freq_per_lane": 16}, SFU, 32, 16, 2),
    ({"freq_per_lane": 8, "blocks_per_sm": 2}, SFU, 32, 8, 2),
    ({"anchor_K": 16}, SFU, 16, 8, 2), ({"phase_budget": 1e-4}, SFU, 32, 8, 2),
    ({"variant": SFU}, SFU, 32, 8, 2), ({"variant": MIX}, MIX, 32, 8, 2),
    ({"variant": PRECISE}, PRECISE, 32, 8, 2)])
def test_engine_and_report(options, variant, K, ft, mb):
    spec, o = _run(options)
    assert (o["variant"], o["anchor_K"], o["freq_per_lane"], o["blocks_per_sm"]) == (variant, K, ft, mb)
    keys = ("variant", "anchor_K", "freq_per_lane", "blocks_per_sm", "poly_per_lane", "phase_budget")
    again, o2 = _run({k: o[k] for k in keys})
    assert o2 == o
    np.testing.assert_array_equal(again, spec)


def test_limit_of_the_automatic_choice():
    """w dt just inside and outside the 32-sample anchors' default phase budget."""
    lim = 1e-4 * 2.0 ** 24 / 31 / 0.05
    assert _run({}, 0.999 * lim)[1]["variant"] == AUTO
    assert _run({}, 1.001 * lim)[1]["variant"] == SFU


@pytest.mark.parametrize("options", [{"blocks_per_sm": 4}, {"freq_per_lane": 8, "blocks_per_sm": 4},
                                     {"variant": SFU, "freq_per_lane": 8, "blocks_per_sm": 4},
                                     {"freq_per_lane": 4}])
def test_builds_that_do_not_exist_are_refused(options):
    import paper_1003_1140_gb300 as R
    with pytest.raises(R.RadError) as e:
        _run(options)
    assert e.value.code == -1
