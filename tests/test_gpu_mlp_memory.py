"""Device memory of a network: its parameters, optimiser state, activations and the scratch of
the products that split, not of those that never do."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("widths,batch", [([768, 512, 393216], 256), ([128, 65536], 512)])
def test_scratch_only_for_split_products(widths, batch):
    """Beyond what the layers hold, at most 64 MiB (allocation granularity, and split products
    of 256 rows x 512 columns in at most 76 slices: 40 MB)."""
    from paper_1003_1140_gb300.mlp import MLP
    MLP([128, 128], 128)                          # the library and its context are up
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net = MLP(widths, batch)
    used = before - torch.cuda.mem_get_info()[0]
    layers = list(zip(widths, widths[1:]))
    held = sum(18 * i * o + 16 * o for i, o in layers)           # W, m, v, dW, BF16 W; b likewise
    held += batch * sum(2 * w for w in widths) + batch * sum(6 * w for w in widths[1:])
    held += 4 * batch * (widths[-1] + widths[0])                 # targets, input staging
    assert held <= used <= held + (64 << 20), (used, held)
    del net
