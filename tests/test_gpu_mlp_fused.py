"""The output layer's fused epilogues (loss gradient, output transform, direct stores) and
products that read an operand stored K-last in place."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _net(widths, max_batch, seed=11):
    from paper_1003_1140_gb300 import mlp
    rng = np.random.default_rng(seed)
    L = len(widths) - 1
    Ws = [(rng.normal(size=(widths[l + 1], widths[l])) / np.sqrt(widths[l])).astype(np.float32)
          for l in range(L)]
    bs = [(rng.normal(size=widths[l + 1]) * 0.1).astype(np.float32) for l in range(L)]
    net = mlp.MLP(widths, max_batch)
    for l in range(L):
        net.set_layer(l, Ws[l], bs[l])
    return net, Ws, bs, rng


@pytest.mark.parametrize("widths,batch", [
    ([128, 2048, 128], 150),       # one output column tile: the loss epilogue of a split product
    ([128, 2048, 128], 256),
    ([128, 128, 20096], 33),       # 157 column tiles: more than one per block
    ([128, 640], 1),               # a single row
    ([128, 155776], 200),          # 1217 column tiles: both row tiles in one block, sums chained
])
def test_loss_epilogue(widths, batch):
    """Loss and gradients against the reference; tolerances as for every other width
    (BF16 roundings that fall on the other side in FP32 than in FP64)."""
    net, Ws, bs, rng = _net(widths, 256)
    x = rng.normal(size=(batch, widths[0])).astype(np.float32)
    t = rng.normal(size=(batch, widths[-1])).astype(np.float32)
    lr, dWr, dbr = ref.gradients([w.astype(np.float64) for w in Ws], bs, x, t)
    td = torch.zeros(t.size + 1, device="cuda")
    for tt in (torch.as_tensor(t, device="cuda"), td[1:].view(t.shape).copy_(torch.as_tensor(t)), t):
        loss = net.gradients(torch.as_tensor(x, device="cuda"), tt)
        assert abs(loss - lr) <= 1e-3 * lr
        for l in range(len(Ws)):
            _, _, dW, db = net.get_layer(l, grads=True)
            assert np.linalg.norm(dW - dWr[l]) <= 2e-3 * np.linalg.norm(dWr[l]), l
            assert np.linalg.norm(db - dbr[l]) <= 2e-3 * np.linalg.norm(dbr[l]), l
    net.close()


@pytest.mark.parametrize("widths", [[128, 256, 384], [128, 2048, 128], [128, 155776]])
@pytest.mark.parametrize("batch", [1, 100, 128, 131])
def test_outputs_in_place_and_staged_agree(widths, batch):
    """forward and predict write the same bits to aligned device memory (directly), to
    misaligned device memory and to host memory, and nothing past the batch's rows."""
    net, _, _, rng = _net(widths, 256)
    wi, wo = widths[0], widths[-1]
    net.set_transform(np.zeros(wi), np.ones(wi), rng.normal(size=wo), rng.uniform(0.1, 0.5, wo), 1e-30)
    x = torch.as_tensor((10.0 ** rng.uniform(-2, 2, size=(batch, wi))).astype(np.float32), device="cuda")
    for call in (net.forward, net.predict):
        host = call(x)
        for off in (0, 1):
            buf = torch.full((off + 300 * wo,), -7.0, device="cuda")
            call(x, buf[off:off + batch * wo].view(batch, wo))
            got = buf.cpu().numpy()
            np.testing.assert_array_equal(got[off:off + batch * wo].reshape(batch, wo), host)
            assert np.all(got[:off] == -7.0) and np.all(got[off + batch * wo:] == -7.0)
    net.close()


@pytest.mark.parametrize("ak,bk", [(True, False), (False, True), (False, False)])
@pytest.mark.parametrize("M,N,K", [(128, 128, 64), (384, 256, 64 * 37), (2560, 1280, 128)])
def test_gemm_k_last_operands(ak, bk, M, N, K):
    """Small integers: every product and sum is exact, so the result is; at 16-byte and at
    2-byte alignment."""
    from paper_1003_1140_gb300 import mlp
    rng = np.random.default_rng(M + K)
    A = rng.integers(-4, 5, size=(M, K)).astype(np.float32)
    B = rng.integers(-4, 5, size=(N, K)).astype(np.float32)
    exp = A @ B.T

    def dev(a, off):
        buf = torch.zeros(a.size + off, dtype=torch.bfloat16, device="cuda")
        buf[off:] = torch.as_tensor(np.ascontiguousarray(a).ravel(), device="cuda").to(torch.bfloat16)
        return buf[off:]

    for off in (0, 1):
        Ad = dev(A, 0) if ak else dev(A.T, off)
        Bd = dev(B, 0) if bk else dev(B.T, off)
        C = torch.empty((M, N), dtype=torch.float32, device="cuda")
        mlp.gemm(Ad, Bd, M, N, K, ak, bk, C)
        mlp.check()
        np.testing.assert_array_equal(C.cpu().numpy(), exp)


@pytest.mark.parametrize("widths,batch", [
    ([128, 256, 640], 130),        # parameter counts that do and do not fill the last block
    ([128, 19584], 5),
])
def test_train_step_is_gradients_then_adam(widths, batch):
    """Bit for bit, gradients included, over two steps."""
    nets = [_net(widths, 256)[0] for _ in range(2)]
    rng = np.random.default_rng(4)
    for step in range(2):
        x = rng.normal(size=(batch, widths[0])).astype(np.float32)
        t = rng.normal(size=(batch, widths[-1])).astype(np.float32)
        la = nets[0].gradients(x, t)
        nets[0].adam(2e-3)
        assert nets[1].train_step(x, t, 2e-3) == la
        for l in range(len(widths) - 1):
            for a, b in zip(nets[0].get_layer(l, grads=True), nets[1].get_layer(l, grads=True)):
                np.testing.assert_array_equal(a, b, err_msg=f"step {step} layer {l}")
    for net in nets:
        net.close()
