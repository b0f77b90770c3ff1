"""MLP calls at batches beyond 16 x 65535 samples (one grid dimension's limit)."""
import numpy as np
import pytest

from oracle import mlp as OM
from tests.gpu_util import need_gpu, to_dev
from tests.test_gpu_learned import _setup, pack, unpack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1048560, 1048561, 1100003])
def test_large_batch(batch):
    torch, bbl = need_gpu()
    H, O = 4, 3
    p, g, tgt = _setup(H, O, 64, seed=7)
    reps, rest = batch // 64, batch % 64
    G, T = np.concatenate([np.tile(g, reps), g[:rest]]), np.concatenate([np.tile(tgt, (reps, 1)), tgt[:rest]])
    net = bbl.MLP(H, O)
    net.set_params(pack(p))
    y = net.forward(to_dev(torch, G, torch.float32)).cpu().numpy()
    small = net.forward(to_dev(torch, g, torch.float32)).cpu().numpy()
    assert (y == np.concatenate([np.tile(small, (reps, 1)), small[:rest]])).all()
    loss = net.loss_grad(to_dev(torch, G, torch.float32), to_dev(torch, T, torch.float32))
    # means over the repeated samples
    yr, c = OM.forward(p, g)
    w = np.full(64, reps / batch) + (np.arange(64) < rest) / batch
    d = yr - tgt
    assert loss == pytest.approx(float((w[:, None] * d * d).sum() / O), rel=1e-4)
    got = unpack(net.get_params()[1], H, O)
    dy = 2.0 * w[:, None] * d / O
    # FP32 sums of `batch` products in turn: batch 2^-25 of the sum of the magnitudes
    # where all roundings of the repeated terms agree
    tol = batch * 2.0 ** -25 + 1e-3
    assert (np.abs(got["W3"] - dy.T @ c["h2"]) <= tol * (np.abs(dy).T @ np.abs(c["h2"]))).all()
    assert (np.abs(got["b3"] - dy.sum(axis=0)) <= tol * np.abs(dy).sum(axis=0)).all()


@pytest.mark.parametrize("H,O,batch", [(4, 32, 64), (8, 3, 40), (16, 300, 5)])
def test_loss_of_large_differences(H, O, batch):
    """The mean is finite although the sum of the squares is not (FP32)."""
    torch, bbl = need_gpu()
    p, g, _ = _setup(H, O, batch, seed=2)
    r = np.random.default_rng(1)
    tgt = (r.uniform(0.8, 1.0, (batch, O)) * 1.2e18).astype(np.float32)
    net = bbl.MLP(H, O)
    net.set_params(pack(p))
    loss = net.loss_grad(to_dev(torch, g, torch.float32), torch.from_numpy(tgt).cuda())
    # squares, scaling and a sum of at most 1500 terms by trees: 2^-24 each
    assert loss == pytest.approx(float((tgt.astype(np.float64) ** 2).mean()), rel=20 * 2.0 ** -24)


def test_a_batch_beyond_the_memory_leaves_the_network_usable():
    torch, bbl = need_gpu()
    p, g, tgt = _setup(1024, 8, 6, seed=3)
    net = bbl.MLP(1024, 8)
    net.set_params(pack(p))
    x, t = to_dev(torch, g, torch.float32), to_dev(torch, tgt, torch.float32)
    want = net.forward(x).cpu().numpy()
    net.train(x, t, 1, 1e-12)
    with pytest.raises(bbl.BBLError, match="OOM"):  # 40 TB of activations; refused before x is read
        bbl._lib.check(bbl._lib.load().bbl_mlp_forward(net.handle, 1600000000, x.data_ptr(), x.data_ptr(), None))
    np.testing.assert_allclose(net.forward(x).cpu().numpy(), want, atol=1e-5)
    net.train(x, t, 1, 1e-12)


@pytest.mark.parametrize("H,O", [(1, 1), (5, 7), (16, 48), (31, 2), (31, 3), (4, 252), (4, 253)])
def test_small_networks_forward(H, O):
    """Either side of the one-kernel forward: a batch in one call and in two large enough
    for the general kernels gives the same bits, and the oracle's values."""
    torch, bbl = need_gpu()
    p, g, _ = _setup(H, O, 400, seed=H + O)
    net = bbl.MLP(H, O)
    net.set_params(pack(p))
    few = net.forward(to_dev(torch, g, torch.float32)).cpu().numpy()
    many = net.forward(to_dev(torch, np.tile(g, 2), torch.float32)).cpu().numpy()
    assert (many == np.tile(few, (2, 1))).all()
    ref = OM.forward(p, g)[0]
    # FP32 sums of at most 31 products, twice, and the FP32 error function
    assert np.abs(few - ref).max() <= 1e-5 * (np.abs(ref).max() + 1.0)
