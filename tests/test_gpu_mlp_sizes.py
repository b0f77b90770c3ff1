"""MLP gradients at layer widths around the tiles of the backward kernel (four
columns per lane where the width is a multiple of four, else one), against the
FP64 oracle; tolerance as in test_gpu_learned (FP32 sums of at most 1024 terms)."""
import numpy as np
import pytest

from oracle import mlp as OM
from tests.gpu_util import need_gpu, to_dev
from tests.test_gpu_learned import PN, _setup, pack, unpack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,O,batch", [(1, 1, 1), (3, 5, 2), (4, 4096, 3), (33, 31, 5), (124, 40, 4), (128, 1, 9), (132, 70, 6),
                                       (257, 33, 3), (516, 9, 2), (1023, 12, 1), (1024, 64, 5)])
def test_gradients_match_the_oracle(H, O, batch):
    torch, bbl = need_gpu()
    p, g, tgt = _setup(H, O, batch, seed=H + O)
    net = bbl.MLP(H, O)
    net.set_params(pack(p))
    loss = net.loss_grad(to_dev(torch, g, torch.float32), to_dev(torch, tgt, torch.float32))
    loss_ref, ref = OM.loss_and_grads(p, g, tgt, bf16_weights=True)
    assert loss == pytest.approx(loss_ref, rel=1e-4)
    got = unpack(net.get_params()[1], H, O)
    for k in PN:
        np.testing.assert_allclose(got[k], ref[k], rtol=0, atol=1e-3 * (np.abs(ref[k]).max() + 1e-30), err_msg=k)
