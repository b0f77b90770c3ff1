"""FP64 Gram and update on the tensor cores (tc64.cu) against extended
precision: tile, chunk and share edges, scales, localised and extreme data."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LD = np.longdouble  # 64-bit significand on x86, 113-bit on aarch64


def _reorth(Q, W):
    import torch

    import paper_2210_15763_gb300 as bbl
    q, w = torch.from_numpy(Q).cuda(), torch.from_numpy(W).cuda()
    C = bbl.block_reorth(q, w, passes=1)
    return C.cpu().numpy()[0], w.cpu().numpy()


def _check(Q, W):
    nb, n, b = Q.shape
    C, W1 = _reorth(Q, W)
    F = Q.transpose(1, 0, 2).reshape(n, nb * b)
    # FP64 sums of n products, entrywise bound n 2^-53 |Q|^T |W|; of m products for the update
    exact = F.astype(LD).T @ W.astype(LD)
    bound = (np.abs(F).T @ np.abs(W)) * min(n, 64) * 2.0 ** -53
    # a split entry is exact to 2^-53 of its line's largest entry within a chunk
    line = np.abs(F).max(axis=0)[:, None] * np.abs(W).sum(axis=0) + np.abs(F).sum(axis=0)[:, None] * np.abs(W).max(axis=0)
    assert (np.abs(C - exact) <= bound + line * 2.0 ** -53).all()
    exactW = W.astype(LD) - F.astype(LD) @ C.astype(LD)
    boundW = (np.abs(W) + np.abs(F) @ np.abs(C)) * min(nb * b, 64) * 2.0 ** -53
    lineW = np.abs(F).max(axis=1)[:, None] * np.abs(C).sum(axis=0) + np.abs(F).sum(axis=1)[:, None] * np.abs(C).max(axis=0)
    assert (np.abs(W1 - exactW) <= boundW + lineW * 2.0 ** -53).all()


@pytest.mark.parametrize("b", [2, 4, 8, 16])
@pytest.mark.parametrize("n,m", [(1, 32), (15, 32), (16, 48), (17, 64), (63, 32), (65, 96), (511, 160), (1025, 32),
                                 (700, 528)])
def test_sizes(b, n, m):
    r = np.random.default_rng(7 * n + m + b)
    _check(r.standard_normal((m // b, n, b)), r.standard_normal((n, b)))


@pytest.mark.parametrize("kind", ["growing", "decaying", "rows", "columns", "sparse", "huge", "tiny", "in span"])
def test_data(kind):
    r = np.random.default_rng(3)
    n, b, nb = 1500, 8, 5
    Q, W = r.standard_normal((nb, n, b)), r.standard_normal((n, b))
    i = np.arange(n)[:, None] / 40.0
    if kind == "growing":
        Q, W = Q * np.exp(i - i.max()), W * np.exp(i - i.max())
    elif kind == "decaying":
        Q, W = Q * np.exp(-i), W * np.exp(-i)
    elif kind == "rows":
        Q, W = Q * 10.0 ** r.uniform(-12, 3, (1, n, 1)), W * 10.0 ** r.uniform(-9, 2, (n, 1))
    elif kind == "columns":
        Q, W = Q * 10.0 ** r.uniform(-30, 30, (nb, 1, b)), W * 10.0 ** r.uniform(-30, 30, (1, b))
    elif kind == "sparse":
        Q, W = Q * (r.random(Q.shape) < 0.02), W * (r.random(W.shape) < 0.05)
    elif kind == "huge":
        Q, W = Q * 1e150, W * 1e-120
    elif kind == "tiny":
        Q, W = Q * 1e-120, W * 1e-110
    else:
        W = 3.0 * Q[-1] + 1e-9 * Q[0]
    _check(Q, W)


def test_not_finite():
    r = np.random.default_rng(4)
    Q, W = r.standard_normal((6, 300, 8)), r.standard_normal((300, 8))
    Q[2, 77, 3] = np.inf
    W[5, 6] = np.nan
    C, _ = _reorth(Q, W)
    bad = ~np.isfinite(C)
    want = np.zeros_like(bad)
    want[2 * 8 + 3, :] = True
    want[:, 6] = True
    assert (bad == want).all()
