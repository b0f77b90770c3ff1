"""FP64 Gram, update and Ritz vectors hold the bound of FP64 sums entry by entry,
whatever the range of the data: a sum that the digits do not certify is formed
again in FP64 (tc64.cu).  Also the paths that only many rows reach: several chunks
per CTA, several row groups per CTA, more coefficients than are staged at once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LD = np.longdouble  # 64-bit significand on x86, 113-bit on aarch64
U = 2.0 ** -53


def _flat(Q):
    nb, n, b = Q.shape
    return Q.transpose(1, 0, 2).reshape(n, nb * b)


def _check(Q, W, cols=None, rows=None):
    """Sums of FP64 products in any order err by at most (terms) 2^-53 sum |q||w|; 64 stands for all longer sums."""
    import torch

    import paper_2210_15763_gb300 as bbl
    q, w = torch.from_numpy(Q).cuda(), torch.from_numpy(W).cuda()
    n, m = Q.shape[1], Q.shape[0] * Q.shape[2]
    C = bbl.block_reorth(q, w, passes=1).cpu().numpy()[0]
    W1 = w.cpu().numpy()
    X = bbl.ritz_vectors(q, torch.from_numpy(C).cuda()).cpu().numpy()
    F = _flat(Q)
    cols = np.arange(m) if cols is None else cols
    rows = np.arange(n) if rows is None else rows
    tiny = n * 5e-324
    with np.errstate(all="ignore"):
        exact = F[:, cols].astype(LD).T @ W.astype(LD)
        mag = np.abs(F[:, cols]).T @ np.abs(W)
        assert (np.abs(C[cols] - exact) <= mag * min(n, 64) * U + tiny).all()
        exact = F[rows].astype(LD) @ C.astype(LD)
        mag = np.abs(F[rows]) @ np.abs(C)
        assert (np.abs(X[rows] - exact) <= mag * min(m, 64) * U + tiny).all()
        assert (np.abs(W1[rows] - (W[rows].astype(LD) - exact)) <= (mag + np.abs(W[rows])) * min(m, 64) * U + tiny).all()


@pytest.mark.parametrize("b", [2, 4, 8, 16])
@pytest.mark.parametrize("kind", ["outlier", "one tiny row", "small where it counts", "steps", "tiny", "huge", "denormal",
                                  "spikes", "zero blocks"])
def test_range(b, kind):
    r = np.random.default_rng(11 + b)
    n, m = 900, 64
    Q, W = r.standard_normal((m // b, n, b)), r.standard_normal((n, b))
    if kind == "outlier":  # a large entry opposite a zero
        Q *= 1e-17
        Q[:, 0] = 1.0
        W[0] = 0.0
    elif kind == "one tiny row":
        Q[:, 5] *= 1e-30
        W[:, 1] *= 1e-25
    elif kind == "small where it counts":
        i = np.arange(n)[:, None]
        Q *= np.where(i % 2, 1e-14, 1.0)
        W *= np.where(i % 2, 1.0, 1e-15)
    elif kind == "steps":  # a scale that grows by more than the digits' reach
        Q *= 10.0 ** (np.arange(n) // 40)[:, None]
        W *= 10.0 ** -(np.arange(n) // 35)[:, None]
    elif kind == "tiny":
        Q, W = Q * 1e-250, W * 1e20
    elif kind == "huge":
        Q, W = Q * 1e140, W * 1e-290
    elif kind == "denormal":
        W[:, 0] *= 1e-311
        Q[0] *= 1e-310
    elif kind == "spikes":
        Q *= r.random(Q.shape) < 0.01
        W *= r.random(W.shape) < 0.01
    else:
        Q[1] = 0.0
        W[:448] = 0.0
    _check(Q, W)


def test_infinities_as_in_fp64():
    import torch

    import paper_2210_15763_gb300 as bbl
    r = np.random.default_rng(4)
    Q, W = r.standard_normal((6, 300, 8)), r.standard_normal((300, 8))
    Q[2, 77, 3], W[5, 6], W[9, 1], W[77, 2] = np.inf, np.nan, -np.inf, 0.0
    C = bbl.block_gram(torch.from_numpy(Q).cuda(), torch.from_numpy(W).cuda()).cpu().numpy()
    with np.errstate(all="ignore"):
        want = (_flat(Q)[:, :, None] * W[:, None, :]).sum(axis=0)
    assert (np.isnan(C) == np.isnan(want)).all()
    inf = np.isinf(want)
    assert inf.any() and (C[inf] == want[inf]).all()


@pytest.mark.parametrize("n,b,m", [(160001, 8, 32), (311297, 4, 48), (170003, 2, 32), (70001, 16, 528), (2049, 8, 1040)])
def test_many_rows(n, b, m):
    r = np.random.default_rng(n)
    Q, W = r.standard_normal((m // b, n, b)), r.standard_normal((n, b))
    _check(Q, W, cols=np.unique(r.integers(0, m, 24)), rows=np.unique(np.r_[r.integers(0, n, 500), n - 1]))


@pytest.mark.parametrize("b,m", [(2, 30), (2, 32), (2, 46), (2, 48), (4, 12), (4, 16), (4, 28), (4, 32), (4, 36), (4, 40), (8, 8), (8, 16), (16, 16)])
def test_either_side_of_the_dispatch(b, m):
    r = np.random.default_rng(b + m)
    for n in (333, 10001):
        _check(r.standard_normal((m // b, n, b)), r.standard_normal((n, b)), rows=np.arange(0, n, 7))


@pytest.mark.parametrize("n", [400000, 400001])
def test_two_columns_of_many_rows(n):
    r = np.random.default_rng(n)
    Q, W = r.standard_normal((16, n, 2)), r.standard_normal((n, 2))
    _check(Q, W, cols=np.arange(0, 32, 3), rows=np.r_[0:200, n - 200:n])
