"""CholQR2 over the exponent range, where its Cholesky replaces divisions by a
reciprocal and where that leaves the normal numbers, and at rows beyond 64 per
thread."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _cholqr2(W):
    import torch

    import paper_2210_15763_gb300 as bbl
    q = torch.from_numpy(W.copy()).cuda()
    B, nd = bbl.cholqr2(q)
    return q.cpu().numpy(), B.cpu().numpy(), nd


@pytest.mark.parametrize("b", [1, 2, 3, 4, 8, 16])
def test_powers_of_two_change_no_bit(b):
    """Integers, so that every product is exact: pivots below 2^-959 and above 2^957 take a division."""
    r = np.random.default_rng(b)
    W = r.integers(-9, 10, (700, b)).astype(np.float64)
    Q0, B0, nd = _cholqr2(W)
    assert nd == 0
    for k in (-485, -482, 300, 479, 484):
        Q, B, nd = _cholqr2(np.ldexp(W, k))
        assert nd == 0 and (Q == Q0).all() and (np.ldexp(B, -k) == B0).all()


@pytest.mark.parametrize("b", [2, 4, 8, 16])
@pytest.mark.parametrize("scale", [1e-157, 1e-155, 1e152])
def test_pivots_without_a_normal_reciprocal(b, scale):
    r = np.random.default_rng(b)
    W = r.standard_normal((5000, b)) * scale
    Q, B, nd = _cholqr2(W)
    assert nd == 0
    # the first Gram matrix holds at least 40 bits, so the second pass corrects 1e-12
    # b to FP64 rounding
    assert np.abs(Q.T @ Q - np.eye(b)).max() <= 1e-14
    assert np.abs(Q @ (B / scale) - W / scale).max() <= 1e-11


@pytest.mark.parametrize("b", [1, 2, 8])
def test_more_than_64_rows_per_thread(b):
    import torch

    import paper_2210_15763_gb300 as bbl
    n = 64 * 608 * 256 + 777
    g = torch.Generator(device="cuda")
    g.manual_seed(b)
    W = torch.randn(n, b, generator=g, device="cuda") + 0.5
    D = W.double()
    R = torch.linalg.cholesky(D.T @ D, upper=True)
    B, nd = bbl.cholqr2(W)
    assert nd == 0
    # FP32 storage of Q (2^-24 of each row), FP32 runs of 64 products
    assert float((B - R).abs().max() / R.abs().max()) <= 1e-6
    Q = W.double()
    assert float((Q.T @ Q - torch.eye(b, dtype=torch.float64, device="cuda")).abs().max()) <= 1e-6
