"""Ritz solve: pairs that cyclic reduction cannot certify fall back to the
sequential kernels one by one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 2, 3, 4, 8, 16])
def test_pairs_fall_back_one_by_one(p):
    """A double value among isolated ones: its two pairs take the sequential
    kernels, the others keep the fast path's bits (those of a call that asks for
    them alone)."""
    import torch

    import paper_2210_15763_gb300 as bbl
    m, nev = 300, 6
    r = np.random.default_rng(p)
    band = np.zeros((m, p + 1))
    band[:, 0] = np.arange(m) * 2.0  # isolated values, 2 apart
    band[:, 1:] = 0.05 * r.standard_normal((m, p))
    for i in range(p):
        band[i, i + 1:] = 0.0
    for i in (m - 2, m - 1):  # decoupled: the double value, between the fourth and the fifth
        band[i] = 0.0
        band[i, 0] = 7.0
    T = torch.from_numpy(band).cuda()
    th, S = (x.cpu().numpy() for x in bbl.ritz_banded(T, nev))
    full = np.diag(band[:, 0])
    for d in range(1, p + 1):
        full += np.diag(band[d:, d], -d) + np.diag(band[d:, d], d)
    w = np.linalg.eigvalsh(full)[:nev]
    assert np.abs(th - w).max() <= 1e-14 * (2 * p + 1) * 600
    assert np.linalg.norm(full @ S - S * th, axis=0).max() <= 1e-14 * (2 * p + 1) * 600
    assert np.abs(S.T @ S - np.eye(nev)).max() <= 1e-12
    th4, S4 = (x.cpu().numpy() for x in bbl.ritz_banded(T, 4))
    assert (th[:4] == th4).all() and (S[:, :4] == S4).all()
