"""Ritz solve by spectrum slicing and block cyclic reduction (ritz_cr.cu)
against LAPACK, at the edges of its blocks (8 rows for p <= 8, 16 above),
windows and shift tiles, over the exponent range, and where a pair cannot be
certified and the sequential kernels take over."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _band_matrix(m, p, seed):
    r = np.random.default_rng(seed)
    T = np.zeros((m, m))
    for d in range(min(p, m - 1) + 1):
        v = r.standard_normal(m - d)
        T += np.diag(v, -d)
        if d:
            T += np.diag(v, d)
    return T


def _solve(T, p, nev):
    import torch

    import paper_2210_15763_gb300 as bbl
    m = T.shape[0]
    band = np.full((m, p + 1), np.nan)  # entries left of the matrix are ignored
    for d in range(p + 1):
        band[d:, d] = np.diagonal(T, -d) if d < m else 0.0
    th, S = bbl.ritz_banded(torch.from_numpy(band).cuda(), nev)
    return th.cpu().numpy(), S.cpu().numpy()


def _check(T, p, nev):
    th, S = _solve(T, p, nev)
    w = np.linalg.eigvalsh(T)
    scale = np.abs(w).max()
    # a certified pair's residual is at most 1e-14 of the Gershgorin bound,
    # which is at most (2p + 1) of the spectrum; the quotient's error is
    # bounded by the residual
    tol = 1e-14 * (2 * p + 1) * scale
    assert np.abs(th - w[:nev]).max() <= tol
    assert np.linalg.norm(T @ S - S * th, axis=0).max() <= tol
    gap = np.diff(w[:nev]).min() / scale if nev > 1 else 1.0
    # two vectors overlap by at most the sum of their residuals over their gap
    # (close values are orthogonalised)
    assert np.abs(S.T @ S - np.eye(nev)).max() <= 1e-14 + 2 * tol / scale / max(gap, 1e-3)
    k = np.argmax(np.abs(S), axis=0)
    assert (S[k, np.arange(nev)] > 0).all()


@pytest.mark.parametrize("p", [0, 1, 2, 3, 4, 8, 9, 16])
@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 15, 16, 17, 18, 63, 64, 65, 129, 500])
def test_sizes(m, p):
    _check(_band_matrix(m, p, 31 * m + p), p, min(m, 6))


@pytest.mark.parametrize("p,m,nev", [(1, 2500, 4), (8, 1800, 3), (16, 1100, 2), (8, 40, 32)])
def test_long_bands_and_many_pairs(p, m, nev):
    _check(_band_matrix(m, p, 5), p, nev)


@pytest.mark.parametrize("scale", [1e-200, 1e-30, 1e30, 1e200])
def test_exponents(scale):
    T = _band_matrix(120, 4, 9)
    th, S = _solve(T * scale, 4, 5)
    w = np.linalg.eigvalsh(T)
    assert np.abs(th / scale - w[:5]).max() <= 1e-14 * 9 * np.abs(w).max()
    assert np.linalg.norm(T @ S - S * (th / scale), axis=0).max() <= 1e-14 * 9 * np.abs(w).max()


@pytest.mark.parametrize("gap", [0.0, 1e-9, 1e-6, 1e-4])
def test_close_values(gap):
    """Two copies of one matrix, the second shifted: every value is (nearly) double."""
    A = _band_matrix(40, 3, 2)
    T = np.zeros((80, 80))
    T[:40, :40] = A
    T[40:, 40:] = A + gap * np.eye(40)
    th, S = _solve(T, 3, 6)
    w = np.linalg.eigvalsh(T)
    scale = np.abs(w).max()
    assert np.abs(th - w[:6]).max() <= 1e-12 * scale
    assert np.abs(S.T @ S - np.eye(6)).max() <= 1e-10
