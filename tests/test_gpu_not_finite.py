"""Non-finite Ritz values: the calls return (a NaN takes its place in the order of
the values and never selects memory), and the next call on the same context is
not affected."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _band(m, p, seed):
    r = np.random.default_rng(seed)
    band = r.standard_normal((m, p + 1))
    band[:, 0] += np.arange(m)
    return band


@pytest.mark.parametrize("p", [1, 3, 8, 16])
@pytest.mark.parametrize("nev", [2, 8, 32])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_band(p, nev, value):
    import torch

    import paper_2210_15763_gb300 as bbl
    good = torch.from_numpy(_band(200, p, 3)).cuda()
    want = bbl.ritz_banded(good, nev)[0].cpu().numpy()
    bad = good.clone()
    bad[77, 1] = value
    theta, S = bbl.ritz_banded(bad, nev)
    # every elimination carries the entry into the vectors and their quotients
    assert np.isnan(theta.cpu().numpy()).all()
    assert theta.shape == (nev,) and S.shape == (200, nev)
    assert (bbl.ritz_banded(good, nev)[0].cpu().numpy() == want).all()


def test_degenerate_band_beyond_fp32():
    """Equal values go to the sequential kernels, whose FP32 pairs overflow above 3.4e38."""
    import torch

    import paper_2210_15763_gb300 as bbl
    band = np.zeros((64, 9))
    band[:, 0] = 1e200
    theta, _ = bbl.ritz_banded(torch.from_numpy(band).cuda(), 8)
    assert theta.shape == (8,)


def test_solve_overflow_is_reported():
    import types

    import paper_2210_15763_gb300 as bbl
    n = 200  # a full matrix and a constant pivot: every FP32 row sum is infinite
    A = types.SimpleNamespace(n=n, row_ptr=np.arange(0, n * n + 1, n, dtype=np.int64),
                              col=np.tile(np.arange(n, dtype=np.int32), n), val=np.full(n * n, 3e38))
    with pytest.raises(bbl.BBLError, match="NUMERICAL"):
        bbl.solve(bbl.Matrix(A, storage="fp32"), 2, 1, pivot=np.ones((n, 1)))
