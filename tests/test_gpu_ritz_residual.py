"""Residuals of the Ritz pairs at the level of FP64 arithmetic, for widths whose
sequential kernels use FP64 throughout as well as for the others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,bound", [(1, 1e-15), (4, 1e-15), (8, 1e-15), (3, 3e-16), (5, 3e-16), (9, 3e-16), (12, 3e-16),
                                     (16, 3e-16)])
def test_residuals(p, bound):
    """bound: of the matrix' row-sum norm.  FP64 forms a residual to (2p + 1)^(1/2) 2^-53 of
    its rows' own sums, of which the norm is the largest; 3e-16 is 2.7 x 2^-53."""
    import torch

    import paper_2210_15763_gb300 as bbl
    r = np.random.default_rng(p)
    for m in (40, 90, 200, 350):
        for kind in range(3):
            band = r.standard_normal((m, p + 1))
            if kind == 1:
                band[:, 0] += 0.1 * np.arange(m)
            elif kind == 2:
                band *= 10.0 ** r.uniform(-4, 0, (m, 1))
            T = np.zeros((m, m), dtype=np.longdouble)
            for d in range(p + 1):
                T += np.diag(band[d:, d], -d) + (np.diag(band[d:, d], d) if d else 0.0)
            th, S = (x.cpu().numpy() for x in bbl.ritz_banded(torch.from_numpy(band).cuda(), 5))
            res = np.sqrt(((T @ S - S * th) ** 2).sum(axis=0).astype(np.float64))
            assert res.max() <= bound * float(np.abs(T).sum(axis=1).max())
