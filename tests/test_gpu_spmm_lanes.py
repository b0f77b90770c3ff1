"""FP64 SpMM with few lanes per row and several running sums per lane
(spmm_csr_kernel): the remainders of every row length, at the row counts and
mean lengths where the number of lanes changes, against extended precision."""
from types import SimpleNamespace

import numpy as np
import pytest

from tests.gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu
LD = np.longdouble


# (rows, row lengths): 16 lanes x 2 sums, 8 x 4, 8 x 2, and just below the row count of each
@pytest.mark.parametrize("n,lengths", [(19_456, (30, 110)), (19_455, (30, 110)), (38_912, (0, 130)), (38_911, (0, 130)),
                                       (19_456, (0, 70)), (19_455, (0, 70))])
@pytest.mark.parametrize("b", [1, 2, 4])
def test_rows_of_every_length(n, lengths, b):
    torch, bbl = need_gpu()
    r = np.random.default_rng(n + b)
    lo, hi = lengths
    ln = lo + np.arange(n) % (hi - lo)
    rp = np.concatenate([[0], np.cumsum(ln)]).astype(np.int64)
    first = np.arange(n) * 7919 % (n - 97 * hi)
    ci = (np.repeat(first, ln) + (np.arange(rp[-1]) - np.repeat(rp[:-1], ln)) * 97).astype(np.int32)
    va = r.standard_normal(rp[-1])
    V = r.standard_normal((n, b))
    A = SimpleNamespace(n=n, row_ptr=rp, col=ci, val=va)
    W = bbl.spmm(bbl.Matrix(A, storage="fp64", fmt="csr"), to_dev(torch, V, torch.float64)).cpu().numpy()
    prod = va[:, None].astype(LD) * V[ci].astype(LD)
    cs = np.concatenate([np.zeros((1, b), LD), np.cumsum(np.abs(prod), axis=0)])
    mag = (cs[rp[1:]] - cs[rp[:-1]]).astype(float)
    exact = np.zeros((n, b), LD)
    nz = ln > 0
    exact[nz] = np.add.reduceat(prod, rp[:-1][nz], axis=0)
    # length products, each rounded once in a chain or a tree of additions
    assert np.all(np.abs(W - exact) <= (ln[:, None] * 2.0 ** -53 + 2.0 ** -50) * mag)
