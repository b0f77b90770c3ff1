"""Batched runs that stop after one to a few blocks, at the basis cap or by
convergence: the graph loop gives what the host-driven loop gives, for every
block size (whose partial sums are laid out and added differently)."""
import numpy as np
import pytest

import synth
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,b", [("fp64", 4), ("fp32", 4), ("fp64", 8), ("fp32", 2), ("fp64", 16)])
@pytest.mark.parametrize("blocks", [1, 2, 3, 4, 5, 8, 9, 40])
def test_graph_and_host_loop_agree_wherever_they_stop(storage, b, blocks):
    torch, bbl = need_gpu()
    mats = [synth.kron_matrix("kron_n2e4", scale=s) for s in (0.1, 0.2, 0.15)]
    B = bbl.Batch(mats, storage=storage)
    kw = dict(tol=1e-3 if blocks == 40 else 1e-12, max_vectors=blocks * b, seed=2, polish=0)
    e1, r1, i1, s1, _ = B.solve(min(4, b), b, use_graph=True, **kw)
    e2, r2, i2, s2, _ = B.solve(min(4, b), b, use_graph=False, **kw)
    np.testing.assert_array_equal(i1, i2)
    np.testing.assert_array_equal(s1, s2)
    np.testing.assert_array_equal(e1, e2)
    np.testing.assert_array_equal(r1, r2)
    assert np.all(i1 <= blocks)
