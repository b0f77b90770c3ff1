"""The rows of the truncated space (radix selection of the smallest diagonal
entries): ties, signs, signed zeros, and sizes around the launch shape.  With
at most b rows the pivot holds their unit vectors, so the set is seen exactly."""
from types import SimpleNamespace

import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _key(d):
    u = d.view(np.uint64)
    return np.where(u >> np.uint64(63), ~u, u | np.uint64(1 << 63))


@pytest.mark.parametrize("kind", ["normal", "equal", "ties", "zeros", "wide", "negative"])
@pytest.mark.parametrize("n", [16, 257, 311_297])
def test_rows_with_the_smallest_diagonal(kind, n):
    torch, bbl = need_gpu()
    r = np.random.default_rng(n)
    d = {"normal": r.standard_normal(n), "equal": np.full(n, 2.5), "ties": r.integers(-2, 3, n).astype(float),
         "zeros": np.where(r.random(n) < 0.5, -0.0, 0.0), "wide": 10.0 ** r.uniform(-300, 300, n) * r.choice([-1, 1], n),
         "negative": -1.0 - r.random(n) * 2.0 ** -40}[kind]
    M = bbl.Matrix(SimpleNamespace(n=n, row_ptr=np.arange(n + 1, dtype=np.int64), col=np.arange(n, dtype=np.int32), val=d))
    d = M.diagonal().cpu().numpy()  # as the matrix holds it: a sum over lanes, -0 becomes +0
    for k in (1, 2, 7, 16):
        P = bbl.pivot_bootstrap(M, k, 16, sub_tol=1e-6).cpu().numpy()
        want = np.sort(np.argsort(_key(d), kind="stable")[:k])     # ties: the lower index first
        got = np.flatnonzero((P[:, :k] == 1.0).any(axis=1) & (np.abs(P[:, :k]).sum(axis=1) == 1.0))
        assert np.array_equal(got, want), (kind, k)
