"""Scratch buffers kept between the single calls (api.cu): reuse over sizes,
streams and threads gives the results of fresh buffers, the idle memory stays
bounded, and a release empties it."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
# (n, b, blocks): scratch of several size classes, up to above the 64 MiB limit
SIZES = [(1, 1, 1), (333, 4, 5), (20_000, 8, 30), (5_000, 16, 128), (100_003, 8, 3), (60_000, 16, 128)]
LIMIT = 256 << 20


def _inputs(k):
    import torch
    n, b, nb = SIZES[k]
    gen = torch.Generator(device="cuda").manual_seed(k)
    Q = torch.randn(nb, n, b, device="cuda", dtype=torch.float64, generator=gen) / n ** 0.5
    return Q, torch.randn(n, b, device="cuda", dtype=torch.float64, generator=gen)


def _run(Q, W, stream=None):
    import paper_2210_15763_gb300 as bbl
    C = bbl.block_gram(Q, W, stream=stream)
    V = W.clone()
    bbl.block_reorth(Q, V, passes=1, stream=stream)
    return C, V


def _agree(got, want, n):
    # two orders of the same n-term FP64 sums: n 2^-53 relative to |Q|^T|W| <= |q||w|
    for a, b in zip(got, want):
        scale = float(b.abs().max()) + 1.0
        assert float((a - b).abs().max()) <= 64 * 2.0 ** -53 * scale * max(1.0, n ** 0.5)


def test_reuse_over_sizes_and_bound():
    import torch

    import paper_2210_15763_gb300 as bbl
    bbl.workspace_release()
    first = {}
    for k in range(len(SIZES)):
        first[k] = _run(*_inputs(k))
        bbl.workspace_release()
        assert bbl.workspace_bytes() == 0
    for k in list(range(len(SIZES))) + list(reversed(range(len(SIZES)))):
        _agree(_run(*_inputs(k)), first[k], SIZES[k][0])
        assert bbl.workspace_bytes() <= LIMIT
    held = bbl.workspace_bytes()
    assert held > 0
    Q, W = _inputs(2)
    _run(Q, W)
    a = bbl.workspace_bytes()
    _run(Q, W)
    assert bbl.workspace_bytes() == a          # the same size takes its own buffers again
    bbl.workspace_release()
    assert bbl.workspace_bytes() == 0
    torch.cuda.synchronize()


def test_streams_and_threads():
    import torch

    import paper_2210_15763_gb300 as bbl
    ins = [_inputs(k) for k in (1, 2, 4)]
    want = [_run(*x) for x in ins]
    torch.cuda.synchronize()
    bad = []

    def work(t):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                for i in range(12):
                    k = (t + i) % len(ins)
                    got = _run(*ins[k], stream=s)
                    s.synchronize()
                    _agree(got, want[k], ins[k][1].shape[0])
        except Exception as e:  # noqa: BLE001
            bad.append(e)

    ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad
    assert bbl.workspace_bytes() <= LIMIT
    bbl.workspace_release()
    assert np.isclose(bbl.workspace_bytes(), 0)
