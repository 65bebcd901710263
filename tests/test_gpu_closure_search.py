"""The closure search (sectors of eight ids, found by interpolation, then by
halving) through wedge_classify, against the oracle: rows of every length
around a sector, rows whose ids are even, clustered at one end, in two far
clumps or a dense run, searched for ids that are there, between two that are,
before the first and after the last.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()


def _row(rng, shape, length, lo, n):
    if shape == "even":
        return np.sort(rng.choice(np.arange(lo, n), length, replace=False))
    if shape == "low":
        return lo + np.arange(length) * 2
    if shape == "high":
        return n - 1 - np.arange(length)[::-1] * 3
    if shape == "clumps":
        half = length // 2
        return np.concatenate([lo + np.arange(half), n - 1 - np.arange(length - half)[::-1]])
    return lo + (n - lo) // 2 + np.arange(length)  # run


@pytest.mark.parametrize("shape", ["even", "low", "high", "clumps", "run"])
def test_rows(shape):
    rng = np.random.default_rng(len(shape))
    n, lo = 200_000, 200
    lengths = list(range(1, 41)) + [63, 64, 65, 127, 500, 1000, 4095, 20_000]
    src, dst = [], []
    for v, k in enumerate(lengths):
        row = _row(rng, shape, k, lo, n)
        src.append(np.full(k, v))
        dst.append(row)
    # one hub larger than every row, joined to each of them, so that theirs are searched for it and for each other
    hub = 199
    src.append(np.full(30_000, hub))
    dst.append(rng.choice(np.arange(lo, n), 30_000, replace=False))
    src, dst = np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)
    g = wedge.graph_build(src, dst, n)
    b = wedge.bin(g)
    off, adj = oracle.csr(src, dst, n)
    deg = np.diff(off)
    v1, v2 = [], []
    for v in range(len(lengths)):
        row = adj[off[v]:off[v + 1]]
        ask = np.concatenate([row, row - 1, row + 1, [0, lo, n - 1, hub]])
        ask = np.unique(ask[(ask >= 0) & (ask < n) & (ask != v)])
        v1.append(np.full(ask.size, v))
        v2.append(ask)
    v1, v2 = np.concatenate(v1).astype(np.int32), np.concatenate(v2).astype(np.int32)
    v0 = np.full(v1.size, hub, np.int32)
    assert deg.max() >= 20_000
    want = oracle.classify(off, adj, 1, 2, v0, v1, v2)
    for a, z in ((v1, v2), (v2, v1)):
        q = torch.zeros(v1.size, dtype=torch.uint8, device="cuda")
        wedge.classify(g, b, *(torch.as_tensor(x).cuda() for x in (v0, a, z)), q)
        assert np.array_equal(q.cpu().numpy(), want)
    assert 0 < np.count_nonzero(want) < want.size
