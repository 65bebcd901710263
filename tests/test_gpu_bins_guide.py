"""Bins and the sampler's guide over the wedge prefix at their edges, against the
oracle: vertex counts around a tile of 4096, degrees at the bins' boundaries,
nearly as many bins as there may be, one bin of every degree (whose cells hold
from many vertices to a fraction of one), bins without vertices. Integers: equal.
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


def _graph(n):
    """Rows of the degrees around powers of two, hubs, and isolated vertices at the end."""
    rng = np.random.default_rng(n)
    want = np.concatenate([[2**k + o for k in range(1, 10) for o in (-1, 0, 1)], [n // 2, n // 3]])
    src, dst = [], []
    for i, k in enumerate(want):
        v = int(rng.integers(0, n - 5))
        others = rng.choice(n - 5, min(int(k), n - 6), replace=False)
        src.append(np.full(others.size, v))
        dst.append(others)
    src.append(rng.integers(0, n - 5, 2 * n))
    dst.append(rng.integers(0, n - 5, 2 * n) // 7)
    return np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32)


@pytest.mark.parametrize("n", [600, 4095, 4096, 4097, 12_289])
@pytest.mark.parametrize("tau,omega", [(1, 2), (2, 2), (3, 5), (240, 2), (1, 10**7)])
def test_bins_and_samples(n, tau, omega):
    src, dst = _graph(n)
    g = wedge.graph_build(src, dst, n)
    off, adj = oracle.csr(src, dst, n)
    b = wedge.bin(g, tau=tau, omega=omega)
    ref = oracle.bins(off, tau, omega)
    info = b.info()
    nb = ref["n_bins"]
    assert info.n_bins == nb
    assert list(info.n_b[:nb]) == [int(x) for x in ref["n_b"]]
    assert list(info.p_b[:nb]) == [int(x) for x in ref["p_b"]]
    deg = np.diff(off)
    lo = np.array([int(x) for x in ref["lo"][:nb]])
    ids = np.nonzero(deg >= 2)[0]
    order = ids[np.argsort(np.searchsorted(lo, deg[ids], side="right"), kind="stable")]
    L, W = b.arrays_numpy()
    assert np.array_equal(L, order)
    assert np.array_equal(W.astype(np.int64), np.concatenate([[0], np.cumsum(deg[order] * (deg[order] - 1) // 2)]))
    c = wedge.sample(g, b, seed=n + tau, k_per_bin=700, k_global=9_000)
    want = oracle.sample(off, adj, tau, omega, n + tau, 700, 9_000)
    assert np.array_equal(c.counts_matrix(), want["counts"])
    assert c.closed_global == int(want["glob"][1]) and np.array_equal(c.stats, want["stats"])
    bins_only = wedge.sample(g, b, seed=n + tau, k_per_bin=700, flags=wedge.FLAG_SORTED_CLOSURE | wedge.FLAG_NO_GLOBAL)
    assert np.array_equal(bins_only.counts_matrix(), want["counts"])
    r = wedge.Requests([{"graph": g, "bins": b, "seed": n + tau, "k_per_bin": 700, "k_global": 9_000}])
    for mapping in (wedge.MAP_THREAD, wedge.MAP_WARP):
        got = wedge.sample_batch(r, {f"mapping_{s}": mapping for s in ("small", "medium", "large")})[0]
        assert np.array_equal(got.counts_matrix(), want["counts"]) and np.array_equal(got.stats, want["stats"])
