"""L, W and the per-bin sums against numpy where the number of bins changes how
vertices are scattered, up to the most there can be, at vertex counts around the
4096-vertex tiles."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


@pytest.mark.parametrize("n", [4095, 4096, 4097, 20_001])
def test_bins_about_the_scatter_forms(n):
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()
    prefix, m = graphgen.chunglu_weights(n, 2.1, 60.0)
    src, dst = graphgen.chunglu_host(prefix, m, seed=n)
    g = wedge.graph_build(src, dst, n)
    deg = np.diff(g.csr_numpy()[0])
    seen = set()
    for tau in [1, 30, *range(36, 56), 120, 200, *range(236, 252)]:
        try:
            b = wedge.bin(g, tau=tau, omega=2)
        except wedge.WedgeError as e:
            assert e.status == 1 and tau > 236  # beyond the last bin id
            continue
        info = b.info()
        nb = info.n_bins
        seen.add(nb)
        which = np.searchsorted(np.array(info.lo_deg[:nb]), deg, side="right") - 1
        some = np.nonzero(deg >= 2)[0]
        order = some[np.argsort(which[some], kind="stable")]
        L, W = np.empty(len(order), np.int32), np.empty(len(order) + 1, np.uint64)
        b.copy(L, W)
        assert np.array_equal(L, order)
        assert np.array_equal(W.astype(np.int64), np.concatenate([[0], np.cumsum(deg[order] * (deg[order] - 1) // 2)]))
        assert list(info.n_b)[1:nb] == np.bincount(which[deg > 0], minlength=nb)[1:].tolist()
        b.free()
    assert {51, 52, 53, 54, 256} <= seen
    g.free()
