"""The server's account of device memory is what its resident graphs hold: the
upload budget is only as good as that."""
import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")

ROUNDING = 8 * 512  # a graph's eight blocks, each rounded up by the pool


@pytest.mark.parametrize("tau", [1, 120])
def test_resident_bytes_are_what_the_pool_hands_out(tau):
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()
    srv = wedge.Server(slots=1, tau=tau)
    torch.cuda.synchronize()
    base = wedge.pool_used_bytes()
    for i, scale in enumerate((16, 17, 15)):
        src, dst = graphgen.kronecker_host(scale, seed=i)
        srv.add_graph(src, dst, 1 << scale)
        torch.cuda.synchronize()
        used, said = wedge.pool_used_bytes() - base, srv.stats()["resident_bytes"]
        assert said <= used <= said + (i + 1) * ROUNDING
    srv.close()


def test_budget_counts_the_guide():
    """Room for one graph and the upload of another, and for the second to stay, but for its guide: evicts the first."""
    n = 1 << 16
    src, dst = graphgen.kronecker_host(16, seed=3)
    m = len(src)
    held = 8 * (n + 1) + 4 * n + 8 * m + 12 * n + 8  # the graph, L and W: what does not depend on the guide
    scratch = 2 * 8 * 2 * m + 2 * m // 16 + 8 * m + 16 * n
    wedge.load()
    srv = wedge.Server(slots=1)
    srv.add_graph(src, dst, n)
    one = srv.stats()["resident_bytes"]
    srv.close()
    g = wedge.graph_build(torch.as_tensor(src).cuda(), torch.as_tensor(dst).cuda(), n)
    n2 = int((np.diff(g.csr_numpy()[0]) >= 2).sum())
    guide = 4 * (n2 // 4)
    g.free()
    assert one >= held - 12 * (n - n2) + guide
    srv = wedge.Server(slots=1, hbm_budget_bytes=(held - 12 * (n - n2)) + guide // 2 + held + scratch)
    srv.add_graph(src, dst, n)
    srv.add_graph(src, dst, n)
    st = srv.stats()
    assert st["evictions"] == 1 and st["resident_graphs"] == 1
    srv.close()
