"""wedge_exact where its row forms and orders change: cliques of many sizes
(closed forms: t_i = C(s - 1, 2), every closed wedge of the last class) on
more vertices than the bit maps hold, vertex counts around the all-pairs
ranking, tails shorter and longer than a warp's list, against the oracle.
"""
import math

import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()


@pytest.mark.parametrize("sizes", [[3] * 50, [2, 3, 33, 34, 130, 700], [1100, 40], list(range(60, 240)) * 3])
def test_cliques(sizes):
    rng = np.random.default_rng(len(sizes))
    n = sum(sizes) + 7
    ids = rng.permutation(n)
    src, dst, t_i = [], [], np.zeros(n, np.int64)
    at = 0
    for s in sizes:
        members = ids[at:at + s]
        at += s
        i, j = np.triu_indices(s, 1)
        src.append(members[i])
        dst.append(members[j])
        t_i[members] = math.comb(s - 1, 2)
    src, dst = (torch.as_tensor(np.concatenate(x).astype(np.int32)).cuda() for x in (src, dst))
    g = wedge.graph_build(src, dst, n)
    b = wedge.bin(g)
    ti = torch.zeros(n, dtype=torch.int64, device="cuda")
    got = wedge.exact(g, b, t_i=ti)
    assert got["triangles"] == sum(math.comb(s, 3) for s in sizes)
    assert np.array_equal(ti.cpu().numpy(), t_i)
    want = np.zeros_like(got["pbq"])
    for s in sizes:
        if s > 2:
            want[(s - 1).bit_length(), 3] += s * math.comb(s - 1, 2)
    assert np.array_equal(got["pbq"], want)
    assert np.array_equal(wedge.exact(g, b)["pbq"], want)  # without t_i


@pytest.mark.parametrize("n,gamma,mean", [(8191, 2.2, 20.0), (8192, 2.2, 20.0), (8193, 2.2, 20.0), (70_000, 2.0, 60.0),
                                          (40_000, 2.6, 6.0)])
def test_power_law(n, gamma, mean):
    prefix, m = graphgen.chunglu_weights(n, gamma, mean)
    src, dst = graphgen.chunglu_host(prefix, m, seed=n)
    g = wedge.graph_build(src, dst, n)
    b = wedge.bin(g, tau=2, omega=2)
    ti = torch.zeros(n, dtype=torch.int64, device="cuda")
    got = wedge.exact(g, b, t_i=ti)
    off, adj = oracle.csr(src, dst, n)
    ref = oracle.exact(off, adj, 2, 2)
    assert got["triangles"] == ref["t"]
    assert np.array_equal(got["pbq"], ref["pbq"])
    assert np.array_equal(ti.cpu().numpy().astype(np.uint64), ref["t_i"])
