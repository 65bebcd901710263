"""The tails' form of wedge_exact in groups of edges, and with rows that fit neither
bit map nor hash table: what takes 2^27 edges, 2^19 ranks above a vertex or rows
of thousands otherwise, on small graphs by lower limits. Every count against the oracle, entry by entry."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")

_cache = {}


def _case(kind):
    """Graph, bins and the oracle's counts, of one kind."""
    if kind not in _cache:
        import __graft_entry__
        __graft_entry__.build()
        wedge.load()
        rng = np.random.default_rng(8)
        if kind == "kronecker":  # few vertices: ranked pair by pair
            src, dst, n = *graphgen.kronecker_host(12, seed=6), 1 << 12
        elif kind == "power law":
            prefix, m = graphgen.chunglu_weights(15_000, 2.05, 40.0)
            src, dst, n = *graphgen.chunglu_host(prefix, m, seed=3), 15_000
        else:  # a clique (rows of up to 1,299) whose members have many other neighbours of lower degree
            ids = rng.permutation(40_000).astype(np.int32)
            i, j = np.triu_indices(1300, 1)
            src = np.concatenate([ids[i], ids[rng.integers(0, 1300, 90_000)], ids[rng.integers(1300, 40_000, 20_000)]])
            dst = np.concatenate([ids[j], ids[rng.integers(1300, 40_000, 90_000)], ids[rng.integers(1300, 40_000, 20_000)]])
            n = 40_000
        off, adj = oracle.csr(src, dst, n)
        g = wedge.graph_build(src, dst, n)
        _cache[kind] = g, wedge.bin(g, tau=2, omega=2), oracle.exact(off, adj, 2, 2), n
    return _cache[kind]


def _check(kind, **limits):
    g, b, ref, n = _case(kind)
    t_i = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    got = wedge.force_exact(g, b, t_i=t_i, form=1, **limits)
    assert got["triangles"] == ref["t"]
    assert np.array_equal(got["pbq"], ref["pbq"])
    assert np.array_equal(t_i.cpu().numpy().astype(np.uint64), ref["t_i"])


@pytest.mark.parametrize("kind", ["kronecker", "power law", "clique"])
@pytest.mark.parametrize("group_edges", [1, 3000, 20_001, 100_000, 1 << 27])
def test_groups(kind, group_edges):
    _check(kind, group_edges=group_edges)


@pytest.mark.parametrize("kind", ["kronecker", "power law", "clique"])
@pytest.mark.parametrize("map_ranks,table_row", [(0, 0xFFFFFFFF), (0, 0), (0, 200), (700, 0), (700, 1100), (1200, 0xFFFFFFFF)])
def test_row_forms(kind, map_ranks, table_row):
    _check(kind, map_ranks=map_ranks, table_row=table_row)


def test_groups_of_every_row_form():
    _check("clique", group_edges=50_000, map_ranks=900, table_row=1150)
    _check("power law", group_edges=9000, map_ranks=3000, table_row=150)


def test_out_of_range():
    g, b, _, _ = _case("kronecker")
    for limits in ({"form": 3}, {"form": -1}, {"form": 1, "group_edges": 0}):
        with pytest.raises(wedge.WedgeError) as e:
            wedge.force_exact(g, b, **limits)
        assert e.value.status == 1
