"""The two forms of wedge_exact on graphs of either kind, each against the oracle
(or a closed form), whatever the rule would take; graphs without a tail to look up, of
as many entries that the call asks first; and memory refused to the one form."""
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
    yield
    wedge.fail_next_allocation(-1)


def _graph(kind):
    rng = np.random.default_rng(5)
    i = np.arange(20_000)
    if kind == "uniform":
        return rng.integers(0, 9001, 60_000), rng.integers(0, 9001, 60_000), 9001
    if kind == "forest":  # most vertices of degree 1 and 2, a few triangles
        return np.concatenate([i[1:], [5, 700, 9000]]), np.concatenate([i[:-1] - i[:-1] % 3 // 2, [7, 702, 9002]]), 20_000
    if kind == "ring":  # alike degrees, many triangles
        return np.repeat(i, 12), (np.repeat(i, 12) + np.tile(np.arange(1, 13), len(i))) % len(i), len(i)
    if kind == "power law":
        prefix, m = graphgen.chunglu_weights(12_000, 2.1, 24.0)
        return *graphgen.chunglu_host(prefix, m, seed=2), 12_000
    if kind == "small":
        return rng.integers(0, 300, 4000), rng.integers(0, 300, 4000), 300
    return *graphgen.kronecker_host(14, seed=3), 1 << 14


@pytest.mark.parametrize("kind", ["uniform", "forest", "ring", "power law", "small", "kronecker"])
def test_forms_agree_with_the_oracle(kind):
    src, dst, n = _graph(kind)
    src, dst = np.asarray(src, np.int32), np.asarray(dst, np.int32)
    off, adj = oracle.csr(src, dst, n)
    g = wedge.graph_build(src, dst, n)
    for tau, omega in ((1, 2), (2, 2), (1, 10**7)):
        ref = oracle.exact(off, adj, tau, omega)
        b = wedge.bin(g, tau=tau, omega=omega)
        for form in (0, 1, 2):
            t_i = torch.full((n,), -1, dtype=torch.int64, device="cuda")
            got = wedge.force_exact(g, b, t_i=t_i, form=form)
            assert got["triangles"] == ref["t"] and np.array_equal(got["pbq"], ref["pbq"])
            assert np.array_equal(t_i.cpu().numpy().astype(np.uint64), ref["t_i"])
            assert np.array_equal(wedge.force_exact(g, b, form=form)["pbq"], ref["pbq"])
        b.free()
    g.free()


@pytest.mark.parametrize("low,high", [(20, 30_000), (700, 1500), (200, 200)])
@pytest.mark.parametrize("triangle", [False, True])
def test_bipartite(low, high, triangle):
    """Complete between two sides: no vertex has neighbours both below and above, until an edge joins two of one side."""
    src, dst = np.repeat(np.arange(low), high), low + np.tile(np.arange(high), low)
    if triangle:
        src, dst = np.append(src, 0), np.append(dst, 1)
    n = low + high
    g = wedge.graph_build(torch.as_tensor(src.astype(np.int32)).cuda(), torch.as_tensor(dst.astype(np.int32)).cuda(), n)
    b = wedge.bin(g)
    for form in (0, 1, 2):
        t_i = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        got = wedge.force_exact(g, b, t_i=t_i, form=form)
        assert got["triangles"] == (high if triangle else 0) and int(t_i.sum()) == 3 * got["triangles"]
        assert int(got["pbq"].sum()) == got["p_total"] == low * math.comb(high, 2) + high * math.comb(low, 2) + (
            2 * high if triangle else 0)
    b.free()
    g.free()


def test_memory_refused():
    """Whatever block the tails' form is refused, the call succeeds by the other one, and nothing leaks."""
    src, dst = graphgen.kronecker_host(14, seed=1)
    off, adj = oracle.csr(src, dst, 1 << 14)
    ref = oracle.exact(off, adj, 1, 2)
    g = wedge.graph_build(src, dst, 1 << 14)
    b = wedge.bin(g)
    t_i = torch.zeros(1 << 14, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    base, refused = wedge.pool_used_bytes(), 0
    for k in range(40):
        wedge.fail_next_allocation(k)
        try:
            wedge.force_exact(g, b, t_i=t_i, form=1)
        except wedge.WedgeError as e:
            assert e.status == 2
            refused += 1
        wedge.fail_next_allocation(k)
        got = wedge.exact(g, b, t_i=t_i)
        wedge.fail_next_allocation(-1)
        assert np.array_equal(got["pbq"], ref["pbq"])
        assert np.array_equal(t_i.cpu().numpy().astype(np.uint64), ref["t_i"])
        torch.cuda.synchronize()
        assert wedge.pool_used_bytes() == base
    assert 5 <= refused < 40
    for k in range(40):  # and the other form
        wedge.fail_next_allocation(k)
        try:
            wedge.force_exact(g, b, form=2)
            break
        except wedge.WedgeError as e:
            assert e.status == 2 and wedge.pool_used_bytes() == base
    wedge.fail_next_allocation(-1)
    assert 5 <= k < 40
