"""wedge_exact on imported CSRs. Symmetry is the importer's promise and is not
checked there; a CSR of which other than half the entries go down in (degree,
id) would not fit the buffers of edges, so nothing may run on it: EINVAL, and
the next call is right."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()


def _graph(rows, n):
    deg = np.zeros(n, np.int64)
    for v, r in rows.items():
        deg[v] = len(r)
    adj = np.concatenate([np.asarray(rows[v], np.int32) for v in sorted(rows)])
    return wedge.graph_from_csr(np.concatenate([[0], np.cumsum(deg)]).astype(np.int64), adj, n)


@pytest.mark.parametrize("n", [100, 9000])
@pytest.mark.parametrize("kind", ["hub", "mixed", "cycle", "edge"])
def test_not_symmetric(kind, n):
    rows = {"hub": {0: range(1, n - 1)},                                 # every entry goes down
            "mixed": {0: [3], 1: [3], 2: [3], 3: [4, 5, 6, 7, 8]},       # five of eight do
            "cycle": {v: [(v + 1) % n] for v in range(n)},               # one of n does
            "edge": {0: [1, 2, 3], 1: [0, 2], 2: [0, 1], 4: [5]}}[kind]  # a triangle and two one-way entries: five of eight
    g = _graph(rows, n)
    b = wedge.bin(g)
    t_i = torch.ones(n, dtype=torch.int64, device="cuda")
    with pytest.raises(wedge.WedgeError) as e:
        wedge.exact(g, b, t_i=t_i)
    assert e.value.status == 1 and "symmetric" in str(e.value)
    assert int(t_i.abs().sum()) == 0
    k4 = _graph({v: [x for x in range(4) if x != v] for v in range(4)}, n)
    assert wedge.exact(k4, wedge.bin(k4), t_i=t_i)["triangles"] == 4
    assert t_i[:4].tolist() == [3] * 4 and int(t_i.sum()) == 12
