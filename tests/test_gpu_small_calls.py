"""Small inputs: sorts of at most one 1536-key tile per SM (whose number of
keys may be known to the device alone), scans of one tile and sample budgets of
less than a full chip take kernels' short forms. Sizes on
either side of each line, against plain sorting by torch (integers: equal) and
against the same samples drawn in one long call.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()
    yield
    wedge.trim()


def _edges(m, n, repeat=1):
    gen = torch.Generator("cuda").manual_seed(m + n)
    src, dst = (torch.randint(0, n, (m // repeat + 1,), generator=gen, device="cuda", dtype=torch.int32) for _ in "sd")
    return src.repeat(repeat)[:m].contiguous(), dst.repeat(repeat)[:m].contiguous()


def _check(src, dst, n):
    torch.cuda.synchronize()
    g = wedge.graph_build(src, dst, n)
    u, v = src.long(), dst.long()
    keys = torch.unique(torch.cat([u * n + v, v * n + u])[torch.cat([u != v, u != v])])
    gi = g.info()
    assert gi.n_adj == keys.numel()
    adj = torch.empty(max(gi.n_adj, 1), dtype=torch.int32, device="cuda")
    off = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    deg = torch.empty(n, dtype=torch.int32, device="cuda")
    g.copy(off=off, adj=adj, deg=deg)
    assert torch.equal(adj[: gi.n_adj].long(), keys % n)
    ref = torch.bincount(keys // n, minlength=n)
    assert torch.equal(deg.long(), ref) and torch.equal(off[1:], torch.cumsum(ref, 0)) and int(off[0]) == 0
    return g, ref


def _lines():
    sm = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1
    return 1536, 1536 * sm


@pytest.mark.parametrize("where", ["tile", "chip"])
@pytest.mark.parametrize("delta", [-1, 0, 1])
@pytest.mark.parametrize("n", [200, 4096, 4097, 70_000])
def test_builds_about_the_small_sort(where, delta, n):
    m = _lines()[where == "chip"] + delta
    _check(*_edges(m, n), n)[0].free()


@pytest.mark.parametrize("m", [1, 2, 3, 1537, 20_000])
@pytest.mark.parametrize("left", [0, 1, 2])
def test_few_edges_left(m, left):
    """Loops, or one or two edges again and again: the transposed sort has `left` keys (its host does not know)."""
    src = torch.arange(m, device="cuda", dtype=torch.int32) % max(left, 1)
    dst = src + 5 if left else src.clone()
    _check(src, dst, 9)[0].free()


@pytest.mark.parametrize("n", [3000, 300_000])
def test_long_list_of_few_edges(n):
    """The forward sort is past the line, the transposed one (repeats dropped) before it."""
    _check(*_edges(_lines()[1] * 3, n, repeat=12), n)[0].free()


@pytest.mark.parametrize("n,m,tau", [(4096, 30_000, 2), (4097, 30_000, 2), (20_000, 3000, 2), (300_000, 900_000, 2),
                                     (3_000_000, 9_000_000, 2), (9_000_000, 20_000_000, 60)])
def test_bins_read_back(n, m, tau):
    g, deg = _check(*_edges(m, n), n)
    b = wedge.bin(g, tau=tau, omega=2)
    info = b.info()
    lo = torch.tensor(list(info.lo_deg)[: info.n_bins])
    which = torch.searchsorted(lo, deg.cpu(), right=True) - 1
    n_b = torch.bincount(which[deg.cpu() > 0], minlength=info.n_bins)
    pairs = (deg * (deg - 1) // 2).cpu()
    p_b = torch.zeros(info.n_bins, dtype=torch.int64).index_add_(0, which, pairs)
    assert list(info.n_b)[1:info.n_bins] == n_b[1:].tolist()
    assert list(info.p_b)[2:info.n_bins] == p_b[2:].tolist()
    b.free()
    g.free()


@pytest.mark.parametrize("k", [1, 255, 257, 20_000, 155_649, 700_000, 1_400_000])
def test_budgets_about_the_full_chip(k):
    """Counts do not depend on how samples are dealt to threads: one call and two calls of a part each agree."""
    n = 5000
    g = _check(*_edges(60_000, n), n)[0]
    b = wedge.bin(g, tau=1, omega=2)

    def draw(count, first):
        c = wedge.sample(g, b, seed=5, k_per_bin=count, k_global=count, first_sample=first)
        return torch.tensor([[int(x) for x in row] for row in c.q]), int(c.closed_global)

    q, closed = draw(k, 0)
    part = (k + 2) // 3
    q0, c0 = draw(part, 0)
    q1, c1 = draw(k - part, part) if k > part else (torch.zeros_like(q0), 0)
    assert torch.equal(q, q0 + q1) and closed == c0 + c1
    b.free()
    g.free()


@pytest.mark.parametrize("k", [1, 2047, 2048, 2049, 40_000, 2_500_000])
def test_triangle_keys_about_a_tile(k):
    """Ratio quartiles and box counts against the records, written whole (aligned) and word by word."""
    n = 700
    g = _check(*_edges(9000, n), n)[0]
    b = wedge.bin(g)
    room = torch.zeros(8 * k + 8, dtype=torch.int32, device="cuda")
    aligned, shifted = room[: 8 * k], torch.zeros(8 * k + 8, dtype=torch.int32, device="cuda")[1 : 8 * k + 1]
    t = wedge.triangle_stats(g, b, 11, k, records=aligned)
    u = wedge.triangle_stats(g, b, 11, k, records=shifted)
    assert torch.equal(aligned, shifted) and int(room[8 * k :].abs().sum()) == 0
    r = aligned.view(-1, 8)
    d = r[r[:, 3] != 0][:, 4:7].cpu().double()
    assert t["closed"] == u["closed"] == len(d)
    lo, hi = (d.min(1).values, d.max(1).values) if len(d) else (d.sum(1), d.sum(1))
    ratio = (hi / lo).sort().values
    if len(d):
        at = [0] + [max(1, -(-len(d) * q // 4)) - 1 for q in (1, 2, 3)] + [len(d) - 1]
        assert list(t["ratio_q"]) == list(u["ratio_q"]) == ratio[at].tolist()
    b.free()
    g.free()
