"""wedge_triangle_stats' box plots against the records of the same call, at numbers
of records about a CTA's tile of them: count, least, median, quartiles, most,
whiskers and outliers of every group, in exact integers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


@pytest.mark.parametrize("k", [1, 31, 2047, 2048, 2049, 6145, 40_000, 2_500_000])
def test_boxes_are_those_of_the_records(k):
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()
    n = 700
    gen = torch.Generator("cuda").manual_seed(3)
    src, dst = ((torch.rand(9000, generator=gen, device="cuda") ** 2 * n).int() for _ in "sd")
    torch.cuda.synchronize()
    g = wedge.graph_build(src, dst, n)
    b = wedge.bin(g)
    records = torch.zeros(8 * k, dtype=torch.int32, device="cuda")
    t = wedge.triangle_stats(g, b, 17, k, records=records)
    r = records.cpu().numpy().reshape(-1, 8)
    d = r[r[:, 3] != 0][:, 4:7].astype(np.int64)
    least, most = (d.min(1), d.max(1)) if len(d) else (d[:, 0], d[:, 0])
    group = np.where(least <= 2, least, 1 + np.ceil(np.log2(np.maximum(least, 2))).astype(np.int64))  # 3..4, 5..8, ...
    want = np.zeros((len(t["box"]), len(wedge.BOX_FIELDS)), np.uint64)
    for i in range(len(want)):
        v = np.sort(most[group == i])
        if not len(v):
            continue
        q1, q2, q3 = (int(v[max(1, -(-len(v) * q // 4)) - 1]) for q in (1, 2, 3))
        inside = v[(2 * v >= 2 * q1 - 3 * (q3 - q1)) & (2 * v <= 2 * q3 + 3 * (q3 - q1))]
        want[i] = [len(v), v[0], q1, q2, q3, v[-1], inside[0], inside[-1], len(v) - len(inside)]
    assert t["closed"] == len(d) and np.array_equal(t["box"], want)
    b.free()
    g.free()
