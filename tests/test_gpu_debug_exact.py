"""The bounds-checked build on the exact counter's forms (rows, in-lists, bit maps,
groups), and on the guide and the wedge prefix that the sampler reads at degrees of
every kind: no index leaves its buffer, and the counts are the release build's."""
import ctypes

import numpy as np
import pytest

import graphgen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


def _ok(lib, st):
    assert st == 0, lib.wedge_last_error().decode()


@pytest.mark.parametrize("kind", ["kronecker", "power law", "star and clique"])
def test_exact_and_sample(kind):
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()
    lib = wedge.load_debug()
    if kind == "kronecker":
        src, dst, n = *graphgen.kronecker_host(13, seed=6), 1 << 13
    elif kind == "power law":
        prefix, m = graphgen.chunglu_weights(20_001, 2.05, 30.0)
        src, dst, n = *graphgen.chunglu_host(prefix, m, seed=3), 20_001
    else:
        i, j = np.triu_indices(1200, 1)
        src = np.concatenate([i, np.zeros(30_000, np.int64)]).astype(np.int32)
        dst = np.concatenate([j, np.arange(1200, 31_200)]).astype(np.int32)
        n = 31_200
    s, d = torch.as_tensor(src).cuda(), torch.as_tensor(dst).cuda()
    g = wedge.graph_build(s, d, n)
    dg, db = ctypes.c_void_p(), ctypes.c_void_p()
    _ok(lib, lib.wedge_graph_build(s.data_ptr(), d.data_ptr(), len(src), n, None, ctypes.byref(dg)))
    for tau, omega in ((1, 2), (2, 2), (100, 2), (1, 10**7)):
        b = wedge.bin(g, tau=tau, omega=omega)
        _ok(lib, lib.wedge_bin(dg, ctypes.byref(wedge.BinParams(tau, omega)), None, ctypes.byref(db)))
        for form, group, ranks, row in ((1, 1 << 27, 1 << 19, 8192), (1, 40_000, 900, 500), (1, 40_000, 0, 0), (2, 1, 0, 0)):
            t_i = torch.zeros(n, dtype=torch.int64, device="cuda")
            want = wedge.force_exact(g, b, t_i=t_i, form=form, group_edges=group, map_ranks=ranks, table_row=row)
            dt, out = torch.zeros_like(t_i), wedge.ExactCounts()
            _ok(lib, lib.wedge_test_exact(dg, db, dt.data_ptr(), None, form, group, ranks, row, ctypes.byref(out)))
            assert out.triangles == want["triangles"] and torch.equal(t_i, dt)
            assert np.array_equal(np.array([list(r) for r in out.pbq[:out.n_bins]], np.uint64), want["pbq"])
        c = wedge.CountsStruct()
        _ok(lib, lib.wedge_sample(dg, db, ctypes.byref(wedge.SampleParams(5, 0.0, 0.0, 3000, 5000, 0, None, None, 0)), None,
                                  ctypes.byref(c)))
        assert np.array_equal(wedge.Counts(c).counts_matrix(),
                              wedge.sample(g, b, seed=5, k_per_bin=3000, k_global=5000).counts_matrix())
        lib.wedge_bins_free(db)
        b.free()
    lib.wedge_graph_free(dg)
    g.free()
