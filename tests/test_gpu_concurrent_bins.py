"""wedge_bin from two threads at once, one with few bins and one with many: the
calls' launches need different amounts of shared memory, and neither may set the
other's limit."""
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
wedge = pytest.importorskip("paper_1301_5887_gb300")


def test_few_and_many_bins_at_once():
    import __graft_entry__
    __graft_entry__.build()
    wedge.load()
    n = 4096
    gen = torch.Generator("cuda").manual_seed(1)
    src, dst = (torch.randint(0, n, (400_000,), generator=gen, device="cuda", dtype=torch.int32) for _ in "sd")
    torch.cuda.synchronize()
    g = wedge.graph_build(src, dst, n)
    failed, sizes = [], {}

    def work(tau):
        stream = torch.cuda.Stream()
        try:
            for _ in range(400):
                b = wedge.bin(g, tau=tau, omega=2, stream=stream.cuda_stream)
                sizes.setdefault(tau, set()).add(tuple(b.info().n_b))
                b.free()
        except Exception as e:  # (reported below, in the test's own thread)
            failed.append((tau, str(e)))

    threads = [threading.Thread(target=work, args=(tau,)) for tau in (1, 100, 200, 48)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed and all(len(s) == 1 for s in sizes.values()) and len(sizes) == 4
