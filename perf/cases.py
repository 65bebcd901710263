"""The work that users of the wedge-sampling library have it do, as measurable cases.

A case is a dict of plain values; ``prepare`` makes what a program holds
before the call (edge lists or resident graphs, on the GPU or in pinned host
memory), ``run`` is one pass through the public entry points, ``work`` the
bytes that a pass cannot do without, ``exact`` the estimates of small cases in
64 bits by plain numpy. Graphs are the repository's own workloads: Graph500
Kronecker (2^scale vertices, ids permuted) and Chung-Lu power laws (any
number of vertices, exponent 2.0-2.6).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import graphgen
import paper_1301_5887_gb300 as wedge

K_EPS_002 = 950_114  # samples per bin and globally for eps = 0.002, delta = 0.001
DELTA = 0.001


def listed():
    return [
        # A small graph from edge list to estimates: launches, synchronisations and host work count.
        {"name": "path_kron_s12", "kind": "path", "graph": "kron", "scale": 12, "ef": 16, "host": False,
         "tau": 1, "omega": 2, "k_bin": 10_000, "k_global": 100_000},
        # The ordinary graph: 16.8 M edges at eps = 0.002 per bin and globally.
        {"name": "path_kron_s20", "kind": "path", "graph": "kron", "scale": 20, "ef": 16, "host": False,
         "tau": 1, "omega": 2, "k_bin": K_EPS_002, "k_global": K_EPS_002},
        # The headline workload: 4.29e9 edges, near the paper's largest synthetic graph.
        {"name": "path_kron_s28", "kind": "path", "graph": "kron", "scale": 28, "ef": 16, "host": False,
         "tau": 1, "omega": 2, "k_bin": K_EPS_002, "k_global": K_EPS_002},
        # The whole path on an edge list in pinned host memory (134 M edges, the paper's default bins).
        {"name": "path_host_s23", "kind": "path", "graph": "kron", "scale": 23, "ef": 16, "host": True,
         "tau": 2, "omega": 2, "k_bin": 100_000, "k_global": K_EPS_002},
        # A heavy-tailed graph with an odd number of vertices, built and its CSR taken out.
        {"name": "build_chunglu_3m", "kind": "build", "graph": "cl", "n": 3_000_017, "gamma": 2.1, "mean_deg": 27.0},
        # Binning a resident graph anew (the paper's default bins).
        {"name": "bin_kron_s24", "kind": "bin", "graph": "kron", "scale": 24, "ef": 16, "tau": 2, "omega": 2},
        # One sampling request on a resident graph, eps = 0.002 per bin and globally.
        {"name": "sample_kron_s24", "kind": "sample", "graph": "kron", "scale": 24, "ef": 16, "mode": "plain",
         "k_bin": K_EPS_002, "k_global": K_EPS_002},
        # Large per-bin budgets with the closure checks in sorted order (Phase 3b's join).
        {"name": "sample_sorted_s22", "kind": "sample", "graph": "kron", "scale": 22, "ef": 16, "mode": "sorted",
         "k_bin": 4_000_000, "k_global": 0},
        # The paper's sampled-triangle statistics (k = 5 M), every sample's record kept.
        {"name": "tristats_kron_s24", "kind": "tristats", "graph": "kron", "scale": 24, "ef": 16, "k": 5_000_000},
        # Exact counts with per-vertex triangles, to hold estimates against.
        {"name": "exact_kron_s20", "kind": "exact", "graph": "kron", "scale": 20, "ef": 16},
        # Many graphs and budgets in one persistent launch.
        {"name": "batch_64", "kind": "batch", "graphs": 64, "lo": 9, "hi": 18, "k_lo": 1_000, "k_hi": 400_000},
        # A burst of requests of three accuracies to the serving loop over resident graphs.
        {"name": "serve_48", "kind": "serve", "graphs": 8, "lo": 12, "hi": 20, "requests": 48},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, lo, hi):
    """A Kronecker graph of lo <= scale <= hi or a Chung-Lu graph of as many vertices."""
    if rng.random() < 0.5:
        return {"graph": "kron", "scale": rng.randint(lo, hi), "ef": rng.randint(4, 32)}
    return {"graph": "cl", "n": _log_uniform(rng, 1 << lo, 1 << min(hi, 22)), "gamma": round(rng.uniform(2.0, 2.6), 3),
            "mean_deg": round(rng.uniform(8.0, 64.0), 2)}


def draw(rng):
    kind = rng.choice(["path", "path", "path", "build", "build", "bin", "sample", "sample", "tristats", "exact",
                       "batch", "serve"])
    tau, omega = rng.choice([(1, 2), (1, 2), (2, 2), (1, 3), (3, 2)])
    if kind == "path":
        host = rng.random() < 0.3
        return {"kind": "path", **_draw_graph(rng, 8, 22 if host else 25), "host": host, "tau": tau, "omega": omega,
                "k_bin": _log_uniform(rng, 1_000, 1_000_000), "k_global": _log_uniform(rng, 1_000, 2_000_000)}
    if kind == "build":
        return {"kind": "build", **_draw_graph(rng, 8, 25)}
    if kind == "bin":
        return {"kind": "bin", **_draw_graph(rng, 10, 25), "tau": tau, "omega": omega}
    if kind == "sample":
        mode = rng.choice(["plain", "plain", "rounding", "sorted"])
        return {"kind": "sample", **_draw_graph(rng, 10, 24), "mode": mode,
                "k_bin": _log_uniform(rng, 1_000, 4_000_000),
                "k_global": _log_uniform(rng, 1_000, 4_000_000) if mode == "plain" else 0}
    if kind == "tristats":
        return {"kind": "tristats", **_draw_graph(rng, 10, 24), "k": _log_uniform(rng, 10_000, 10_000_000)}
    if kind == "exact":
        return {"kind": "exact", **_draw_graph(rng, 8, 20)}
    if kind == "batch":
        return {"kind": "batch", "graphs": rng.randint(2, 96), "lo": 8, "hi": rng.randint(12, 18),
                "k_lo": _log_uniform(rng, 100, 2_000), "k_hi": _log_uniform(rng, 20_000, 1_000_000)}
    return {"kind": "serve", "graphs": rng.randint(1, 12), "lo": 10, "hi": rng.randint(12, 20),
            "requests": rng.randint(4, 96)}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _n_vertices(case):
    return 1 << case["scale"] if case["graph"] == "kron" else case["n"]


def _edges(case, seed):
    """Device edge list (src, dst) of the case's graph."""
    stream = torch.cuda.current_stream().cuda_stream
    if case["graph"] == "kron":
        m = case["ef"] << case["scale"]
        src = torch.empty(m, dtype=torch.int32, device="cuda")
        dst = torch.empty(m, dtype=torch.int32, device="cuda")
        graphgen.kronecker_device(case["scale"], src.data_ptr(), dst.data_ptr(), m, stream, seed=seed)
        torch.cuda.current_stream().synchronize()  # the server reads uploads on a stream of its own
        return src, dst
    prefix, m = graphgen.chunglu_weights(case["n"], case["gamma"], case["mean_deg"])
    weights = torch.from_numpy(prefix.view(np.int64)).cuda()
    src = torch.empty(m, dtype=torch.int32, device="cuda")
    dst = torch.empty(m, dtype=torch.int32, device="cuda")
    graphgen.chunglu_device(weights.data_ptr(), case["n"], src.data_ptr(), dst.data_ptr(), m, seed, stream_ptr=stream)
    torch.cuda.current_stream().synchronize()  # the weights are freed here; as above
    return src, dst


def _resident(case, seed, tau=1, omega=2):
    graph = wedge.graph_build(*_edges(case, seed), _n_vertices(case))
    return graph, wedge.bin(graph, tau=tau, omega=omega)


def _mix(rng, lo, hi):
    """One graph of a mixed pool: Kronecker or Chung-Lu, 2^lo to 2^hi vertices."""
    if rng.random() < 0.5:
        return {"graph": "kron", "scale": int(rng.integers(lo, hi + 1)), "ef": 16}
    return {"graph": "cl", "n": int(2 ** rng.uniform(lo, hi)), "gamma": float(rng.uniform(2.0, 2.6)),
            "mean_deg": float(rng.uniform(8, 32))}


def prepare(case, seed):
    state = {"case": case, "seed": seed}
    kind = case["kind"]
    if kind in ("path", "build"):
        src, dst = _edges(case, seed)
        if case.get("host"):
            # pinned host arrays, as a loader that feeds a GPU keeps them
            pinned = torch.empty(2, src.numel(), dtype=torch.int32, pin_memory=True)
            pinned[0].copy_(src)
            pinned[1].copy_(dst)
            src, dst = pinned[0], pinned[1]
        state.update(src=src, dst=dst, n=_n_vertices(case))
        if kind == "build":
            state.update(off=torch.empty(state["n"] + 1, dtype=torch.int64, device="cuda"),
                         deg=torch.empty(state["n"], dtype=torch.int32, device="cuda"),
                         adj=torch.full((2 * src.numel(),), -1, dtype=torch.int32, device="cuda"))
    elif kind in ("bin", "sample", "tristats", "exact"):
        state["graph"], state["bins"] = _resident(case, seed, case.get("tau", 1), case.get("omega", 2))
        n = _n_vertices(case)
        if kind == "bin":  # room for every vertex; what a graph does not fill stays -1
            state.update(L=torch.full((n,), -1, dtype=torch.int32, device="cuda"),
                         W=torch.full((n + 1,), -1, dtype=torch.int64, device="cuda"))
        elif kind == "tristats":
            state["records"] = torch.empty(8 * case["k"], dtype=torch.int32, device="cuda")
        elif kind == "exact":
            state["t_i"] = torch.empty(n, dtype=torch.int64, device="cuda")
    else:
        rng = np.random.default_rng(seed)
        pool = [_mix(rng, case["lo"], case["hi"]) for _ in range(case["graphs"])]
        if kind == "batch":
            items = []
            for i, spec in enumerate(pool):
                graph, bins = _resident(spec, seed + i)
                budgets = 10 ** rng.uniform(math.log10(case["k_lo"]), math.log10(case["k_hi"]), bins.info().n_bins)
                items.append({"graph": graph, "bins": bins, "seed": seed + i, "k_bin": budgets.astype(np.uint64),
                              "k_global": int(case["k_hi"])})
            state["requests"] = wedge.Requests(items)
            # the launch shape that the repository's benchmark settles on for such mixes
            state["config"] = {"block_threads": 512, "samples_per_tile": 4096}
        else:
            server = wedge.Server(slots=2, max_batch_samples=4_000_000, gpu_filling_samples=4_000_000,
                                  launch={"block_threads": 512, "samples_per_tile": 4096})
            ids = [server.add_graph(*_edges(spec, seed + i), _n_vertices(spec)) for i, spec in enumerate(pool)]
            state.update(server=server,
                         asks=[(ids[int(rng.integers(len(ids)))], seed + i, float(rng.choice([0.01, 0.005, 0.002])))
                               for i in range(case["requests"])])
    return state


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _pad(rows):
    """The per-bin rows, with zeros up to 64 bins: as many for every graph."""
    out = np.zeros((64, *rows.shape[1:]), rows.dtype)
    out[:len(rows)] = rows
    return out


def _counts(c):
    return {"k_b": _pad(c.k_b), "q": _pad(c.q), "n_b": _pad(c.n_b), "p_b": _pad(c.p_b), "k_global": c.k_global,
            "closed_global": c.closed_global, "stats": c.stats}


def _estimates(e):
    bins = {k: _pad(np.array(e[k], np.float64)) for k in ("c_b", "t_b")}
    return {**bins, **{k: np.array(e[k], np.float64) for k in ("c_hat", "t_hat", "c_hat_global", "t_hat_global")}}


def run(state):
    case, seed, kind = state["case"], state["seed"], state["case"]["kind"]
    if kind == "path":
        graph = wedge.graph_build(state["src"], state["dst"], state["n"])
        bins = wedge.bin(graph, tau=case["tau"], omega=case["omega"])
        counts = wedge.sample(graph, bins, seed=seed, k_per_bin=case["k_bin"], k_global=case["k_global"])
        estimates = wedge.estimate(counts, DELTA)
        bins.free()
        graph.free()
        return {"counts": _counts(counts), "estimates": _estimates(estimates)}
    if kind == "build":
        graph = wedge.graph_build(state["src"], state["dst"], state["n"])
        graph.copy(state["off"], state["adj"], state["deg"])
        graph.free()
        return {"off": state["off"], "adj": state["adj"], "deg": state["deg"]}  # adj: -1 past the off[n] entries
    if kind == "bin":
        bins = wedge.bin(state["graph"], tau=case["tau"], omega=case["omega"])
        bins.copy(state["L"], state["W"])
        info = bins.info()
        n_b, p_b = np.array(info.n_b, np.int64), np.array(info.p_b, np.int64)
        bins.free()
        return {"L": state["L"], "W": state["W"], "n_b": n_b, "p_b": p_b}
    if kind == "sample":
        flags = {"plain": 0, "rounding": wedge.FLAG_ROUNDING | wedge.FLAG_NO_GLOBAL,
                 "sorted": wedge.FLAG_SORTED_CLOSURE | wedge.FLAG_NO_GLOBAL}[case["mode"]]
        counts = wedge.sample(state["graph"], state["bins"], seed=seed, k_per_bin=case["k_bin"],
                              k_global=case["k_global"], flags=flags)
        return {"counts": _counts(counts), "estimates": _estimates(wedge.estimate(counts, DELTA))}
    if kind == "tristats":
        out = wedge.triangle_stats(state["graph"], state["bins"], seed, case["k"], records=state["records"])
        return {**out, "records": state["records"]}
    if kind == "exact":
        out = wedge.exact(state["graph"], state["bins"], t_i=state["t_i"])
        return {**out, "p_b": _pad(out["p_b"]), "pbq": _pad(out["pbq"]), "t_i": state["t_i"]}
    if kind == "batch":
        all_counts = wedge.sample_batch(state["requests"], state["config"])
    else:
        tickets = [state["server"].submit(gid, seed=s, eps=eps, delta=DELTA) for gid, s, eps in state["asks"]]
        all_counts = [state["server"].wait(t)[0] for t in tickets]
    return {"k_b": np.stack([_pad(c.k_b) for c in all_counts]), "q": np.stack([_pad(c.q) for c in all_counts]),
            "closed_global": np.array([c.closed_global for c in all_counts]),
            "stats": np.stack([c.stats for c in all_counts])}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

#: A sample's random 32-byte sectors that no cache holds: centre, its offsets, two neighbours, their offsets and the
#: last steps of the two searches.
_SAMPLE_BYTES = 8 * 32


def _sizes(case):
    """Vertices and generated edges of a graph spec."""
    n = _n_vertices(case)
    return n, case["ef"] << case["scale"] if case["graph"] == "kron" else int(n * case["mean_deg"] / 2)


def _bins_used(m, n):
    """About the number of nonempty degree bins: powers of two up to the largest degree of a heavy-tailed graph."""
    return max(2, int(math.log2(max(4, 2 * m / n))) + int(math.log2(n) / 2))


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        mid = (case["lo"] + case["hi"]) / 2
        bins = _bins_used(16 * 2 ** mid, 2 ** mid)
        if kind == "batch":
            mean = (case["k_hi"] - case["k_lo"]) / math.log(case["k_hi"] / case["k_lo"])
            samples = case["graphs"] * (bins * mean + case["k_hi"])
        else:
            samples = case["requests"] * (bins + 1) * (38_005 + 152_019 + 950_114) / 3
        return {"bytes": samples * _SAMPLE_BYTES, "flops": 0}
    n, m = _sizes(case)
    csr = 8 * (n + 1) + 4 * 2 * m + 4 * n
    bins = _bins_used(m, n)
    if kind == "build":
        return {"bytes": 8 * m + csr, "flops": 0}
    if kind == "bin":
        return {"bytes": 4 * n + 12 * n, "flops": 0}
    if kind == "exact":
        return {"bytes": csr + 8 * n, "flops": 0}
    if kind == "tristats":
        return {"bytes": case["k"] * (_SAMPLE_BYTES + 32), "flops": 0}
    sampling = (case["k_bin"] * bins + case["k_global"]) * _SAMPLE_BYTES
    if kind == "sample":
        return {"bytes": sampling, "flops": 0}
    return {"bytes": 8 * m + csr + 16 * n + sampling, "flops": 0}


# ---------------------------------------------------------------------------
# The estimates of small graphs, in 64 bits by numpy
# ---------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al., SC 2011) on arrays of counters: four uint64 arrays of 32-bit words."""
    mask, s32 = np.uint64(0xFFFFFFFF), np.uint64(32)
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = ((p1 >> s32) ^ c1 ^ np.uint64(k0), p1 & mask, (p0 >> s32) ^ c3 ^ np.uint64(k1), p0 & mask)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1, c2, c3


def _mulhi(lo, hi, p):
    """floor((lo + 2^32 hi) p / 2^64) for 32-bit words lo, hi and 64-bit p."""
    mask, s32 = np.uint64(0xFFFFFFFF), np.uint64(32)
    pl, ph = p & mask, p >> s32
    mid = hi * pl + ((lo * pl) >> s32)
    return hi * ph + (mid >> s32) + (((mid & mask) + lo * ph) >> s32)


def _reference(src, dst, n, tau, omega, seed, k_bin, k_global):
    lo_, hi_ = np.minimum(src, dst).astype(np.int64), np.maximum(src, dst).astype(np.int64)
    edges = np.unique((lo_ * n + hi_)[lo_ != hi_])
    rows = np.sort(np.concatenate([edges, edges % n * n + edges // n]))  # x n + y, both directions
    adj, deg = rows % n, np.bincount(rows // n, minlength=n)
    off = np.concatenate([[0], np.cumsum(deg)])
    low = [0]
    while low[-1] <= deg.max():
        k = len(low)
        low.append(k if k <= tau else low[-1] + omega ** (k - 1 - tau))
    bin_of = np.searchsorted(np.array(low), deg, side="right") - 1
    n_bins = max(2, len(low) - 1)
    some = np.nonzero(deg >= 2)[0]
    order = some[np.argsort(bin_of[some], kind="stable")]
    prefix = np.concatenate([[0], np.cumsum(deg[order] * (deg[order] - 1) // 2)])
    start = np.concatenate([[0], np.cumsum(np.bincount(bin_of[some], minlength=n_bins))])
    p = np.diff(prefix[start])

    def closed(a, z, bin_id, tag, k):
        """Class (0 open) of k samples over order[a:z]."""
        s = np.arange(k, dtype=np.uint64)
        r = _philox(s, np.zeros_like(s), np.full_like(s, bin_id), np.full_like(s, tag), seed)
        t = _mulhi(r[0], r[1], np.uint64(prefix[z] - prefix[a])).astype(np.int64)
        v0 = order[np.searchsorted(prefix, prefix[a] + t, side="right") - 1]
        d = deg[v0]
        u = _mulhi(r[2], r[3], (d * (d - 1)).astype(np.uint64)).astype(np.int64)
        i, j = u // (d - 1), u % (d - 1)
        j += j >= i
        v1, v2 = adj[off[v0] + i], adj[off[v0] + j]
        at = np.searchsorted(rows, v1 * n + v2)
        shut = rows[np.minimum(at, len(rows) - 1)] == v1 * n + v2
        return np.where(shut, 1 + (bin_of[v1] == bin_id) + (bin_of[v2] == bin_id), 0)

    c_b, t_b = np.zeros(n_bins), np.zeros(n_bins)
    for b in range(2, n_bins):
        if p[b]:
            q = np.bincount(closed(start[b], start[b + 1], b, 0, k_bin), minlength=4)
            c_b[b] = q[1:].sum() / k_bin
            t_b[b] = float(p[b]) * (q[1] + q[2] / 2 + q[3] / 3) / k_bin
    total = float(prefix[-1])
    c_glob = np.count_nonzero(closed(0, len(order), 0, 1, k_global)) / k_global if k_global and total else 0.0
    c_hat = float((p / total * c_b).sum()) if total else 0.0
    return {"c_b": _pad(c_b), "t_b": _pad(t_b), "c_hat": np.array(c_hat), "t_hat": np.array(c_hat * total / 3),
            "c_hat_global": np.array(c_glob), "t_hat_global": np.array(c_glob * total / 3)}


def exact(case, seed):
    if case["kind"] not in ("path", "sample") or case.get("mode") == "rounding":
        return None
    n, m = _sizes(case)
    if m + 2 * (case["k_bin"] * _bins_used(m, n) + case["k_global"]) > 12_000_000:
        return None  # over about 20 seconds
    src, dst = (x.cpu().numpy() for x in _edges(case, seed))
    return {"counts": {k: None for k in ("k_b", "q", "n_b", "p_b", "k_global", "closed_global", "stats")},
            "estimates": _reference(src, dst, n, case.get("tau", 1), case.get("omega", 2), seed, case["k_bin"],
                                    case["k_global"])}
