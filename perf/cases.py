"""The work that users of the library have it do, as measurable cases.

Each case is one call, or one short chain of calls, that a program makes
through the public entry points of ``paper_1411_4942_gb300``: answering an
estimate request on a resident graph, counting a graph held in host memory,
loading a graph and sampling it, sampling a resident graph, sampling until the
bars are narrow, a batch of graphs in one launch, a served burst of requests,
exact counting, and turning an edge list into a CSR graph.

Graphs are drawn on the GPU from a seed: R-MAT (edge factor and the
probabilities 0.57 / 0.19 / 0.19 / 0.05) and Chung-Lu graphs with power-law
weights, vertex ids permuted, rows sorted.  ``exact`` replays the method in
plain torch (64-bit integers and doubles).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1411_4942_gb300 import batch as psb
from paper_1411_4942_gb300 import pathsample as ps
from paper_1411_4942_gb300 import serve as pss

DELTA = 0.01


# ------------------------------------------------------------------- the cases

def listed():
    return [
        # one estimate request at the smallest served k on a small resident
        # graph: two launches, one read-back, latency only
        {"name": "request_5k", "kind": "request", "family": "chung_lu", "n": 5000, "mean": 20.0, "gamma": 2.5,
         "w_max": 500.0, "k": 1 << 14},
        # a small graph counted end to end from host memory (the 1% accuracy
        # configuration: n = 5,000, k = 10^6 of each sampler)
        {"name": "host_count_5k", "kind": "host_count", "family": "chung_lu", "n": 5000, "mean": 20.0, "gamma": 2.5,
         "w_max": 500.0, "k": 1_000_000},
        # a request for a graph that is not resident (a served graph of middle
        # size, after an eviction): load, prefixes, sampling, estimate
        {"name": "cold_request_150k", "kind": "cold_request", "family": "chung_lu", "n": 150_001, "mean": 20.0,
         "gamma": 2.4, "w_max": 1732.0, "k": 1 << 17},
        # the whole path on a graph in device memory, R-MAT scale 20
        {"name": "step_rmat20", "kind": "step", "family": "rmat", "scale": 20, "edge_factor": 16.0, "k3": 1 << 24,
         "kc": 1 << 24},
        # the same on the social-network-shaped graph of 3M vertices
        {"name": "step_social3m", "kind": "step", "family": "chung_lu", "n": 3_000_000, "mean": 78.0, "gamma": 2.1,
         "w_max": 33000.0, "k3": 1 << 27, "kc": 1 << 26},
        # more samples of a resident graph of 1M vertices, a ragged number
        {"name": "resident_1m", "kind": "resident", "family": "chung_lu", "n": 1_000_000, "mean": 20.0, "gamma": 2.3,
         "w_max": 4472.0, "k3": 3_000_017, "kc": 3_000_017},
        # sampling a resident graph until every bar is within 5%
        {"name": "adaptive_100k", "kind": "adaptive", "family": "chung_lu", "n": 100_000, "mean": 20.0, "gamma": 2.6,
         "w_max": 1414.0, "target": 0.05, "k0": 1 << 16, "k_max": 1 << 24},
        # many graphs of uneven size, each with its own k, in one launch
        {"name": "batch_96", "kind": "batch", "graphs": 96, "scale_lo": 10, "scale_hi": 17, "k_lo": 16, "k_hi": 22,
         "captured": True},
        # a burst of estimate requests on a pool of resident graphs
        {"name": "serve_burst_200", "kind": "serve", "graphs": 12, "n_lo": 10_000, "n_hi": 300_000, "requests": 200,
         "k_lo": 14, "k_hi": 20},
        # exact counts of the R-MAT scale 20 graph (ground truth for accuracy studies)
        {"name": "exact_rmat20", "kind": "exact", "family": "rmat", "scale": 20, "edge_factor": 16.0},
        # edge lists as they come (each draw once, repeats and self-loops in it)
        {"name": "ingest_rmat20", "kind": "ingest", "family": "rmat", "scale": 20, "edge_factor": 16.0},
        {"name": "ingest_40k", "kind": "ingest", "family": "chung_lu", "n": 4001, "mean": 20.0, "gamma": 2.5,
         "w_max": 400.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, n_lo, n_hi, mean_hi):
    if rng.random() < 0.4:
        scale = int(round(rng.uniform(math.log2(n_lo), min(20.0, math.log2(n_hi)))))
        return {"family": "rmat", "scale": scale, "edge_factor": round(rng.uniform(8.0, min(32.0, mean_hi / 2)), 2)}
    n = _log_int(rng, n_lo, n_hi)
    mean = round(math.exp(rng.uniform(math.log(8.0), math.log(mean_hi))), 2)
    return {"family": "chung_lu", "n": n, "mean": mean, "gamma": round(rng.uniform(2.1, 2.8), 3),
            "w_max": round(math.sqrt(mean * n), 1)}


def draw(rng):
    kind = rng.choice(["request", "host_count", "cold_request", "step", "step", "resident", "resident", "adaptive",
                       "batch", "serve", "exact", "ingest"])
    case = {"kind": kind}
    if kind == "request":
        case.update(_draw_graph(rng, 3000, 1_000_000, 32.0), k=_log_int(rng, 1 << 14, 1 << 22))
    elif kind == "host_count":
        case.update(_draw_graph(rng, 3000, 300_000, 32.0), k=_log_int(rng, 1 << 14, 1 << 20))
    elif kind == "cold_request":
        case.update(_draw_graph(rng, 10_000, 1_000_000, 32.0), k=_log_int(rng, 1 << 14, 1 << 20))
    elif kind == "step":
        case.update(_draw_graph(rng, 30_000, 3_000_000, 64.0), k3=_log_int(rng, 1 << 20, 1 << 26))
        case["kc"] = _log_int(rng, 1 << 20, 1 << 26)
    elif kind == "resident":
        case.update(_draw_graph(rng, 100_000, 3_000_000, 40.0), k3=_log_int(rng, 1 << 17, 1 << 25))
        case["kc"] = _log_int(rng, 1 << 17, 1 << 25)
    elif kind == "adaptive":
        case.update(_draw_graph(rng, 5000, 500_000, 24.0), target=round(rng.uniform(0.03, 0.1), 3),
                    k0=_log_int(rng, 1 << 14, 1 << 17), k_max=1 << 23)
    elif kind == "batch":
        case.update(graphs=rng.randrange(12, 97), scale_lo=10, scale_hi=rng.randrange(13, 18), k_lo=15, k_hi=21,
                    captured=rng.random() < 0.5)
    elif kind == "serve":
        case.update(graphs=rng.randrange(3, 13), n_lo=10_000, n_hi=_log_int(rng, 30_000, 300_000),
                    requests=rng.randrange(30, 201), k_lo=14, k_hi=20)
    elif kind == "exact":
        case.update(_draw_graph(rng, 2000, 300_000, 40.0))
    else:
        case.update(_draw_graph(rng, 2000, 800_000, 36.0))
    return case


# ------------------------------------------------------------------ the inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _size(case):
    """(vertices, drawn edges) of a case's graph."""
    if case["family"] == "rmat":
        return 1 << case["scale"], int(case["edge_factor"] * (1 << case["scale"]))
    return case["n"], int(case["mean"] * case["n"] / 2)


def _rmat_pairs(scale, edges, gen):
    u = torch.zeros(edges, dtype=torch.int64, device="cuda")
    v = torch.zeros(edges, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        x = torch.rand(edges, generator=gen, device="cuda")
        u = 2 * u + (x >= 0.76)
        v = 2 * v + (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
    return u, v


def _chung_lu_pairs(n, mean, gamma, w_max, edges, gen):
    """Both ends drawn in proportion to weights c (i + i0)^(-1 / (gamma - 1)),
    i0 such that the largest expected degree is w_max (by inverting the
    integral of the weights)."""
    a = 1.0 / (gamma - 1.0)

    def top(i0):
        return mean * n * i0 ** -a * (1.0 - a) / ((n + i0) ** (1.0 - a) - i0 ** (1.0 - a))

    lo, hi = 1e-6, float(n)
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if top(mid) > w_max else (lo, mid)
    i0 = 0.5 * (lo + hi)
    first, last = i0 ** (1.0 - a), (n + i0) ** (1.0 - a)

    def ends():
        x = torch.rand(edges, generator=gen, device="cuda", dtype=torch.float64)
        i = (first + x * (last - first)) ** (1.0 / (1.0 - a)) - i0
        return i.to(torch.int64).clamp_(0, n - 1)

    return ends(), ends()


def _pairs(case, gen):
    """The graph's drawn vertex pairs with permuted ids: repeats and
    self-loops as they fall."""
    n, edges = _size(case)
    if case["family"] == "rmat":
        u, v = _rmat_pairs(case["scale"], edges, gen)
    else:
        u, v = _chung_lu_pairs(n, case["mean"], case["gamma"], case["w_max"], edges, gen)
    perm = torch.randperm(n, generator=gen, device="cuda")
    return n, perm[u], perm[v]


def _csr(n, u, v):
    """Sorted CSR (int64 offsets, int32 columns) of the simple undirected graph."""
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    off = torch.searchsorted(key, torch.arange(n + 1, dtype=torch.int64, device="cuda") * n)
    return off, (key % n).to(torch.int32)


def _graph(case, gen):
    n, u, v = _pairs(case, gen)
    return _csr(n, u, v)


def _sample_seed(seed, i=0):
    return (int(seed) * 1_000_003 + 7919 * i + 11) & 0x7FFFFFFF


def _batch_specs(case, seed):
    rs = np.random.Generator(np.random.PCG64(int(seed)))
    graphs, requests = [], []
    for i in range(case["graphs"]):
        graphs.append({"family": "rmat", "scale": int(rs.integers(case["scale_lo"], case["scale_hi"] + 1)),
                       "edge_factor": float(rs.integers(8, 33))})
        k = 1 << int(rs.integers(case["k_lo"], case["k_hi"] + 1))
        requests += [(i, 0, k, _sample_seed(seed, i)), (i, 1, k, _sample_seed(seed, i))]
    return graphs, requests


def _serve_specs(case, seed):
    rs = np.random.Generator(np.random.PCG64(int(seed)))
    graphs, requests = {}, []
    for i in range(case["graphs"]):
        n = int(round(math.exp(rs.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        graphs[f"g{i}"] = {"family": "chung_lu", "n": n, "mean": 20.0, "gamma": float(rs.uniform(2.1, 2.8)),
                           "w_max": math.sqrt(20.0 * n)}
    for i in range(case["requests"]):
        requests.append((f"g{int(rs.integers(0, case['graphs']))}", 1 << int(rs.integers(case["k_lo"], case["k_hi"] + 1)),
                         int(rs.integers(1, 2 ** 62))))
    return graphs, requests


def prepare(case, seed):
    kind = case["kind"]
    gen = _generator(seed)
    st = {"kind": kind, "case": case, "seed": _sample_seed(seed)}
    if kind in ("request", "resident", "adaptive", "exact"):
        off, col = _graph(case, gen)
        st["graph"] = ps.Graph(off, col)
        if kind == "exact":
            # the program's own array for the triangles per edge
            st["te"] = torch.zeros(_size(case)[1], dtype=torch.int32, device="cuda")
    elif kind in ("cold_request", "step"):
        st["off"], st["col"] = _graph(case, gen)
    elif kind == "ingest":
        n, u, v = _pairs(case, gen)
        st["n"], st["src"], st["dst"] = n, u.to(torch.int32), v.to(torch.int32)
        st["ws"] = torch.empty(ps.ps_ingest_workspace_bytes(n, u.numel()), dtype=torch.uint8, device="cuda")
        st["off"] = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        st["col"] = torch.zeros(2 * u.numel(), dtype=torch.int32, device="cuda")
    elif kind == "host_count":
        off, col = _graph(case, gen)
        st["off"], st["col"] = off.cpu().pin_memory(), col.cpu().pin_memory()
        n, nnz = off.numel() - 1, col.numel()
        nbytes = ps.ps_end_to_end_workspace_bytes(n, nnz) + ps.ps_ordered_scratch_bytes(case["k"])
        st["ws"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    elif kind == "batch":
        graphs, requests = _batch_specs(case, seed)
        st["set"] = psb.GraphSet([ps.Graph(*_graph(g, gen)) for g in graphs])
        st["runner"] = psb.BatchRunner(st["set"], [psb.Request(*r) for r in requests],
                                       psb.LaunchConfig(block_size=512, chunk=1 << 12))
        if case["captured"]:
            st["runner"].capture()
    elif kind == "serve":
        graphs, requests = _serve_specs(case, seed)
        sources = {}
        for key, g in graphs.items():
            off, col = _graph(g, gen)
            sources[key] = (off.cpu().numpy(), col.cpu().numpy())
        pool = pss.GraphPool(sources, budget_bytes=40 << 30)
        for key in sources:
            pool.acquire(key)
            pool.release(key)
        st["server"] = pss.Server(pool)
        st["requests"] = [pss.EstimateRequest(i, g, k, s) for i, (g, k, s) in enumerate(requests)]
    if kind == "step":
        n, nnz = st["off"].numel() - 1, st["col"].numel()
        st["ws"] = torch.empty(ps.ps_graph_workspace_bytes(n, nnz), dtype=torch.uint8, device="cuda")
        chunk = min(max(case["k3"], case["kc"]), 1 << 27)
        st["scratch"] = torch.empty(ps.ps_ordered_scratch_bytes(chunk), dtype=torch.uint8, device="cuda")
        st["hist"] = torch.zeros(16, dtype=torch.int64, device="cuda")
    return st


# -------------------------------------------------------------------- the pass

OK_OR_EMPTY = (ps.PS_OK, ps.PS_NO_PATHS)


def _totals(s):
    return [int(s.W), int(s.Lambda), s.N1, int(s.m), int(s.d_max)]


def _run_step(st):
    """The benchmark's step: load, prefixes, both samplers in draw order,
    read-back, estimates, in buffers that the program keeps."""
    case, seed, hist, scratch, ws = st["case"], st["seed"], st["hist"], st["scratch"], st["ws"]
    off, col = st["off"], st["col"]
    rc, h = ps.ps_load_csr(off.numel() - 1, col.numel(), off.data_ptr(), col.data_ptr(), ws.data_ptr(), ws.numel())
    ps._check(rc, "ps_load_csr")
    try:
        rc, stats = ps.ps_tau_prefix(h)
        ps._check(rc, "ps_tau_prefix", OK_OR_EMPTY)
        hist.zero_()
        rc = ps.ps_sample_3paths_ordered(h, case["k3"], seed, 0, hist.data_ptr(), scratch.data_ptr(), scratch.numel())
        ps._check(rc, "ps_sample_3paths_ordered", OK_OR_EMPTY)
        rc = ps.ps_sample_centered_ordered(h, case["kc"], seed, 0, hist.data_ptr() + 64, scratch.data_ptr(),
                                           scratch.numel())
        ps._check(rc, "ps_sample_centered_ordered", OK_OR_EMPTY)
        host = hist.cpu().numpy()
    finally:
        ps.ps_graph_free(h)
    rc, est, lo, hi = ps.ps_estimate(stats, host[:6], case["k3"], host[8:12], case["kc"], DELTA)
    ps._check(rc, "ps_estimate", OK_OR_EMPTY)
    return [host[:6], host[8:12], _totals(stats), est, lo, hi]


def run(st):
    kind, case, seed = st["kind"], st["case"], st["seed"]
    if kind == "request":
        G, k = st["graph"], case["k"]
        h6, h4 = G.sample_3paths(k, seed), G.sample_centered(k, seed)
        est, lo, hi = G.estimate(h6, k, h4, k, DELTA)
        return [h6[:6], h4[:4], est, lo, hi]
    if kind == "resident":
        G = st["graph"]
        return [G.sample_3paths_ordered(case["k3"], seed)[:6], G.sample_centered_ordered(case["kc"], seed)[:4]]
    if kind == "adaptive":
        k, h6, h4, est, lo, hi = st["graph"].count_adaptive(seed, case["target"], DELTA, case["k0"], case["k_max"])
        return [k, h6.astype(np.int64), h4.astype(np.int64), est, lo, hi]
    if kind == "exact":
        N, C, te = st["graph"].count_exact()
        st["te"][:te.numel()].copy_(te)
        return [N.astype(np.int64), C, st["te"]]
    if kind == "cold_request":
        G, k = ps.Graph(st["off"], st["col"]), case["k"]
        h6, h4 = G.sample_3paths(k, seed), G.sample_centered(k, seed)
        est, lo, hi = G.estimate(h6, k, h4, k, DELTA)
        totals = _totals(G.stats)
        G.close()
        return [h6[:6], h4[:4], totals, est, lo, hi]
    if kind == "step":
        return _run_step(st)
    if kind == "host_count":
        rc, est, lo, hi, h6, h4, stats = ps.ps_count_motifs_host(
            st["off"].numpy(), st["col"].numpy(), case["k"], case["k"], seed, DELTA, st["ws"].data_ptr(),
            st["ws"].numel())
        ps._check(rc, "ps_count_motifs_host", OK_OR_EMPTY)
        return [h6.astype(np.int64), h4.astype(np.int64), _totals(stats), est, lo, hi]
    if kind == "batch":
        if case["captured"]:
            st["runner"].replay()
        else:
            st["runner"].launch()
        return [st["runner"].d_hist]
    if kind == "serve":
        results, _ = st["server"].run(st["requests"], realtime=False)
        results.sort(key=lambda r: r.rid)
        return [np.stack([getattr(r, f) for r in results]).astype(t)
                for f, t in (("hist6", np.int64), ("hist4", np.int64), ("est", np.float64), ("lo", np.float64),
                             ("hi", np.float64))]
    rc, nnz = ps.ps_csr_from_edges(st["n"], st["src"].numel(), st["src"].data_ptr(), st["dst"].data_ptr(),
                                   st["ws"].data_ptr(), st["ws"].numel(), st["off"].data_ptr(), st["col"].data_ptr())
    ps._check(rc, "ps_csr_from_edges")
    return [nnz, st["off"], st["col"]]


# -------------------------------------------------------------------- the work

def _sampling_bytes(k3, kc, n, m):
    """Per sample one 32-byte sector per random access of the method (9 for a
    3-path, 7 for a centred one), but no more than every array read once: 32 B
    of edge record, 8 B of prefix and 8 B of adjacency per edge and sampler."""
    graph = 48 * m + 8 * n
    return min(288 * k3, graph) + min(224 * kc, graph)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        graphs, requests = _batch_specs(case, 1)
        total = 0
        for i, g in enumerate(graphs):
            n, m = _size(g)
            k = requests[2 * i][2]
            total += _sampling_bytes(k, k, n, m)
        return {"bytes": total, "flops": 0}
    if kind == "serve":
        graphs, requests = _serve_specs(case, 1)
        return {"bytes": sum(_sampling_bytes(k, k, *_size(graphs[g])) for g, k, _ in requests), "flops": 0}
    n, m = _size(case)
    # CSR in; canonical CSR, 32-byte records, two prefixes and 8 B of
    # adjacency structure per edge out
    load = 8 * n + 8 * m + 8 * n + 8 * m + 32 * m + 16 * m + 8 * m
    if kind in ("request", "host_count", "cold_request"):
        sampling = _sampling_bytes(case["k"], case["k"], n, m)
        return {"bytes": sampling + (0 if kind == "request" else load), "flops": 0}
    if kind in ("step", "resident"):
        sampling = _sampling_bytes(case["k3"], case["kc"], n, m)
        return {"bytes": sampling + (load if kind == "step" else 0), "flops": 0}
    if kind == "adaptive":
        return {"bytes": _sampling_bytes(case["k0"], case["k0"], n, m), "flops": 0}
    if kind == "exact":
        return {"bytes": 8 * n + 8 * m + 4 * m, "flops": 0}
    return {"bytes": 8 * m + 8 * n + 8 * m, "flops": 0}


# ------------------------------------------- the method in plain 64-bit torch

M32 = 0xFFFFFFFF


def _mul32(x, c):
    """(high, low) 32-bit halves of x * c, x and c in [0, 2^32) (x a tensor)."""
    lo = x & 0xFFFF
    hi = x >> 16
    return (c * hi + ((c * lo) >> 16)) >> 16, (x * c) & M32


def _philox(seed, ids, t, stream):
    """Philox4x32-10 (Salmon et al., SC'11), counter (id, t, stream), key seed."""
    c0, c1 = ids & M32, (ids >> 32) & M32
    c2, c3 = torch.full_like(ids, t), torch.full_like(ids, stream)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for i in range(10):
        if i:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        h0, l0 = _mul32(c0, 0xD2511F53)
        h1, l1 = _mul32(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
    return c0, c1, c2, c3


def _bounded64(x0, x1, s):
    """Lemire's bounded draw from the 64-bit word (x1, x0), s < 2^63: the
    value and whether it is accepted."""
    s0, s1 = s & M32, s >> 32
    ah, al = _mul32(x0, s0)
    bh, bl = _mul32(x1, s0)
    ch, cl = _mul32(x0, s1)
    dh, dl = _mul32(x1, s1)
    mid = ah + bl + cl
    top = (mid >> 32) + bh + ch + dl + (dh << 32)
    thr = (1 << 64) % s
    l1, l0 = mid & M32, al
    t1, t0 = thr >> 32, thr & M32
    return top, (l1 > t1) | ((l1 == t1) & (l0 >= t0))


def _bounded32(x, s):
    h, low = _mul32(x, s)
    return h, low >= (1 << 32) % s.clamp(min=1)


def _draws(seed, ids, stream, total):
    """The edge draw r of each id and its two neighbour words."""
    w0, w1, w2, w3 = _philox(seed, ids, 0, stream)
    r, ok = _bounded64(w0, w1, total)
    t = 0
    while not bool(ok.all()):
        t += 1
        bad = (~ok).nonzero().squeeze(1)
        a, b, _, _ = _philox(seed, ids[bad], t, stream)
        r[bad], ok[bad] = _bounded64(a, b, total)
    return r, w2, w3


def _small_draw(seed, ids, stream, slot, word, s):
    v, ok = _bounded32(word, s)
    t = 0
    while not bool(ok.all()):
        t += 1
        bad = (~ok).nonzero().squeeze(1)
        v[bad], ok[bad] = _bounded32(_philox(seed, ids[bad], t, stream)[slot], s[bad])
    return v


class _Plain:
    """The degree-ordered graph, its edges, weights and prefixes."""

    def __init__(self, off, col):
        n = off.numel() - 1
        deg = off[1:] - off[:-1]
        order = torch.sort(deg, stable=True).indices
        rank = torch.empty_like(order)
        rank[order] = torch.arange(n, device="cuda")
        src = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
        self.key = torch.sort(rank[src] * n + rank[col.to(torch.int64)]).values
        self.n, self.d = n, deg[order]
        self.off = torch.cat([self.d.new_zeros(1), torch.cumsum(self.d, 0)])
        row = torch.div(self.key, n, rounding_mode="floor")
        self.col = self.key - row * n
        up = (row < self.col).nonzero().squeeze(1)
        self.u, self.v = row[up], self.col[up]
        self.iu = up - self.off[self.u]
        self.jv = torch.searchsorted(self.key, self.v * n + self.u) - self.off[self.v]
        du, dv = self.d[self.u], self.d[self.v]
        self.ptau = torch.cumsum((du - 1) * (dv - 1), 0)
        self.plam = torch.cumsum((du - 1 - self.iu) * (dv - 1 - self.jv), 0)
        m = self.u.numel()
        self.W = int(self.ptau[-1]) if m else 0
        self.Lambda = int(self.plam[-1]) if m else 0
        d = [int(x) for x in torch.unique(self.d)]
        c = torch.unique(self.d, return_counts=True)[1].tolist()
        self.N1 = sum(k * (x * (x - 1) * (x - 2) // 6) for x, k in zip(d, c))
        self.totals = [self.W, self.Lambda, self.N1, m, max(d)]

    def edge(self, x, y):
        q = x * self.n + y
        i = torch.searchsorted(self.key, q).clamp_(max=self.key.numel() - 1)
        return self.key[i] == q

    def hist6(self, k, seed, first=0, chunk=1 << 23):
        h = torch.zeros(6, dtype=torch.int64, device="cuda")
        for lo in range(first, first + (k if self.W else 0), chunk):
            ids = torch.arange(lo, min(first + k, lo + chunk), device="cuda")
            r, w2, w3 = _draws(seed, ids, 0, self.W)
            j = torch.searchsorted(self.ptau, r, right=True)
            u, v = self.u[j], self.v[j]
            du, dv = self.d[u], self.d[v]
            a = _small_draw(seed, ids, 0, 2, w2, du - 1)
            b = _small_draw(seed, ids, 0, 3, w3, dv - 1)
            x = self.col[self.off[u] + torch.where(a == self.iu[j], du - 1, a)]
            y = self.col[self.off[v] + torch.where(b == self.jv[j], dv - 1, b)]
            e1, e2, e3 = self.edge(x, v), self.edge(u, y), self.edge(x, y)
            s = e1.long() + e2.long() + e3.long()
            cls = torch.tensor([1, 2, 4, 5], device="cuda")[s] + ((s == 1) & e3)
            h += torch.bincount(torch.where(x == y, 0, cls), minlength=6)
        return h.cpu().numpy()

    def hist4(self, k, seed, first=0, chunk=1 << 23):
        h = torch.zeros(4, dtype=torch.int64, device="cuda")
        for lo in range(first, first + (k if self.Lambda else 0), chunk):
            ids = torch.arange(lo, min(first + k, lo + chunk), device="cuda")
            r, w2, w3 = _draws(seed, ids, 1, self.Lambda)
            j = torch.searchsorted(self.plam, r, right=True)
            u, v = self.u[j], self.v[j]
            a = _small_draw(seed, ids, 1, 2, w2, self.d[u] - 1 - self.iu[j])
            b = _small_draw(seed, ids, 1, 3, w3, self.d[v] - 1 - self.jv[j])
            x = self.col[self.off[u] + self.iu[j] + 1 + a]
            y = self.col[self.off[v] + self.jv[j] + 1 + b]
            cls = 1 + self.edge(x, v).long() + self.edge(u, y).long()
            h += torch.bincount(torch.where(self.edge(x, y), cls, 0), minlength=4)
        return h.cpu().numpy()

    def bars(self, h6, k3, h4, kc, delta=DELTA):
        return _bars(self.W, self.Lambda, self.N1, h6, k3, h4, kc, delta)


def _kl(a, b):
    x = a * math.log(a / b) if a > 0 else 0.0
    return x + ((1 - a) * math.log((1 - a) / (1 - b)) if a < 1 else 0.0)


def _bar(count, k, delta):
    """The roots p of exp(-k D(count / k, p)) = delta on both sides."""
    if count == 0:
        return 0.0, 1.0 - delta ** (1.0 / k)
    if count == k:
        return delta ** (1.0 / k), 1.0
    alpha, target, ends = count / k, math.log(1.0 / delta) / k, []
    for far in (0.0, 1.0):
        near, out = alpha, far
        for _ in range(200):
            mid = 0.5 * (near + out)
            if mid == near or mid == out:
                break
            near, out = (near, mid) if _kl(alpha, mid) > target else (mid, out)
        ends.append(0.5 * (near + out))
    return ends[0], ends[1]


def _bars(W, Lambda, N1, h6, k3, h4, kc, delta):
    per3, perc = {2: 1, 3: 2, 4: 4, 5: 6, 6: 12}, {4: 1, 5: 1, 6: 3}
    c, lo, hi = [0.0] * 7, [0.0] * 7, [0.0] * 7
    for i, a in per3.items():
        if W:
            x = int(h6[i - 1])
            c[i] = x * W / k3 / a
            lo[i], hi[i] = (p * (W / a) for p in _bar(x, k3, delta))
    c1 = float(N1) - c[3] - 2 * c[5] - 4 * c[6]
    below = (c[3] - lo[3]) + 2 * (c[5] - lo[5]) + 4 * (c[6] - lo[6])
    above = (hi[3] - c[3]) + 2 * (hi[5] - c[5]) + 4 * (hi[6] - c[6])
    for i, b in perc.items():
        c[i] = lo[i] = hi[i] = 0.0
        if Lambda:
            x = int(h4[i - 3])
            c[i] = x * Lambda / kc / b
            lo[i], hi[i] = (p * (Lambda / b) for p in _bar(x, kc, delta))
    c[1], lo[1], hi[1] = c1, c1 - above, c1 + below
    return [np.array(z[1:]) for z in (c, lo, hi)]


def _exact_adaptive(g, case, seed):
    looks, k = 1, case["k0"]
    while k < case["k_max"]:
        k = min(2 * k, case["k_max"])
        looks += 1
    h6, h4, done, k = np.zeros(6, np.int64), np.zeros(4, np.int64), 0, case["k0"]
    while True:
        h6 = h6 + g.hist6(k - done, seed, done)
        h4 = h4 + g.hist4(k - done, seed, done)
        done = k
        est, lo, hi = g.bars(h6, k, h4, k, DELTA / looks)
        half = np.maximum(hi - est, est - lo)
        if (half <= case["target"] * np.abs(est)).all() or k == case["k_max"] or not (g.W and g.Lambda):
            return [done, h6, h4, est, lo, hi]
        k = min(2 * k, case["k_max"])


def exact(case, seed):
    kind, gen, s = case["kind"], _generator(seed), _sample_seed(seed)
    if kind == "exact":
        return None  # the enumeration's wedges: minutes in plain torch
    if kind == "ingest":
        n, u, v = _pairs(case, gen)
        off, col = _csr(n, u, v)
        return [col.numel(), off, torch.cat([col, col.new_zeros(2 * u.numel() - col.numel())])]
    if kind == "batch":
        graphs, requests = _batch_specs(case, seed)
        out = np.zeros((len(requests), 6), np.int64)
        for i, spec in enumerate(graphs):
            g = _Plain(*_graph(spec, gen))
            k, sd = requests[2 * i][2:]
            out[2 * i], out[2 * i + 1, :4] = g.hist6(k, sd), g.hist4(k, sd)
        return [torch.from_numpy(out.reshape(-1))]
    if kind == "serve":
        graphs, requests = _serve_specs(case, seed)
        plain = {key: _Plain(*_graph(spec, gen)) for key, spec in graphs.items()}
        rows = []
        for key, k, sd in requests:
            h6, h4 = plain[key].hist6(k, sd), plain[key].hist4(k, sd)
            rows.append([h6, h4, *plain[key].bars(h6, k, h4, k)])
        return [np.stack(x) for x in zip(*rows)]
    g = _Plain(*_graph(case, gen))
    if kind == "adaptive":
        return _exact_adaptive(g, case, s)
    k3, kc = case.get("k3", case.get("k")), case.get("kc", case.get("k"))
    h6, h4 = g.hist6(k3, s), g.hist4(kc, s)
    if kind == "resident":
        return [torch.from_numpy(h6), torch.from_numpy(h4)]
    est, lo, hi = g.bars(h6, k3, h4, kc)
    if kind == "request":
        return [torch.from_numpy(h6), torch.from_numpy(h4), est, lo, hi]
    return [h6, h4, g.totals, est, lo, hi]
