"""The work that libeic's users have it do, as measurable cases.

Each case is one call (or one build, one batch, one burst of requests) through
the package's public entry points on synthetic graphs of the shapes of the
benchmark and the tests: uniform random graphs, RMAT (Kronecker) graphs with
several weight distributions, and road-like grids. Graphs are made on the GPU
with torch from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2506_19349_gb300 as eic

# Entries of the weight-sorted rows that a query has to look at, per vertex:
# the lower end of the 3.16-5.38 traversals per reachable vertex that the paper
# measures with its pruning (Section 4, nTrav).
TRAVERSED = 3


def listed():
    return [
        # One query on a small uniform graph (2^14 vertices, 2^17 edges): the
        # latency of the smallest real call.
        {"name": "urand14", "kind": "query", "graph": "urand", "n": 1 << 14, "edges": 1 << 17, "weights": "uniform",
         "wmax": 255},
        # The allocation-free entry point near its size limits, as called from
        # a loop that may not allocate.
        {"name": "noalloc17", "kind": "noalloc", "graph": "kron", "n": 131071, "edges": 16 * 131071,
         "weights": "uniform", "wmax": 255},
        # Wide weights (2^24: no ring of distances) and the shortest-path tree.
        {"name": "kron18_wide_parent", "kind": "query", "graph": "kron", "n": 250007, "edges": 16 * 250007,
         "weights": "uniform", "wmax": (1 << 24) - 1, "parent": True},
        # A mid-size query whose distances are wanted on the host: the result
        # goes to a page-locked array.
        {"name": "kron22_host", "kind": "query", "graph": "kron", "n": (1 << 22) - 3, "edges": 16 << 22,
         "weights": "uniform", "wmax": 255, "host": True},
        # The benchmark's graph: RMAT scale 25, edge factor 16.
        {"name": "kron25", "kind": "query", "graph": "kron", "n": 1 << 25, "edges": 16 << 25, "weights": "uniform",
         "wmax": 255},
        # Heavy-tailed weights on an RMAT graph of no round size.
        {"name": "kron24_lognormal", "kind": "query", "graph": "kron", "n": 15000001, "edges": 16 * 15000001,
         "weights": "lognormal", "wmax": 65535},
        # Road-like: many steps of few vertices, at the paper's step width.
        {"name": "grid4096", "kind": "query", "graph": "grid", "rows": 4096, "cols": 4096, "weights": "uniform",
         "wmax": 4095},
        # A ragged road-like grid at the step width that the tuners pick for
        # grids (exact for every width).
        {"name": "grid1531x977_wide_steps", "kind": "query", "graph": "grid", "rows": 1531, "cols": 977,
         "weights": "uniform", "wmax": 255, "gap_shift": 4},
        # A prepared batch of uneven graphs (RMAT 12..20, grids 256^2..1024^2),
        # 8 sources each, replayed: the batched benchmark's set but for its
        # largest graphs.
        {"name": "batch_set", "kind": "batch", "kron_min": 12, "kron_max": 20, "grid_min": 256, "grid_max": 1024,
         "grids": 6, "sources": 8, "wmax": 255},
        # A one-shot batch call: some sources on a few small graphs.
        {"name": "batch_call", "kind": "batch_call", "kron_min": 12, "kron_max": 16, "grid_min": 0, "grid_max": 0,
         "grids": 0, "sources": 10, "wmax": 255},
        # A burst of requests to a running server, results read back on the host.
        {"name": "serve_burst", "kind": "serve", "kron_min": 16, "kron_max": 20, "grid_min": 512, "grid_max": 512,
         "grids": 1, "sources": 6, "wmax": 255},
        # A new graph: its preprocessing from tuples on the GPU and a first query.
        {"name": "build_kron21", "kind": "build", "graph": "kron", "n": 2000003, "edges": 16 * 2000003,
         "weights": "uniform", "wmax": 255},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["query", "query", "query", "query", "noalloc", "build", "batch", "batch_call", "serve"])
    if kind in ("query", "noalloc", "build"):
        graph = rng.choice(["urand", "kron", "kron", "grid"])
        weights, wmax = rng.choice([("uniform", 255), ("uniform", 255), ("uniform", 4095), ("lognormal", 65535),
                                    ("uniform", (1 << 24) - 1)])
        if kind == "noalloc" and wmax > 65535:
            weights, wmax = "uniform", 65535
        c = {"kind": kind, "graph": graph, "weights": weights, "wmax": wmax}
        if graph == "grid":
            side = _log_int(rng, 64, {"query": 3200, "noalloc": 400, "build": 2000}[kind])
            c["rows"] = side
            c["cols"] = max(48, int(side * rng.uniform(0.7, 1.25)))
            if weights == "uniform" and wmax > 65535:
                c["wmax"] = 4095
            if kind == "query" and rng.random() < 0.5:
                c["gap_shift"] = rng.choice([2, 3, 4])
        else:
            hi = {"query": 1 << 24, "noalloc": 130000, "build": 1 << 21}[kind]
            c["n"] = _log_int(rng, 1 << 12, hi)
            c["edges"] = c["n"] * (8 if graph == "urand" else 16)
        if kind == "query" and c.get("n", 1 << 20) <= 1 << 22:
            if rng.random() < 0.3:
                c["parent"] = True
            if rng.random() < 0.3:
                c["host"] = True
        if kind == "build" and rng.random() < 0.4:
            c["host_tuples"] = True
        return c
    hi = rng.randint(14, {"batch": 20, "batch_call": 17, "serve": 20}[kind])
    grids = rng.randint(0, {"batch": 6, "batch_call": 2, "serve": 2}[kind])
    gmax = _log_int(rng, 64, {"batch": 1024, "batch_call": 256, "serve": 512}[kind]) if grids else 0
    return {"kind": kind, "kron_min": rng.randint(11, hi - 2), "kron_max": hi, "grid_min": gmax // 2,
            "grid_max": gmax, "grids": grids, "sources": rng.randint(3, 8 if kind != "serve" else 5),
            "wmax": rng.choice([255, 255, 4095])}


# ------------------------------------------------------------------- inputs

_CHUNK = 1 << 26


def _rmat(n, edges, g):
    """`edges` RMAT tuples (0.57, 0.19, 0.19, 0.05) over n vertices: drawn over
    the next power of two, folded into [0, n), ids permuted."""
    scale = max(1, (n - 1).bit_length())
    src = torch.empty(edges, dtype=torch.int32, device="cuda")
    dst = torch.empty(edges, dtype=torch.int32, device="cuda")
    perm = torch.randperm(n, generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    for at in range(0, edges, _CHUNK):
        k = min(_CHUNK, edges - at)
        a = torch.zeros(k, dtype=torch.int32, device="cuda")
        b = torch.zeros(k, dtype=torch.int32, device="cuda")
        for _ in range(scale):
            r = torch.rand(k, generator=g, device="cuda")
            down = r >= 0.76
            right = ((r >= 0.57) & ~down) | (r >= 0.95)
            a.mul_(2).add_(down)
            b.mul_(2).add_(right)
        src[at:at + k] = perm.index_select(0, a.remainder_(n))
        dst[at:at + k] = perm.index_select(0, b.remainder_(n))
    return src, dst


def _grid(rows, cols, g):
    """4-neighbour grid with 10% of the edges deleted and 2% diagonal shortcuts."""
    ids = torch.arange(rows * cols, dtype=torch.int32, device="cuda").view(rows, cols)
    src = torch.cat([ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)])
    dst = torch.cat([ids[:, 1:].reshape(-1), ids[1:].reshape(-1)])
    keep = torch.rand(src.numel(), generator=g, device="cuda") >= 0.10
    k = int(0.02 * src.numel())
    r = torch.randint(0, rows - 1, (k,), generator=g, device="cuda", dtype=torch.int32)
    c = torch.randint(0, cols - 1, (k,), generator=g, device="cuda", dtype=torch.int32)
    side = torch.randint(0, 2, (k,), generator=g, device="cuda", dtype=torch.int32)
    s = r * cols + c + side
    d = (r + 1) * cols + c + 1 - side
    return torch.cat([src[keep], s]), torch.cat([dst[keep], d])


def _weights(kind, wmax, count, g):
    w = torch.empty(count, dtype=torch.int32, device="cuda")
    for at in range(0, count, _CHUNK):
        k = min(_CHUNK, count - at)
        if kind == "lognormal":
            z = torch.randn(k, generator=g, device="cuda")
            w[at:at + k] = torch.exp(3.0 + 1.5 * z).round_().clamp_(1, wmax).to(torch.int32)
        else:
            w[at:at + k] = torch.randint(1, wmax + 1, (k,), generator=g, device="cuda", dtype=torch.int32)
    return w


def _tuples(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if case["graph"] == "grid":
        n = case["rows"] * case["cols"]
        src, dst = _grid(case["rows"], case["cols"], g)
    elif case["graph"] == "kron":
        n = case["n"]
        src, dst = _rmat(n, case["edges"], g)
    else:
        n = case["n"]
        src = torch.randint(0, n, (case["edges"],), generator=g, device="cuda", dtype=torch.int32)
        dst = torch.randint(0, n, (case["edges"],), generator=g, device="cuda", dtype=torch.int32)
    return n, src, dst, _weights(case["weights"], case["wmax"], src.numel(), g)


def _sources(n, src, dst, count, seed):
    """Uniform over the vertices with at least two tuples."""
    rng = np.random.RandomState(seed % (1 << 31))
    got = []
    while len(got) < count:
        v = int(rng.randint(0, n))
        if int((src == v).sum() + (dst == v).sum()) >= 2:
            got.append(v)
    return got


def _single(case):
    return case["kind"] in ("query", "noalloc", "build")


def _set(case):
    """The graphs of a batch or a server, as single cases."""
    wmax = case["wmax"]
    cs = [{"graph": "kron", "n": 1 << s, "edges": 16 << s, "weights": "uniform", "wmax": wmax}
          for s in range(case["kron_min"], case["kron_max"] + 1)]
    for i in range(case["grids"]):
        f = i / max(1, case["grids"] - 1)
        side = max(32, int(round(case["grid_min"] ** (1 - f) * case["grid_max"] ** f)))
        cs.append({"graph": "grid", "rows": side, "cols": side, "weights": "uniform", "wmax": wmax})
    return cs


def _arrivals(count):
    """The order in which a server's requests come in: the graphs mixed."""
    return np.random.RandomState(7).permutation(count)


def prepare(case, seed):
    kind = case["kind"]
    if _single(case):
        n, src, dst, w = _tuples(case, seed)
        st = {"case": case, "n": n, "source": _sources(n, src, dst, 1, seed)[0]}
        if kind == "build":
            st["tuples"] = [src, dst, w]
            if case.get("host_tuples"):
                st["tuples"] = [x.cpu().numpy().view(np.uint32) for x in (src, dst, w)]
        else:
            st["graph"] = eic.Graph(n, src, dst, w)
        host = bool(case.get("host"))
        st["dist"] = torch.empty(n, dtype=torch.int32, pin_memory=True) if host else eic.new_dist(n)
        if case.get("parent"):
            st["parent"] = torch.empty(n, dtype=torch.int32, pin_memory=True) if host else eic.new_dist(n)
        if case.get("gap_shift"):
            st["params"] = eic.default_params(gap_shift=case["gap_shift"])
        return st
    graphs, requests = [], []
    for i, c in enumerate(_set(case)):
        n, src, dst, w = _tuples(c, seed * 1009 + i)
        graphs.append(eic.Graph(n, src, dst, w))
        requests += [(i, s) for s in _sources(n, src, dst, case["sources"], seed * 1009 + i)]
    st = {"case": case, "graphs": graphs, "requests": requests}
    if kind == "serve":
        # a short idle time: the kernel leaves the GPU soon after the burst
        st["server"] = eic.Server(graphs, idle_us=200)
        st["requests"] = [requests[k] for k in _arrivals(len(requests))]
        return st
    flat = torch.empty(sum(graphs[i].n for i, _ in requests), dtype=torch.int32, device="cuda")
    dists, at = [], 0
    for i, _ in requests:
        dists.append(flat[at:at + graphs[i].n])
        at += graphs[i].n
    st["flat"] = flat
    st["args"] = ([graphs[i] for i, _ in requests], [s for _, s in requests], dists)
    if kind == "batch":
        st["batch"] = eic.Batch(*st["args"])
    return st


# --------------------------------------------------------------------- runs

def run(state):
    kind = state["case"]["kind"]
    if kind == "query":
        eic.sssp(state["graph"], state["source"], dist=state["dist"], parent=state.get("parent"),
                 params=state.get("params"))
        return [state["dist"], state["parent"]] if "parent" in state else [state["dist"]]
    if kind == "noalloc":
        status = eic.sssp_noalloc(state["graph"], state["source"], state["dist"])
        return [state["dist"], status]
    if kind == "build":
        g = eic.Graph(state["n"], *state["tuples"])
        eic.sssp(g, state["source"], dist=state["dist"])
        facts = [g.m, g.max_deg, g.max_w, g.min_w, g.highd0]
        g.close()
        return [state["dist"]] + facts
    if kind == "batch":
        state["batch"].run()
        return [state["flat"], state["batch"].wait()]
    if kind == "batch_call":
        return [state["flat"], eic.sssp_batch(*state["args"])]
    server = state["server"]
    tickets = [server.submit(i, s) for i, s in state["requests"]]
    out = []
    for (i, _), t in zip(state["requests"], tickets):
        server.wait(t)
        out.append(server.result(t, state["graphs"][i].n)[0])
        server.release(t)
    return out


# ------------------------------------------------------------------ figures

def _query_work(case):
    """One query: a row offset read and a distance written per vertex, and the
    (neighbour, weight) entries that the pruned search has to look at."""
    n = case["rows"] * case["cols"] if case["graph"] == "grid" else case["n"]
    m = int(1.82 * n) if case["graph"] == "grid" else case["edges"]
    entries = min(2 * m, TRAVERSED * n)
    return n, m, 8 * n + 8 * entries, entries


def work(case):
    if _single(case):
        n, m, b, entries = _query_work(case)
        if case.get("parent"):
            b += 4 * n
        if case["kind"] == "build":
            b += 12 * m + 2 * 8 * m + 4 * n  # tuples read, both directions and the offsets written
        return {"bytes": b, "flops": entries}
    b = f = 0
    for c in _set(case):
        _, _, qb, entries = _query_work(c)
        b += case["sources"] * qb
        f += case["sources"] * entries
    return {"bytes": b, "flops": f}


# ------------------------------------------------- the same in plain torch

_INF = 1 << 40


def _bellman_ford(n, src, dst, w, source):
    """Distances by repeated relaxation of every tuple, both ways, in int64."""
    a = torch.cat([src, dst]).to(torch.int64)
    b = torch.cat([dst, src]).to(torch.int64)
    ww = torch.cat([w, w]).to(torch.int64)
    d = torch.full((n,), _INF, dtype=torch.int64, device="cuda")
    d[source] = 0
    while True:
        new = d.clone()
        for _ in range(8):
            new.scatter_reduce_(0, b, new[a] + ww, "amin")
        new.clamp_(max=_INF)
        if torch.equal(new, d):
            return d, a, b, ww
        d = new


def _out(d):
    return torch.where(d >= _INF, torch.full_like(d, -1), d)


def _passes(c):
    """About how many relaxation passes the tuples need."""
    return 4 * (c["rows"] + c["cols"]) if c["graph"] == "grid" else 64


def _tuple_count(c):
    return 2 * c["rows"] * c["cols"] if c["graph"] == "grid" else c["edges"]


def exact(case, seed):
    cs = [case] if _single(case) else _set(case)
    per = 1 if _single(case) else case["sources"]
    if sum(per * _passes(c) * (_tuple_count(c) + 20000) for c in cs) > 2e10 or max(_tuple_count(c) for c in cs) > 1 << 27:
        return None
    if _single(case):
        n, src, dst, w = _tuples(case, seed)
        s = _sources(n, src, dst, 1, seed)[0]
        d, a, b, ww = _bellman_ford(n, src, dst, w, s)
        if case["kind"] == "query" and case.get("parent"):
            tight = (d[a] < _INF) & (d[a] + ww == d[b]) & (a != b)
            p = torch.full((n,), _INF, dtype=torch.int64, device="cuda")
            p.scatter_reduce_(0, b[tight], a[tight], "amin")
            p[s] = s
            return [_out(d), _out(p)]
        if case["kind"] == "noalloc":
            return [_out(d), 0]
        if case["kind"] == "build":
            return [_out(d), None, None, None, None, None]
        return [_out(d)]
    flat = []
    for i, c in enumerate(cs):
        n, src, dst, w = _tuples(c, seed * 1009 + i)
        for s in _sources(n, src, dst, per, seed * 1009 + i):
            flat.append(_out(_bellman_ford(n, src, dst, w, s)[0]))
    if case["kind"] == "serve":
        return [flat[k] for k in _arrivals(len(flat))]
    return [torch.cat(flat), np.zeros(len(flat), np.int32)]
