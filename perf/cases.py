"""Performance cases: the calls a program makes of this library, over the sizes
and options it is used with.

A case names a graph family with its sizes, the weights, the options of the
graph handle and the entry point.  prepare() builds the graph from the seed
(on the GPU, then copied to the host arrays that sssp_create takes) and keeps
what a program would keep: handles, servers and output buffers.  run() is one
call.  Distances of unreachable vertices are SSSP_DIST_INF, -1 as int64.
"""
from __future__ import annotations

import math
import random
import weakref

import numpy as np
import torch

import paper_1812_10499_gb300 as sssp


def listed():
    return [
        # The smallest call: one query on a graph of a few thousand vertices,
        # distances left on the device (26 dependent rounds, all latency).
        dict(name="random4096", kind="random", n=4096, dmin=8, dmax=8, wmax=100,
             rule="threshold", layout="auto", entry="device"),
        # An ordinary query on a skewed graph, distances into page-locked host memory.
        dict(name="rmat20-host", kind="rmat", scale=20, factor=16, wmax=255,
             rule="cheap", layout="auto", entry="host"),
        # The headline workload: R-MAT scale 22, the cheaper fixing rules first.
        dict(name="rmat22", kind="rmat", scale=22, factor=16, wmax=255,
             rule="cheap", layout="auto", entry="device"),
        # Every output (distances, parents, fixing rounds, lower bounds, counters)
        # to the host, with the 32-byte records of graphs with large weights.
        dict(name="rmat18-all-wide", kind="rmat", scale=18, factor=16, wmax=1000000,
             rule="threshold", layout="wide", entry="all"),
        # A road-like network: thousands of rounds with a thin wave front.
        dict(name="grid1024", kind="grid", rows=1024, cols=1024, wmax=10000,
             rule="threshold", layout="auto", entry="device"),
        # The unweighted variant, on a ragged grid.
        dict(name="unitgrid2001x1500", kind="grid", rows=2001, cols=1500, wmax=1,
             rule="threshold", layout="auto", entry="device"),
        # Road-like with the windowed relaxation, the option made for such graphs.
        dict(name="grid-windowed", kind="grid", rows=700, cols=1300, wmax=10000,
             rule="windowed", layout="auto", entry="device"),
        # A layered DAG: hundreds of rounds of middling size; n * max weight
        # needs the 32-byte records.
        dict(name="dag512x8192", kind="dag", layers=512, width=8192, deg=8, skip=4, wmax=1000,
             rule="threshold", layout="auto", entry="device"),
        # Batched: independent graphs of uneven size solved in one call.
        dict(name="batch128", kind="batch", count=128, nmin=1024, nmax=262144, wmax=1000,
             rule="threshold", layout="auto", entry="device"),
        # Batched: many sources on one skewed graph.
        dict(name="sources64-rmat18", kind="sources", scale=18, factor=16, count=64, wmax=255,
             rule="threshold", layout="auto", entry="device"),
        # Served: a burst of queries of different sizes through the query server,
        # a tenth of them on a larger skewed graph.
        dict(name="serve96", kind="serve", graphs=16, nmin=1024, nmax=131072, scale=17,
             queries=96, wmax=1000, rule="threshold", layout="auto", entry="host"),
        # One-off use: build the graph from host arrays, one query, release it.
        dict(name="oneshot-rmat18", kind="rmat", scale=18, factor=16, wmax=255,
             rule="threshold", layout="auto", entry="oneshot"),
    ]


def draw(rng):
    """One more case of the listed ones' ranges."""
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["random", "rmat", "grid", "dag", "batch", "sources", "serve"])
    c = dict(kind=kind, wmax=rng.choice([100, 255, 1000, 10000]), rule="threshold",
             layout="auto", entry="device")
    if kind in ("random", "rmat", "dag"):
        c["rule"] = rng.choice(["threshold", "cheap"])
        c["layout"] = rng.choice(["auto", "auto", "wide"])
        c["entry"] = rng.choice(["device", "host", "all"])
    if kind == "random":
        dmin = rng.randint(2, 8)
        c.update(n=logint(1000, 300000), dmin=dmin, dmax=dmin + rng.randint(0, 8))
        c["entry"] = rng.choice(["device", "host", "all", "oneshot"])
    elif kind == "rmat":
        c.update(scale=rng.randint(13, 21), factor=rng.randint(6, 16))
        if c["scale"] <= 18:
            c["entry"] = rng.choice(["device", "host", "all", "oneshot"])
    elif kind == "grid":
        c.update(rows=logint(60, 1000), cols=logint(60, 1000), wmax=rng.choice([1, 100, 10000]))
        c["rule"] = rng.choice(["threshold", "windowed"]) if c["wmax"] > 1 else "threshold"
    elif kind == "dag":
        c.update(layers=logint(16, 500), width=logint(300, 8000), deg=rng.randint(4, 8),
                 skip=rng.randint(1, 4))
    elif kind == "batch":
        nmin = logint(300, 5000)
        c.update(count=logint(4, 128), nmin=nmin, nmax=logint(2 * nmin, 200000))
    elif kind == "sources":
        c.update(scale=rng.randint(12, 18), factor=rng.randint(6, 16), count=logint(3, 64))
    else:
        nmin = logint(300, 5000)
        c.update(graphs=rng.randint(3, 16), nmin=nmin, nmax=logint(2 * nmin, 100000),
                 scale=rng.randint(12, 16), queries=logint(8, 96))
    return c


# ------------------------------------------------------------------- graphs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, lo, hi, n):
    """n integers in [lo, hi)."""
    return torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=torch.int64)


def _csr(n, src_sorted, col, w):
    ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(src_sorted, minlength=n), 0)
    return n, ptr, src_sorted, col, w


def _random(n, dmin, dmax, wmax, g):
    """Out-degree uniform in [dmin, dmax], uniform targets other than the vertex itself."""
    deg = _rand(g, dmin, dmax + 1, n)
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
    m = src.numel()
    col = (src + 1 + _rand(g, 0, n - 1, m)) % n
    return _csr(n, src, col, _rand(g, 1, wmax + 1, m))


def _rmat(scale, factor, wmax, g):
    """R-MAT (.57, .19, .19, .05), relabelled, self-loops and duplicates removed."""
    n = 1 << scale
    m = n * factor
    src = torch.zeros(m, dtype=torch.int64, device="cuda")
    col = torch.zeros_like(src)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device="cuda")
        src = src * 2 + (r >= 0.76)
        col = col * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    label = torch.randperm(n, generator=g, device="cuda")
    key = torch.unique(label[src] * n + label[col])
    src, col = key // n, key % n
    keep = src != col
    src, col = src[keep], col[keep]
    return _csr(n, src, col, _rand(g, 1, wmax + 1, src.numel()))


def _grid(rows, cols, wmax, g):
    """4-neighbour grid, both directions, vertex (i, j) = i * cols + j."""
    n = rows * cols
    v = torch.arange(n, device="cuda")
    i, j = v // cols, v % cols
    ok = torch.stack([i > 0, j > 0, j < cols - 1, i < rows - 1], 1)
    to = torch.stack([v - cols, v - 1, v + 1, v + cols], 1)
    src = v[:, None].expand(n, 4)[ok]
    return _csr(n, src, to[ok], _rand(g, 1, wmax + 1, src.numel()))


def _dag(layers, width, deg, skip, wmax, g):
    """deg edges per vertex to layer + U{1..skip}; edges past the last layer dropped."""
    n = layers * width
    src = torch.arange(n, device="cuda").repeat_interleave(deg)
    lay = src // width + _rand(g, 1, skip + 1, src.numel())
    col = lay * width + _rand(g, 0, width, src.numel())
    keep = lay < layers
    src, col = src[keep], col[keep]
    return _csr(n, src, col, _rand(g, 1, wmax + 1, src.numel()))


def _sources(graph, count, g):
    """Sources among the vertices with out-edges."""
    cand = torch.nonzero(graph[1][1:] > graph[1][:-1]).flatten()
    return cand[_rand(g, 0, cand.numel(), count)].tolist()


def _corner(rows, cols, g):
    """A source in the sixteenth of the grid's rows and columns nearest vertex 0."""
    i, j = _rand(g, 0, 1 << 20, 2).tolist()
    return i % max(1, rows // 16) * cols + j % max(1, cols // 16)


def _sizes(count, nmin, nmax):
    """Vertex counts spread evenly over the logarithm of [nmin, nmax], unordered."""
    r = random.Random(count)
    u = [(i + r.random()) / count for i in range(count)]
    r.shuffle(u)
    return [int(nmin * (nmax / nmin) ** x) for x in u]


def _problem(c, seed):
    """(graphs, queries): queries are (graph index, source)."""
    g = _gen(seed)
    k = c["kind"]
    if k == "random":
        graphs = [_random(c["n"], c["dmin"], c["dmax"], c["wmax"], g)]
    elif k == "rmat":
        graphs = [_rmat(c["scale"], c["factor"], c["wmax"], g)]
    elif k == "grid":
        return ([_grid(c["rows"], c["cols"], c["wmax"], g)],
                [(0, _corner(c["rows"], c["cols"], g))])
    elif k == "dag":
        return [_dag(c["layers"], c["width"], c["deg"], c["skip"], c["wmax"], g)], [(0, 0)]
    elif k == "batch":
        graphs = [_random(n, 4, 16, c["wmax"], g)
                  for n in _sizes(c["count"], c["nmin"], c["nmax"])]
        return graphs, [(i, _sources(x, 1, g)[0]) for i, x in enumerate(graphs)]
    elif k == "sources":
        graphs = [_rmat(c["scale"], c["factor"], c["wmax"], g)]
        return graphs, [(0, s) for s in _sources(graphs[0], c["count"], g)]
    else:
        graphs = [_random(n, 4, 16, c["wmax"], g)
                  for n in _sizes(c["graphs"], c["nmin"], c["nmax"])]
        graphs.append(_rmat(c["scale"], 16, 255, g))
        which = [c["graphs"] if i % 10 == 0 else i % c["graphs"] for i in range(c["queries"])]
        return graphs, [(i, _sources(graphs[i], 1, g)[0]) for i in which]
    return graphs, [(0, _sources(graphs[0], 1, g)[0])]


# -------------------------------------------------------------------- cases

class _State:
    """Handles, server and buffers of one case, released with the state."""


def _options(c):
    o = sssp.sssp_options_default()
    o.rule = {"threshold": sssp.SSSP_RULE_THRESHOLD, "cheap": sssp.SSSP_RULE_CHEAP_FIRST,
              "windowed": sssp.SSSP_RULE_WINDOWED}[c["rule"]]
    o.layout = {"auto": sssp.SSSP_LAYOUT_AUTO, "wide": sssp.SSSP_LAYOUT_WIDE}[c["layout"]]
    if c["rule"] == "windowed":
        o.delta = max(1, c["wmax"] // 4)      # max weight / max degree of a grid
    return o


def _host(graph):
    n, ptr, _, col, w = graph
    return (n, ptr.cpu().numpy().astype(np.uint64), col.to(torch.int32).cpu().numpy().view(np.uint32),
            w.to(torch.int32).cpu().numpy().view(np.uint32))


def _release(server, handles):
    torch.cuda.synchronize()
    sssp.sssp_serve_close(server)
    for h in handles:
        sssp.sssp_destroy(h)


def prepare(case, seed):
    s = _State()
    s.case = case
    s.options = _options(case)
    graphs, s.queries = _problem(case, seed)
    host = [_host(x) for x in graphs]
    del graphs
    s.server, s.handles = None, []
    if case["entry"] == "oneshot":
        s.host = host[0]
        s.out = sssp.host_empty(host[0][0])
        return s
    s.handles = [sssp.sssp_create(*x, options=s.options) for x in host]
    ns = [host[i][0] for i, _ in s.queries]
    at = np.concatenate([[0], np.cumsum(ns)]).tolist()
    if case["kind"] == "serve":
        s.server = sssp.sssp_serve_open(budget_bytes=2 << 30)
        s.flat = np.zeros(at[-1], dtype=np.uint64)
    elif case["entry"] == "device":
        s.flat = torch.zeros(at[-1], dtype=torch.int64, device="cuda")
    elif case["entry"] == "host":
        s.flat = sssp.host_empty(at[-1])
    else:
        s.flat = None
    if s.flat is not None:
        s.outs = [s.flat[a:b] for a, b in zip(at[:-1], at[1:])]
    s.hs = [s.handles[i] for i, _ in s.queries]
    s.sources = [v for _, v in s.queries]
    weakref.finalize(s, _release, s.server, s.handles)
    return s


def run(s):
    c = s.case
    kind, entry = c["kind"], c["entry"]
    if kind in ("batch", "sources"):
        rounds = sssp.sssp_solve_batch_device(s.hs, s.sources, s.outs,
                                              stream=torch.cuda.current_stream())
        return {"dist": s.flat, "rounds": rounds}
    if kind == "serve":
        tickets = [sssp.sssp_serve_submit(s.server, h, v, o)
                   for h, v, o in zip(s.hs, s.sources, s.outs)]
        rounds = []
        for t in tickets:
            status, info = sssp.sssp_serve_wait(s.server, t, 60000)
            if status != sssp.SSSP_OK:
                raise RuntimeError("a query did not finish")
            rounds.append(info["rounds"])
        return {"dist": s.flat.view(np.int64), "rounds": np.array(rounds)}
    if entry == "oneshot":
        h = sssp.sssp_create(*s.host, options=s.options)
        try:
            dist, rounds = sssp.sssp_solve(h, s.queries[0][1], out=s.out)
        finally:
            sssp.sssp_destroy(h)
        return {"dist": dist.view(np.int64), "rounds": rounds}
    if entry == "host":
        dist, rounds = sssp.sssp_solve(s.hs[0], s.sources[0], out=s.outs[0])
        return {"dist": dist.view(np.int64), "rounds": rounds}
    if entry == "all":
        r = sssp.sssp_solve_ex(s.hs[0], s.sources[0], parent=True, fixed_round=True, lower=True)
        return {"dist": r["dist"].view(np.int64), "parent": r["parent"].view(np.int32),
                "fixed_round": r["fixed_round"], "lower": r["lower"].view(np.int64),
                "rounds": r["info"]["rounds"], "reached": r["info"]["reached"],
                "out_scanned": r["info"]["out_scanned"], "in_scanned": r["info"]["in_scanned"]}
    sssp.sssp_solve_device(s.hs[0], s.sources[0], s.outs[0], stream=torch.cuda.current_stream())
    return {"dist": s.flat}


def work(case):
    """Each query reads its graph once (8-byte offsets, 4-byte targets and
    weights) and writes 8-byte distances; an addition and a comparison per edge."""
    k = case["kind"]
    if k == "random":
        n, m = case["n"], case["n"] * (case["dmin"] + case["dmax"]) / 2
    elif k in ("rmat", "sources"):
        n = 1 << case["scale"]
        m = n * case["factor"]                  # a few per cent are duplicates
    elif k == "grid":
        n = case["rows"] * case["cols"]
        m = 4 * n - 2 * (case["rows"] + case["cols"])
    elif k == "dag":
        n = case["layers"] * case["width"]
        m = n * case["deg"]
    elif k == "batch":
        n = case["count"] * (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
        m = 10 * n
    else:
        n = (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
        n = case["queries"] * (0.9 * n + 0.1 * (1 << case["scale"]))
        m = 10.6 * n
    if k == "sources":                          # one graph, many outputs
        return {"bytes": 8 * (n + 1) + 8 * m + 8 * n * case["count"],
                "flops": 2 * m * case["count"]}
    extra = 16 * n if case["entry"] == "all" else 0    # parents, fixing rounds, lower bounds
    return {"bytes": 8 * (n + 1) + 8 * m + 8 * n + extra, "flops": 2 * m}


def exact(case, seed):
    """Distances by Bellman-Ford over all edges; the other outputs depend on
    the rounds and have no value of their own."""
    graphs, queries = _problem(case, seed)
    inf = torch.iinfo(torch.int64).max // 4
    dist = []
    for i, source in queries:
        n, _, src, col, w = graphs[i]
        d = torch.full((n,), inf, dtype=torch.int64, device="cuda")
        d[source] = 0
        sweeps = 0
        while True:
            sweeps += 1
            before = d.clone() if sweeps % 16 == 0 else None
            d.scatter_reduce_(0, col, d[src] + w, "amin")
            if before is not None and torch.equal(before, d):
                break
        dist.append(torch.where(d >= inf, torch.full_like(d, -1), d))
    dist = torch.cat(dist)
    out = {"dist": dist, "rounds": None, "parent": None, "fixed_round": None, "lower": None,
           "reached": None, "out_scanned": None, "in_scanned": None}
    if case["entry"] == "all":
        out["reached"] = int((dist >= 0).sum())
        return out
    return {"dist": dist} if case["entry"] == "device" and case["kind"] not in ("batch", "sources") \
        else {"dist": dist, "rounds": None}
