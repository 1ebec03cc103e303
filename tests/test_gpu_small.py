"""The cluster kernel of the small rounds against the oracle, at the sizes where
its lists, its three ways of reading an entry's edges and its hand-over change."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.test_gpu_parity import LAYOUTS, assert_parity

pytestmark = pytest.mark.gpu


def tree(fan, depth_weights, seed):
    """Levels of fan[i] children per vertex, below a path of three vertices, with
    an edge from every leaf's parent to a common sink."""
    edges = [(0, 1, 5), (1, 2, 5), (2, 3, 5)]
    level, n = [3], 4
    for f, w in zip(fan, depth_weights):
        nxt = []
        for u in level:
            ws = gg.uniform(seed, n, f, 1, w)
            edges += [(u, n + i, int(ws[i])) for i in range(f)]
            nxt += range(n, n + f)
            n += f
        level = nxt
    sink = n
    step = max(1, len(level) // 700)
    edges += [(u, sink, 3) for u in level[::step]]
    return gg.from_edges(n + 1, edges)


def layers(sizes, wmax, seed):
    """Layers of the given sizes, each fully linked to the next, behind a path."""
    sizes = [1, 1] + list(sizes)
    start = np.concatenate([[0], np.cumsum(sizes)])
    n = int(start[-1])
    deg = np.zeros(n, dtype=np.int64)
    cols = []
    for i in range(len(sizes) - 1):
        deg[start[i]:start[i + 1]] = sizes[i + 1]
        cols.append(np.tile(np.arange(start[i + 1], start[i + 2], dtype=np.uint32), sizes[i]))
    col = np.concatenate(cols)
    row_ptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.uint64)
    return gg.Graph(n, row_ptr, col, gg.uniform(seed, 1, len(col), 1, wmax).astype(np.uint32))


MODES = pytest.mark.parametrize("mode,delta", [(oracle.RULE_THR, None), (oracle.RULE_MIND, None),
                                               (oracle.CHEAP_FIRST, None), (oracle.RULE_THR, 7)],
                                ids=["threshold", "mind", "cheap", "windowed"])


@LAYOUTS
@MODES
@pytest.mark.parametrize("fan", [(3, 5), (100, 300), (40, 33, 17), (1, 1, 1500)],
                         ids=["tiny", "overflow", "groups", "star"])
def test_lists_grow_and_overflow(sssp_lib, layout, mode, delta, fan):
    """Lists from a handful of entries to more than the cluster holds."""
    assert_parity(sssp_lib, tree(fan, [50, 9, 1000], 11), 0, mode=mode, delta=delta, layout=layout)


@LAYOUTS
@MODES
@pytest.mark.parametrize("sizes,hub", [((15,) * 6, 0), ((33,) * 6, 0), ((130,) * 4, 0),
                                       ((520, 520), 0), ((520, 1200, 3), 1 << 20)],
                         ids=["group", "row", "rows", "hub", "cta"])
def test_entries_read_by_group_warp_and_cta(sssp_lib, layout, mode, delta, sizes, hub):
    """Degrees on both sides of the limits between lanes, warp and CTA; the last
    has more large entries than a CTA's list of them holds."""
    opt = {"hub_degree": hub, "chunk_edges": 1024} if hub else {}
    assert_parity(sssp_lib, layers(sizes, 40, len(sizes)), 0, mode=mode, delta=delta,
                  layout=layout, **opt)


@LAYOUTS
@pytest.mark.parametrize("tail_items", ["1", "2", "40"])
def test_hand_over_between_the_kernels(sssp_lib, layout, tail_items, monkeypatch):
    """Rounds that cross the size limit in both directions, at both hand-over
    points (after the relaxation, and at the end of a round)."""
    monkeypatch.setenv("SSSP_TAIL_ITEMS", tail_items)
    for g, s in ((gg.grid(60, 45, 1, 300, 3), 7), (gg.random_graph(3000, 5, 1, 60, 4), 1)):
        assert_parity(sssp_lib, g, s, layout=layout)
        assert_parity(sssp_lib, g, s, delta=20, layout=layout)


@pytest.mark.parametrize("given_csc", [False, True])
@pytest.mark.parametrize("where", ["first", "last", "every"])
def test_self_loops_are_dropped(sssp_lib, given_csc, where):
    """A loop at either end of the edge list, or at every vertex, with and
    without the caller's CSC: the graph is the one without the loops."""
    n = 333
    base = gg.random_graph(n, 4, 1, 50, 8)
    src, col, w = base.edges()
    at = {"first": [0], "last": [n - 1], "every": list(range(n))}[where]
    edges = list(zip(src.tolist(), col.tolist(), w.tolist()))
    g = gg.from_edges(n, edges + [(v, v, 1) for v in at])
    csc = {}
    if given_csc:
        s, c, ww = g.edges()
        order = np.argsort(c, kind="stable")
        ptr = np.concatenate([[0], np.cumsum(np.bincount(c, minlength=n))])
        csc = dict(col_ptr=ptr.astype(np.uint64), row=s[order], w_in=ww[order])
    h = sssp_lib.sssp_create(g.n, g.row_ptr, g.col, g.w, **csc)
    try:
        assert sssp_lib.sssp_num_edges(h) == base.m
        out = sssp_lib.sssp_solve_ex(h, 5, parent=True)
    finally:
        sssp_lib.sssp_destroy(h)
    ref = oracle.round_r(base, 5)
    assert np.array_equal(out["dist"], ref.dist) and np.array_equal(out["parent"], ref.parent)


WEIGHTS = {"unit": [1], "pair": [1, 2], "fifteen": list(range(1, 17)), "steps": [15, 16, 17, 31, 32, 33],
           "range": list(range(1, 256)), "spread": [1, 1000, 1 << 20], "top": [1, 1 << 31, 0xFFFFFFFF]}


@LAYOUTS
@pytest.mark.parametrize("given_csc", [False, True])
@pytest.mark.parametrize("mode,delta", [(oracle.RULE_THR, None), (oracle.RULE_MIND, None),
                                        (oracle.CHEAP_FIRST, None), (oracle.LABEL_CORRECT, None),
                                        (oracle.RULE_THR, 40)],
                         ids=["threshold", "mind", "cheap", "correcting", "windowed"])
@pytest.mark.parametrize("weights", list(WEIGHTS))
def test_in_edges_by_weight_class(sssp_lib, layout, given_csc, mode, delta, weights):
    """The lower bounds of the full-grid kernels, over rows in order of weight class
    and (the caller's CSC) over rows in any order: weights at the edges of the
    classes, rows of no in-edge up to several hub chunks, both round drivers."""
    P, n = sssp_lib, 2500
    g = gg.random_var_graph(n, 0, 9, 1, 50, 21)
    src, col, _ = g.edges()
    extra = np.arange(1, n, dtype=np.uint32)
    src = np.concatenate([src, extra, np.zeros(40, np.uint32)])
    col = np.concatenate([col, np.where(extra == 7, 8, 7).astype(np.uint32),   # a hub at 7
                          np.arange(1, 41, dtype=np.uint32)])
    pick = gg.uniform(9, 2, len(src), 0, len(WEIGHTS[weights]) - 1)
    w = np.array(WEIGHTS[weights], dtype=np.uint32)[pick.astype(np.int64)]
    g = gg.from_edges(n, list(zip(src.tolist(), col.tolist(), w.tolist())))
    csc = {}
    if given_csc:
        s, c, ww = g.edges()
        order = np.argsort(c, kind="stable")[::-1]
        order = order[np.argsort(c[order], kind="stable")]
        ptr = np.concatenate([[0], np.cumsum(np.bincount(c, minlength=n))])
        csc = dict(col_ptr=ptr.astype(np.uint64), row=s[order], w_in=ww[order])
    ref = oracle.round_r(g, 0, mode=mode, delta=delta)
    for loop in (P.SSSP_LOOP_HOST, P.SSSP_LOOP_GRAPH):
        opt = P.sssp_options_default()
        opt.layout = layout if n * max(WEIGHTS[weights]) < 2**31 - 1 else P.SSSP_LAYOUT_WIDE
        opt.loop_mode, opt.rule = loop, mode
        opt.hub_degree, opt.chunk_edges = 64, 512
        if delta is not None:
            opt.rule, opt.delta = P.SSSP_RULE_WINDOWED, delta
        h = P.sssp_create(g.n, g.row_ptr, g.col, g.w, options=opt, **csc)
        try:
            out = P.sssp_solve_ex(h, 0, parent=True, fixed_round=True, lower=True)
        finally:
            P.sssp_destroy(h)
        assert np.array_equal(out["dist"], ref.dist) and np.array_equal(out["parent"], ref.parent)
        assert np.array_equal(out["fixed_round"], ref.fixed_round)
        assert np.array_equal(out["lower"], ref.C)
        assert out["info"]["in_scanned"] == ref.stats["in_scanned"]
