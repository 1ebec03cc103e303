"""Limits that the sizes of a call cross: hub chunks in the cluster kernel's rounds,
device memory, queries of a batch, the end of the adjacency."""
import numpy as np
import pytest

import graphgen as gg
import oracle
from tests.test_gpu_parity import LAYOUTS, assert_parity

pytestmark = pytest.mark.gpu


@LAYOUTS
@pytest.mark.parametrize("mode,delta", [(oracle.RULE_THR, None), (oracle.RULE_THR, 9)],
                         ids=["threshold", "windowed"])
@pytest.mark.parametrize("hub,chunk,n,deg", [(1, 32, 250, 4), (4, 64, 250, 5), (16, 64, 250, 18),
                                             (16, 64, 900, 18), (256, 1024, 250, 4)])
def test_small_hubs_stay_in_the_cluster_kernel(sssp_lib, layout, mode, delta, hub, chunk, n, deg):
    """With a small hub degree most vertices of a small round are hubs of a single short
    chunk: every round after the first runs in the cluster kernel (n = 900: rounds
    with more chunks than it takes, too)."""
    P = sssp_lib
    g = gg.random_graph(n, deg, 1, 60, 17)
    assert_parity(P, g, 3, mode=mode, delta=delta, layout=layout, hub_degree=hub, chunk_edges=chunk)
    opt = P.sssp_options_default()
    opt.layout, opt.rule, opt.hub_degree, opt.chunk_edges = layout, mode, hub, chunk
    if delta is not None:
        opt.rule, opt.delta = P.SSSP_RULE_WINDOWED, delta
    h = P.sssp_create(g.n, g.row_ptr, g.col, g.w, options=opt)
    try:
        P.sssp_profile(h, True)
        _, rounds = P.sssp_solve(h, 3)
        prof = P.sssp_profile(h, False)
    finally:
        P.sssp_destroy(h)
    assert 0 < prof["tail_rounds"] <= rounds - 1
    if n == 250:
        assert prof["tail_rounds"] == rounds - 1


class Budget:
    """Device allocator hooks that count, and refuse what would pass a number of bytes."""

    def __init__(self, P, nbytes=1 << 40):
        import torch
        self.live, self.left, self.calls = {}, nbytes, 0

        def alloc(size, _ctx):
            self.calls += 1
            if size > self.left:
                return None
            t = torch.empty(max(size, 1), dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = (t, size)
            self.left -= size
            return t.data_ptr()

        def free(p, _ctx):
            torch.cuda.synchronize()
            self.left += self.live.pop(p)[1]

        self.options = P.sssp_options_default()
        self.options.alloc, self.options.free = P.ALLOC_FN(alloc), P.FREE_FN(free)


@pytest.mark.parametrize("n", [2, 300, 4000])
def test_allocations_of_a_small_graph(sssp_lib, n):
    """Creating a small graph takes 31 allocations: 7 for the graph (five arrays, the
    descriptions, the packed outWeights), 6 of scratch (two for the upload, three for the
    transposition, the hub counts), 18 for the solve state; none to look for self-loops."""
    P = sssp_lib
    g = gg.random_graph(n, min(n - 1, 6), 1, 50, 2)
    b = Budget(P)
    h = P.sssp_create(g.n, g.row_ptr, g.col, g.w, options=b.options)
    calls = b.calls
    P.sssp_destroy(h)
    assert calls <= 31 and not b.live


@pytest.mark.parametrize("given_csc", [False, True])
@pytest.mark.parametrize("loops", [False, True])
def test_graph_that_fits_without_descriptions(sssp_lib, loops, given_csc):
    """A memory budget that holds the graph (28 bytes per vertex and 16 per edge), its
    compact state (52 per vertex), the lower bounds on their way to the host (8 per vertex)
    and the control slots, but no vertex descriptions: the graph is created, self-loops
    take no room, and every output is the oracle's.  A budget that does not hold the
    graph gives SSSP_E_NOMEM and everything is handed back."""
    P = sssp_lib
    g = gg.grid(300, 200, 1, 900, 5)
    full = g
    if loops:
        src, col, w = g.edges()
        every = np.arange(g.n, dtype=np.uint32)
        full = gg.from_edges(g.n, np.stack([np.concatenate([src, every]), np.concatenate([col, every]),
                                            np.concatenate([w, np.ones_like(every)])], 1).tolist())
    csc = {}
    if given_csc:
        s, c, ww = full.edges()
        order = np.argsort(c, kind="stable")
        ptr = np.concatenate([[0], np.cumsum(np.bincount(c, minlength=g.n))])
        csc = dict(col_ptr=ptr.astype(np.uint64), row=s[order], w_in=ww[order])
    b = Budget(P, 89 * g.n + 16 * g.m + (1 << 17))
    h = P.sssp_create(g.n, full.row_ptr, full.col, full.w, options=b.options, **csc)
    try:
        assert P.sssp_num_edges(h) == g.m
        out = P.sssp_solve_ex(h, 123, parent=True, fixed_round=True, lower=True)
    finally:
        P.sssp_destroy(h)
    assert not b.live
    ref = oracle.round_r(g, 123)
    assert np.array_equal(out["dist"], ref.dist) and np.array_equal(out["parent"], ref.parent)
    assert np.array_equal(out["fixed_round"], ref.fixed_round) and np.array_equal(out["lower"], ref.C)
    b = Budget(P, 16 * g.m)
    with pytest.raises(P.SsspError) as e:
        P.sssp_create(g.n, full.row_ptr, full.col, full.w, options=b.options, **csc)
    assert e.value.code == P.SSSP_E_NOMEM and not b.live


@LAYOUTS
@pytest.mark.parametrize("mode,delta", [(oracle.RULE_THR, None), (oracle.RULE_THR, 9)],
                         ids=["threshold", "windowed"])
def test_last_vertex_without_out_edges(sssp_lib, layout, mode, delta):
    """The adjacency fills its 2 MB exactly and the last vertices have no out-edge: their
    rows begin at its end."""
    n, sinks = 8192, 40
    src = np.repeat(np.arange(n, dtype=np.uint32), 32)
    col = (src + gg.uniform(3, 1, len(src), 1, n + sinks - 1).astype(np.uint32)) % np.uint32(n + sinks)
    w = gg.uniform(3, 2, len(src), 1, 70).astype(np.uint32)
    row_ptr = np.concatenate([np.arange(n + 1) * 32, np.full(sinks, 32 * n)]).astype(np.uint64)
    g = gg.Graph(n + sinks, row_ptr, col, w)
    assert 8 * g.m == 1 << 21
    assert_parity(sssp_lib, g, 0, mode=mode, delta=delta, layout=layout)


@LAYOUTS
@pytest.mark.parametrize("mode,delta", [(oracle.RULE_THR, None), (oracle.LABEL_CORRECT, None),
                                        (oracle.RULE_THR, 15)],
                         ids=["threshold", "correcting", "windowed"])
def test_more_queries_than_a_cta_keeps_minima_of(sssp_lib, layout, mode, delta):
    """1100 queries of one batch: the minima and counts of those after the 1024th go to
    global memory one by one.  Every query's distances and rounds are its own run's."""
    P, n, k = sssp_lib, 170, 1100
    g = gg.random_var_graph(n, 1, 7, 1, 40, 12)
    opt = P.sssp_options_default()
    opt.layout, opt.rule = layout, mode
    if delta is not None:
        opt.rule, opt.delta = P.SSSP_RULE_WINDOWED, delta
    refs = [oracle.round_r(g, s, mode=mode, delta=delta) for s in range(n)]
    sources = [(7 * i) % n for i in range(k)]
    h = P.sssp_create(g.n, g.row_ptr, g.col, g.w, options=opt)
    try:
        dist, rounds = P.sssp_solve_batch([h] * k, sources)
    finally:
        P.sssp_destroy(h)
    for i, s in enumerate(sources):
        assert rounds[i] == refs[s].rounds, i
        assert np.array_equal(dist[i], refs[s].dist), i
