"""Limits that the sizes of a call cross: hub chunks in the cluster kernel's rounds."""
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
