"""A CTA that never arrives, in launches with thread-block clusters, on the GPU.

The missing CTA sits in the first cluster (whose CTAs run small phases alone), in
another one, or in a launch without clusters.  The call reports the failure
within the wait limit, and the context solves correctly afterwards, with squads.
"""
import time

import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid,cta", [(8, 0), (8, 5), (16, 0), (16, 3), (16, 7), (16, 8), (16, 15), (24, 23),
                                      (7, 0), (9, 4)])
def test_a_missing_cta_ends_the_call_and_leaves_the_context_usable(grid, cta):
    G = W.GridSegmentation(side=97, seed=807, window=16, origin=(30, 30), step=2)
    g = G.graph()
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, grid_blocks=grid, wait_limit_s=0.05)
    assert S.stats()["grid_blocks"] == grid
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    for k in range(2):
        t0 = time.perf_counter()
        assert native.load().maxflow_test_stalled_barrier(S.h, cta) == native.ERR_INTERNAL
        assert time.perf_counter() - t0 < 2.0
        b = G.window_batch(k)
        es.apply(b.u, b.v, b.cap)
        S.update(b.u, b.v, b.cap)
        u, v, c = es.coo()
        ref = oracle.maxflow(g.n, u, v, c, g.s, g.t)
        val, side, cut = S.query(side=True, cut=True)
        assert val == ref.value == cut and np.array_equal(side, ref.smax)
    S.close()
