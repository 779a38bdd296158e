"""Discharge rounds of both kinds within one iteration, on the GPU.

Bipartite matching graphs whose right side has rows of 600 to 2100 slots (a round
with one of them active is never a short one) beside short rows, and a sink row
above n / 8 (no near iterations): rounds over hub rows are followed by rounds
without any, which queue behind stamps.  Exact against the oracle, and no residual below zero.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

from helpers import assert_certificate

pytestmark = pytest.mark.gpu


def _matching(left, hubs, small, seed):
    """s -> left -> hubs and small right vertices -> t, small right vertices among one another, and an edge from
    every fourth left vertex to t."""
    rng = np.random.default_rng(seed)
    L = np.arange(1, left + 1)
    H = np.arange(left + 1, left + hubs + 1)
    R = np.arange(left + hubs + 1, left + hubs + small + 1)
    n = left + hubs + small + 2
    s, t = 0, n - 1
    src = [np.full(left, s), np.repeat(L, 8), np.repeat(L, 3), H, R, R, L[::4]]
    dst = [L, rng.choice(H, 8 * left), rng.choice(R, 3 * left), np.full(hubs, t), np.full(small, t),
           rng.permutation(R), np.full(L[::4].size, t)]
    src, dst = np.concatenate(src), np.concatenate(dst)
    cap = rng.integers(1, 8, src.size)
    cap[src == s] = rng.integers(1, 20, left)
    cap[(dst == t) & (src > left)] = rng.integers(1, 30, hubs + small)
    keep = np.zeros(src.size, bool)
    keep[np.unique(src * n + dst, return_index=True)[1]] = True       # each pair once
    keep &= src != dst
    return W.Graph(n, src[keep].astype(np.int32), dst[keep].astype(np.int32), cap[keep].astype(np.int32), s, t)


@pytest.mark.parametrize("seed", range(8))
@pytest.mark.parametrize("left,hubs,small", [(3000, 30, 1500), (3000, 9, 300), (6000, 20, 4000)])
def test_rounds_of_both_kinds_keep_the_flow_feasible(left, hubs, small, seed):
    g = _matching(left, hubs, small, 900 + seed)
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    rng = np.random.default_rng(950 + seed)
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t)
    deg = np.bincount(S.residual()[0], minlength=g.n)
    assert S.stats()["slot_capacity"] >= 65536 and deg[g.t] > g.n // 8
    assert ((deg[1:-1] > 600) & (deg[1:-1] < 2400)).sum() >= hubs
    for k in range(5):
        if k:
            b = W.mixed_batch(es, 500, rng, ins_cap_hi=20, st_bias=(g.s, g.t, 0.5))
            es.apply(b.u, b.v, b.cap)
            S.update(b.u, b.v, b.cap)
        assert S.check()["pair_violations"] == 0
        u, v, c = es.coo()
        val = S.query()[0]
        assert val == oracle.maxflow(g.n, u, v, c, g.s, g.t).value
        su, sv, scap, scf = S.residual()
        assert scf.min() >= 0
        h, e = S.vertex_state()
        assert_certificate(g.n, g.s, g.t, su, sv, scap, scf, h, e, val)
    S.close()
