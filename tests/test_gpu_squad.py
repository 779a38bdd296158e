"""Short discharge rounds and small phases in the squad (the first thread-block cluster) on the GPU.

Cases at the edges of what picks them: launches with and without clusters
(grids of 7, 8 and 9 CTAs), frontiers around the squad's limit, rows of 8 and 9
slots (a thread or a warp), of 512 and 513 (short round or not), work that
leaves the squad again, and the library's own choice.  Exact against the oracle.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

from helpers import assert_certificate

pytestmark = pytest.mark.gpu


def _ladder(length, width, seed, hub=0):
    """`width` parallel chains of `length` vertices with rungs between neighbours: a BFS of `length` levels of
    `width` vertices.  With hub > 0 one inner vertex (four slots of its own) joins that many others."""
    rng = np.random.default_rng(seed)
    idx = np.arange(length * width).reshape(length, width)
    a = [idx[:-1].ravel(), idx[:, :-1].ravel(), idx[:, 1:].ravel()]
    b = [idx[1:].ravel(), idx[:, 1:].ravel(), idx[:, :-1].ravel()]
    n = length * width + 2
    s, t = n - 2, n - 1
    a += [np.full(width, s), idx[-1]]
    b += [idx[0], np.full(width, t)]
    if hub:
        far = idx[length // 2 + 2:].ravel()[:hub]
        assert far.size == hub
        a.append(np.full(hub, idx[length // 2, width // 2]))
        b.append(far)
    src, dst = np.concatenate(a), np.concatenate(b)
    return W.Graph(n, src.astype(np.int32), dst.astype(np.int32),
                   rng.integers(1, 100, src.size).astype(np.int32), s, t)


CASES = {
    "deep_narrow": lambda: _ladder(300, 6, 801),
    "deep_at_limit": lambda: _ladder(40, 256, 802),          # one CTA's limit
    "deep_squad_limit": lambda: _ladder(24, 2048, 803),      # the cluster's
    "deep_above": lambda: _ladder(24, 2049, 804),
    "row_of_512": lambda: _ladder(64, 60, 805, hub=508),
    "row_of_513": lambda: _ladder(64, 60, 806, hub=509),     # leaves the squad
    "row_of_1800": lambda: _ladder(64, 60, 807, hub=1796),
    "grid97": lambda: W.GridSegmentation(side=97, seed=807, window=16, origin=(30, 30), step=2).graph(),
    "geometric": lambda: W.geometric(5001, seed=808, avg_deg=9.0),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("grid", [0, 7, 8, 9])
def test_squad_phases_equal_the_oracle(name, grid):
    g = CASES[name]()
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    rng = np.random.default_rng(810)
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, grid_blocks=grid)
    for k in range(3):
        if k:
            b = W.mixed_batch(es, 200, rng, ins_cap_hi=99, st_bias=(g.s, g.t, 0.3))
            es.apply(b.u, b.v, b.cap)
            S.update(b.u, b.v, b.cap)
        u, v, c = es.coo()
        ref = oracle.maxflow(g.n, u, v, c, g.s, g.t)
        val, side, cut = S.query(side=True, cut=True)
        assert val == ref.value and cut == ref.value
        assert np.array_equal(side, ref.smax)
        su, sv, scap, scf = S.residual()
        h, e = S.vertex_state()
        assert_certificate(g.n, g.s, g.t, su, sv, scap, scf, h, e, val)
    S.close()
