"""Near iterations (global relabels cut short, excess walked down the BFS forest) on the GPU.

They run on push solves with the default schedule when the graph has at least
65536 reserved slots and the sink's row at most n / 8 slots.  The cases sit
around those lines and around the walks' two ways of taking a residual (up to
8192 by subtraction, above by compare and swap); every state is compared with
the oracle exactly and has to be a max-flow certificate.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

from helpers import assert_certificate

pytestmark = pytest.mark.gpu


def _sink_row(n, into, seed, cap_hi):
    """Random digraph whose sink has exactly `into` in-edges, and a source with n / 16 out-edges."""
    rng = np.random.default_rng(seed)
    g = W.erdos_renyi(n, 8 * n, seed=seed, cap_hi=cap_hi)
    keep = (g.dst != g.t) & (g.src != g.t) & (g.src != g.s) & (g.dst != g.s)
    tails = rng.choice(np.arange(1, n - 1), size=into, replace=False)
    heads = rng.choice(np.arange(1, n - 1), size=n // 16, replace=False)
    src = np.concatenate([g.src[keep], tails, np.zeros(heads.size, np.int64)]).astype(np.int32)
    dst = np.concatenate([g.dst[keep], np.full(into, g.t), heads]).astype(np.int32)
    cap = rng.integers(1, cap_hi + 1, size=src.size).astype(np.int32)
    return W.Graph(n, src, dst, cap, 0, n - 1)


CASES = {
    "rmat13": lambda: W.rmat(13, 16, 0.57, 0.19, 0.19, seed=701, cap_hi=1000),
    "rmat13_wide": lambda: W.rmat(13, 16, 0.57, 0.19, 0.19, seed=702, cap_hi=1 << 20),     # compare and swap
    "rmat13_at_8192": lambda: W.rmat(13, 16, 0.57, 0.19, 0.19, seed=703, cap_hi=8193),
    "er": lambda: W.erdos_renyi(6001, 48013, seed=704, cap_hi=100),
    "layered": lambda: W.layered_dag(6000, seed=705),
    "sink_row_at": lambda: _sink_row(8192, 1024, 706, 300),         # n / 8: near
    "sink_row_above": lambda: _sink_row(8192, 1025, 706, 300),      # one more: not
}


@pytest.mark.parametrize("name", list(CASES))
def test_near_iterations_equal_the_oracle(name):
    g = CASES[name]()
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    rng = np.random.default_rng(710)
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t)
    cap_hi = int(g.cap.max())
    for k in range(5):
        if k:
            bias = (g.s, g.t, 0.3) if k % 2 else None
            b = W.mixed_batch(es, (300, 4000)[k // 2 % 2], rng, ins_cap_hi=cap_hi, inc_hi=cap_hi // 2, st_bias=bias)
            es.apply(b.u, b.v, b.cap)
            S.update(b.u, b.v, b.cap)
        if k == 4:
            S.resolve_static()
        u, v, c = es.coo()
        ref = oracle.maxflow(g.n, u, v, c, g.s, g.t)
        val, side, cut = S.query(side=True, cut=True)
        assert val == ref.value and cut == ref.value
        assert np.array_equal(side, ref.smax)      # A = {h = n}: all that cannot reach t
        su, sv, scap, scf = S.residual()
        h, e = S.vertex_state()
        assert_certificate(g.n, g.s, g.t, su, sv, scap, scf, h, e, val)
    S.close()
