"""maxflow_set_bfs_tail on the GPU: 0 keeps every BFS level on the grid.

The labels are the oracle's either way, on graphs whose BFS enters and leaves the
first cluster several times, before and after the 16th level.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _bellows(widths, seed):
    """Layers of the given widths, each vertex with three edges into the next one: a BFS of that many levels."""
    rng = np.random.default_rng(seed)
    first = np.concatenate([[1], 1 + np.cumsum(widths)])
    src, dst = [np.zeros(widths[0], np.int64)], [np.arange(1, 1 + widths[0])]
    n = int(first[-1]) + 1
    for k in range(len(widths)):
        a = np.arange(first[k], first[k + 1])
        if k + 1 == len(widths):
            src.append(a)
            dst.append(np.full(a.size, n - 1))
        else:
            b = np.arange(first[k + 1], first[k + 2])
            src += [np.repeat(a, 3), rng.choice(a, b.size)]
            dst += [rng.choice(b, 3 * a.size), b]
    src, dst = np.concatenate(src), np.concatenate(dst)
    _, at = np.unique(src * n + dst, return_index=True)
    return W.Graph(n, src[at].astype(np.int32), dst[at].astype(np.int32),
                   rng.integers(1, 50, at.size).astype(np.int32), 0, n - 1)


CASES = {
    "wide_and_narrow": lambda: _bellows([40, 6000, 30, 5000, 20] * 2 + [300] * 12 + [5000, 9] * 3, 1001),
    "narrow": lambda: _bellows([25] * 40, 1002),
    "grid": lambda: W.GridSegmentation(side=97, seed=1003, window=16, origin=(30, 30), step=2).graph(),
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("grid", [0, 5, 16])
def test_zero_turns_levels_of_the_first_cluster_off(name, grid):
    g = CASES[name]()
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, grid_blocks=grid)
    off, one = S.clone(), S.clone()
    off.set_bfs_tail(0)
    one.set_bfs_tail(1 << 20)
    b = W.mixed_batch(es, 100, np.random.default_rng(1004), ins_cap_hi=50)
    es.apply(b.u, b.v, b.cap)
    for X in (S, off, one):
        X.update(b.u, b.v, b.cap)
        assert X.query()[0] == oracle.maxflow(g.n, *es.coo(), g.s, g.t).value
        X.global_relabel()
        h, _ = X.vertex_state()
        su, sv, scap, scf = X.residual()
        R = oracle.Residual(g.n, *es.coo())
        keep = scap > 0
        R.set_flow(su[keep], sv[keep], np.maximum(scap[keep].astype(np.int64) - scf[keep], 0).astype(np.int32))
        assert np.array_equal(h, R.heights(g.s, g.t, deficit_roots=True))
    # a barrier per level and more across the grid; fewer where the first cluster runs levels alone
    st = off.stats()
    assert st["barriers"] > st["bfs_levels"]
    if st["bfs_levels"] > 12:
        assert S.stats()["barriers"] < st["barriers"]
    for X in (S, off, one):
        X.close()
