"""Solves that end at a cap, on graphs where relabels may be cut short, on the GPU.

A solve that ends at its time limit or iteration cap leaves complete labels (the
oracle's on the same preflow), and its value is summed over them.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cap", [dict(time_limit_s=1e-9), dict(time_limit_s=2e-4), dict(max_iters=1), dict(max_iters=2)],
                         ids=str)
@pytest.mark.parametrize("family", ["rmat", "er"])
def test_a_capped_solve_leaves_complete_labels(family, cap):
    if family == "rmat":
        g = W.rmat(13, 16, 0.57, 0.19, 0.19, seed=1101, cap_hi=1000)
    else:
        g = W.erdos_renyi(6001, 48013, seed=1102, cap_hi=100)
    # a graph without capacity converges at once; the batch then gives it all of them
    S = native.Solver(g.n, g.src, g.dst, np.zeros_like(g.cap), g.s, g.t, **cap)
    assert S.stats()["slot_capacity"] >= 65536
    try:
        S.update(g.src, g.dst, g.cap)
    except native.MaxflowError as ex:
        assert ex.code == native.ERR_NOT_CONVERGED
    else:
        assert cap != dict(time_limit_s=1e-9)
    h, e = S.vertex_state()
    su, sv, scap, scf = S.residual()
    R = oracle.Residual(g.n, g.src, g.dst, g.cap)
    keep = scap > 0
    R.set_flow(su[keep], sv[keep], np.maximum(scap[keep].astype(np.int64) - scf[keep], 0).astype(np.int32))
    assert np.array_equal(h, R.heights(g.s, g.t, deficit_roots=True))
    below = h < g.n
    below[g.s] = False
    assert S.stats()["value"] == int(e[below].sum())
    assert S.check()["pair_violations"] == 0
    S.close()
