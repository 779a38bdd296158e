"""Saturation across the last cut (push-pull updates) over rows of 511 to 5000 slots, on the GPU: up to 512 slots
a warp's, above the whole CTA's."""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

from helpers import assert_certificate

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("row", [511, 512, 513, 1024, 5000])
@pytest.mark.parametrize("grid", [1, 3, 0])
def test_no_residual_edge_crosses_the_last_cut(row, grid):
    # s -> hubs (wide), hubs -> leaves (narrow), leaves -> t (wide): the cut runs through the hubs' rows, and raising
    # their capacities opens residual edges across it
    rng = np.random.default_rng(1400 + row)
    hubs = 20
    leaves = row - 1 + 50
    H, L = np.arange(1, hubs + 1), np.arange(hubs + 1, hubs + 1 + leaves)
    n = hubs + leaves + 2
    t = n - 1
    src, dst, cap = [np.zeros(hubs, np.int64), L], [H, np.full(leaves, t)], [np.full(hubs, 10 ** 7), np.full(leaves, 10 ** 4)]
    for h in H:
        src.append(np.full(row - 1, h))                    # and the slot to s
        dst.append(rng.choice(L, row - 1, replace=False))
        cap.append(rng.integers(1, 5, row - 1))
    src, dst, cap = (np.concatenate(x).astype(np.int32) for x in (src, dst, cap))
    es = W.EdgeSet(n, src, dst, cap)
    S = native.Solver(n, src, dst, cap, 0, t, grid_blocks=grid)
    inner = np.flatnonzero((src > 0) & (src <= hubs))
    for k in range(3):
        at = rng.choice(inner, inner.size // 2, replace=False)
        b = src[at], dst[at], (cap[at] + rng.integers(0, 9, at.size)).astype(np.int32)
        side = S.query(side=True)[1]                       # True: the source's side
        es.apply(*b)
        C = S.clone()
        C.update_pp(*b, stop_after=1)
        su, sv, scap, scf = C.residual()
        assert not (scf[side[su] & ~side[sv]] > 0).any()
        chk = C.check()
        assert chk["pair_violations"] == 0 and chk["excess_mismatch"] == 0
        C.close()
        S.update_pp(*b)
        val = S.query()[0]
        assert val == oracle.maxflow(n, *es.coo(), 0, t).value
        su, sv, scap, scf = S.residual()
        h, e = S.vertex_state()
        assert_certificate(n, 0, t, su, sv, scap, scf, h, e, val)
    S.close()
