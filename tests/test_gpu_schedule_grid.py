"""Scheduled updates with few CTAs, on the GPU: one CTA asks the network while the others look up the batch's
slots, or does both where it is alone."""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [1, 2, 3, 8, 9])
@pytest.mark.parametrize("hidden", [5, 33, 64])
def test_scheduled_updates_find_every_slot_and_pick_as_the_network_does(grid, hidden):
    g = W.erdos_renyi(2000, 14000, seed=1301, cap_hi=100)
    A = len(native.maxflow_sched_actions())
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, grid_blocks=grid)
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    rng = np.random.default_rng(1302)
    mlp = native.MLP(16, hidden, A, seed=1303)
    for size in (1, 31, 512, 2049):
        b = W.mixed_batch(es, size, rng, ins_cap_hi=100)
        y = mlp.forward(S.features(b.u, b.v, b.cap)[None])[0]
        a = S.update_scheduled(b.u, b.v, b.cap, mlp)
        assert y[a] <= y.min() + 1e-4, (size, a, y)
        es.apply(b.u, b.v, b.cap)
        assert S.query()[0] == oracle.maxflow(g.n, *es.coo(), g.s, g.t).value
        su, sv, scap, _ = S.residual()
        got = {(int(x), int(z)): int(c) for x, z, c in zip(su, sv, scap) if c}
        u, v, c = es.coo()
        assert got == {(int(x), int(z)): int(k) for x, z, k in zip(u, v, c) if k}
    mlp.close()
    S.close()
