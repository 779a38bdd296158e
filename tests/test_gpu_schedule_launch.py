"""The learned schedule inside the launch of the batch, on the GPU.

The action a launch picks is the network's minimum over the batch's features as
maxflow_features and the network's own forward pass give them (fp32 sums of up
to 256 terms in another order: outputs within 1e-4 of the smallest are ties),
for networks of 1, 64 and 256 hidden units.  Networks of zero weights that
prefer one action run it, incremental or from zero flow; each value is the
oracle's.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GRAPHS = {
    "small": lambda: W.erdos_renyi(300, 2000, seed=881, cap_hi=100),
    "er": lambda: W.erdos_renyi(4000, 24000, seed=882, cap_hi=100),
    "rmat": lambda: W.rmat(12, 16, 0.57, 0.19, 0.19, seed=883, cap_hi=1000),     # near iterations
}


def _value(g, es):
    u, v, c = es.coo()
    return oracle.maxflow(g.n, u, v, c, g.s, g.t).value


@pytest.mark.parametrize("graph", GRAPHS)
@pytest.mark.parametrize("hidden", [1, 64, 256])
def test_the_launch_picks_what_the_network_prefers(graph, hidden):
    g = GRAPHS[graph]()
    A = len(native.maxflow_sched_actions())
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t)
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    rng = np.random.default_rng(884)
    for k, size in enumerate((1, 33, 511, 700)):
        b = W.mixed_batch(es, size, rng, ins_cap_hi=100, st_bias=(g.s, g.t, 0.3) if k % 2 else None)
        mlp = native.MLP(16, hidden, A, seed=885 + k)
        y = mlp.forward(S.features(b.u, b.v, b.cap)[None])[0]
        a = S.update_scheduled(b.u, b.v, b.cap, mlp)
        es.apply(b.u, b.v, b.cap)
        assert y[a] <= y.min() + 1e-4, (size, a, y)
        assert S.query()[0] == _value(g, es)
        mlp.close()
    S.close()


@pytest.mark.parametrize("graph", ["er", "rmat"])
def test_every_action_runs_in_the_launch(graph):
    g = GRAPHS[graph]()
    A = len(native.maxflow_sched_actions())
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t)
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    rng = np.random.default_rng(886)
    mlp = native.MLP(16, 8, A, seed=1)
    for a in range(A):
        p = np.zeros_like(mlp.params)
        p[p.size - A + a] = -1.0                   # the last layer's bias
        mlp.params = p
        b = W.mixed_batch(es, 400, rng, ins_cap_hi=100)
        assert S.update_scheduled(b.u, b.v, b.cap, mlp) == a
        es.apply(b.u, b.v, b.cap)
        assert S.query()[0] == _value(g, es), a
    mlp.close()
    S.close()
