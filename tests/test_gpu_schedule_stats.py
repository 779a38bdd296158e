"""Statistics of a scheduled update on the GPU: those of the action that it picked."""
import numpy as np
import pytest

from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_cycles", [0, 7])
def test_a_scheduled_update_reports_what_its_action_reports(own_cycles):
    g = W.erdos_renyi(4000, 24000, seed=1201, cap_hi=100)
    acts = native.maxflow_sched_actions()
    S = native.Solver(g.n, g.src, g.dst, g.cap, g.s, g.t, kernel_cycles=own_cycles)
    es = W.EdgeSet(g.n, g.src, g.dst, g.cap)
    b = W.mixed_batch(es, 300, np.random.default_rng(1202), ins_cap_hi=100)
    mlp = native.MLP(16, 8, len(acts), seed=1)
    for a in range(len(acts)):
        p = np.zeros_like(mlp.params)
        p[p.size - len(acts) + a] = -1.0               # the last layer's bias
        mlp.params = p
        A, B = S.clone(), S.clone()
        A.run_action(b.u, b.v, b.cap, a)
        assert B.update_scheduled(b.u, b.v, b.cap, mlp) == a
        sa, sb = A.stats(), B.stats()
        for key in ("kernel_cycles", "rounds", "solves", "updates", "rebuilds", "slots", "slot_capacity", "m_edges",
                    "value"):
            assert sa[key] == sb[key], (a, key, sa[key], sb[key])
        A.close()
        B.close()
    mlp.close()
    S.close()
