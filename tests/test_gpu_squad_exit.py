"""The first cluster keeps the levels at the end of a deep BFS, on the GPU.

From the 16th level on no level turns bottom-up, so the first cluster does not leave
its run of small levels for one: the BFS of a ladder, 300 levels of 6 vertices, ends
in one run, however little is left unexplored.
"""
import numpy as np
import pytest

from paper_2511_01235_gb300 import native

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [5, 8, 16])
@pytest.mark.parametrize("alpha,limit", [(0, 8), (14, 8), (1000, 8 + 2 * 16)])
def test_a_deep_bfs_ends_in_one_run_of_the_first_cluster(grid, alpha, limit):
    length, width = 300, 6
    idx = np.arange(length * width).reshape(length, width)
    n = length * width + 2
    src = np.concatenate([np.full(width, n - 2), idx[:-1].ravel(), idx[-1]]).astype(np.int32)
    dst = np.concatenate([idx[0], idx[1:].ravel(), np.full(width, n - 1)]).astype(np.int32)
    cap = np.where(src == n - 2, 1, 5).astype(np.int32)        # saturated at the source only: t is reached from all
    S = native.Solver(n, src, dst, cap, n - 2, n - 1, grid_blocks=grid)
    S.set_bfs_switch(alpha, 24)
    S.global_relabel()
    st = S.stats()
    assert S.query()[0] == width
    assert np.array_equal(S.vertex_state()[0][idx], np.repeat(np.arange(length, 0, -1)[:, None], width, 1))
    assert st["bfs_levels"] >= length
    # the roots, one run, the launch's first and last barrier; a level that changes direction ends a run, but only
    # among the first 16, and takes one barrier or two
    assert st["barriers"] <= limit, st["barriers"]
    S.close()
