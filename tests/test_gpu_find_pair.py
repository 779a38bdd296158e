"""The row in which a batch's slots are looked up, on the GPU.

A pair between a vertex with a long sorted row and one whose row grew by
insertions is looked up in the long row: its slots take a few reads, inserted ones
are read one by one.  The slots read show in the statistics.
"""
import numpy as np
import pytest

import oracle
from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("inserted", [0, 1, 3, 400])
def test_a_row_of_many_inserted_slots_is_not_searched_for_a_long_sorted_one(inserted):
    n, hub, small = 4000, 1, 2
    far = np.arange(10, 1500)
    src = np.concatenate([[0, 0], np.full(far.size, hub), far]).astype(np.int32)
    dst = np.concatenate([[hub, small], far, np.full(far.size, n - 1)]).astype(np.int32)
    cap = np.full(src.size, 5, np.int32)
    es = W.EdgeSet(n, src, dst, cap)
    S = native.Solver(n, src, dst, cap, 0, n - 1)

    def change(u, v, c):
        u, v, c = (np.asarray(x, np.int32) for x in (u, v, c))
        S.update(u, v, c)
        es.apply(u, v, c)

    if inserted:
        change(np.full(inserted, small), np.arange(2000, 2000 + inserted), np.full(inserted, 3))
    for c in (9, 4):                               # the pair is new, then there
        change([hub], [small], [c])
        # 60 bytes for the update, 48 for a clamp, 4 for every slot read: the source's two, seven per division by
        # eight of the hub's 1491 base slots and nine at the end, and the inserted ones of the row searched
        reads = 2 + 3 * 7 + 9 + 1
        assert S.stats()["bytes_apply"] <= 60 + 48 + 4 * reads, (c, S.stats()["bytes_apply"])
    ue, ve, ce = es.coo()
    assert S.query()[0] == oracle.maxflow(n, ue, ve, ce, 0, n - 1).value
    S.close()
