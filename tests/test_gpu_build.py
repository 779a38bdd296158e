"""The residual layout made on the device against the one made on the host, slot for slot.

Edge lists from 16384 entries on are built on the device.  The cases sit around
that line, around the digits of the sort (vertex counts at and beside powers of
two), and hold parallel edges, self-loops, zero capacities and hub rows.  The
host's layout is pinned to the oracle on the CPU (test_layout_host.py).
"""
import numpy as np
import pytest

from paper_2511_01235_gb300 import native
from paper_2511_01235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _random(n, m, seed, cap_hi=50, hub=0.0):
    rng = np.random.default_rng(seed)
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    u[rng.random(m) < hub] = 0
    c = rng.integers(0, cap_hi + 1, m)
    return n, u.astype(np.int32), v.astype(np.int32), c.astype(np.int32)


CASES = {
    "below_the_line": lambda: _random(3000, 16383, 1),
    "at_the_line": lambda: _random(3000, 16384, 2),
    "two_vertices": lambda: _random(2, 20000, 3, cap_hi=3),
    "n_255": lambda: _random(255, 20011, 4),             # row n is the last one of the first digit
    "n_256": lambda: _random(256, 20011, 5),
    "n_257": lambda: _random(257, 20011, 6),
    "n_65535": lambda: _random(65535, 70001, 7),
    "n_65536": lambda: _random(65536, 70001, 8),
    "hub": lambda: _random(20000, 100003, 9, hub=0.4),
    "one_tile": lambda: _random(5000, 2048 * 8, 10),
    "loops_only": lambda: (5000, np.arange(20000, dtype=np.int32) % 5000, np.arange(20000, dtype=np.int32) % 5000,
                           np.ones(20000, np.int32)),
    "rmat14": lambda: (lambda g: (g.n, g.src, g.dst, g.cap))(W.rmat(14, 16, seed=11)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_device_layout_equals_the_host_layout(name):
    n, u, v, c = CASES[name]()
    L = native.build_layout(n, u, v, c)
    S = native.Solver(n, u, v, c, 0, n - 1)
    st = S.stats()
    used = int(L["deg"].sum())
    assert st["slots"] == used and st["slot_capacity"] == L["dst"].size
    rows = np.repeat(np.arange(n), L["deg"])
    pos = np.arange(used) - np.repeat(np.cumsum(L["deg"]) - L["deg"], L["deg"])
    x = L["off"][rows] + pos
    assert st["m_edges"] == int((L["cap"][x] > 0).sum())
    su, sv, scap, _ = S.residual()                   # used slots in slot order
    np.testing.assert_array_equal(su, rows)
    np.testing.assert_array_equal(sv, L["dst"][x])
    np.testing.assert_array_equal(scap, L["cap"][x])
    chk = S.check()                                  # reverse indices and pair sums of every slot
    assert chk["pair_violations"] == 0 and chk["excess_mismatch"] == 0 and chk["active"] == 0, chk
    # the spare slots are where the host leaves them: insertions find their room
    rng = np.random.default_rng(12)
    S.update(rng.integers(0, n, 200), rng.integers(0, n, 200), rng.integers(0, 9, 200))
    assert S.check()["pair_violations"] == 0
    S.close()


def test_device_layout_refuses_what_the_host_refuses():
    n, u, v, c = _random(3000, 20000, 13)
    for field, at, bad, code in (("u", 77, 3000, native.ERR_INVALID), ("v", 19999, -1, native.ERR_INVALID),
                                 ("c", 0, -5, native.ERR_INVALID)):
        a = {"u": u.copy(), "v": v.copy(), "c": c.copy()}
        a[field][at] = bad
        with pytest.raises(native.MaxflowError) as e:
            native.Solver(n, a["u"], a["v"], a["c"], 0, n - 1)
        assert e.value.code == code
    big = c.copy()
    u2, v2 = u.copy(), v.copy()
    u2[:2], v2[:2], big[:2] = 5, 6, 2 ** 30 + 1            # parallel edges above INT32_MAX together
    with pytest.raises(native.MaxflowError) as e:
        native.Solver(n, u2, v2, big, 0, n - 1)
    assert e.value.code == native.ERR_TOO_LARGE
    u2[:2], v2[:2] = [5, 6], [6, 5]                        # the two directions of a pair
    with pytest.raises(native.MaxflowError) as e:
        native.Solver(n, u2, v2, big, 0, n - 1)
    assert e.value.code == native.ERR_TOO_LARGE
