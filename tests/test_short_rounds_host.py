"""Short discharge rounds queue every vertex once, on the CPU.

A short round queues behind stamps or without.  The model below runs two vertices
through a round of several cycles (always behind stamps) and through short rounds,
over every interleaving of their accesses, and asks the header's own rule
(mf_round_stamps, compiled here) which kind a short round is: its list never holds
a vertex twice, and without stamps never one that has no excess.  A round of the
first cluster does without stamps by dropping the entries without excess first.
"""
import os
import subprocess

import pytest

from paper_2511_01235_gb300 import build_ext

PROBE = """
#include <cstdio>
#include "mf_internal.h"
int main() {
    for (int i = 0; i < 16; ++i) std::printf("%d\\n", mf_round_stamps(i >> 2, i >> 1 & 1, i & 1));
}
"""


@pytest.fixture(scope="module")
def stamps(tmp_path_factory):
    d = tmp_path_factory.mktemp("short")
    (d / "probe.cpp").write_text(PROBE)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build_ext._nvcc())))
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", build_ext.CSRC,
                           str(d / "probe.cpp"), "-o", str(d / "probe")])
    out = subprocess.check_output([str(d / "probe")], text=True).split()
    return lambda round_, last_short, last_stamped: out[4 * min(round_, 3) + 2 * last_short + last_stamped] == "1"


# p above u above w: p's slots to u (a slot is one push), u's to w
START = {"e": {"p": 5, "u": 1, "w": 0}, "cf": {"p": (1, 1, 2, 1), "u": (1, 2, 1, 9)}, "to": {"p": "u", "u": "w"}}
CYCLES = 2


def _long(v):
    """KERNEL_CYCLES pushes, the excess read again before each pass; queueing behind a stamp."""
    left = CYCLES
    while left:
        eu = yield ("read", v)
        if eu <= 0:
            break
        sent = 0
        while left and sent < eu:
            got = yield ("push", v, eu - sent, True)
            if not got:
                break
            sent += got
            left -= 1
        yield ("take", v, sent)
        if not sent:
            break
    if (yield ("read", v)) > 0:
        yield ("queue", v, True)


def _short(v, stamp):
    """One cycle on the excess read at first."""
    eu = yield ("read", v)
    if eu <= 0:
        return
    sent = 0
    for _ in range(2):                     # the slots of the lowest neighbour
        if sent < eu:
            sent += yield ("push", v, eu - sent, stamp)
    if (yield ("take", v, sent)) > 0:
        yield ("queue", v, stamp)


def _outcomes(state, body):
    """Next lists and states over all interleavings of one round."""
    seen, out = set(), {}

    def replay(order):
        e, cf, nxt = dict(state["e"]), dict(state["cf"]), []
        act = [body(v) for v in state["list"]]
        ask = [next(a, None) for a in act]
        for k in order:
            what, v = ask[k][0], ask[k][1]
            ans = None
            if what == "read":
                ans = e[v]
            elif what == "push":
                c = cf[v][0] if cf[v] else 0
                ans = min(ask[k][2], c)
                if ans:
                    cf[v] = cf[v][1:] if ans == c else (c - ans,) + cf[v][1:]
                    z = START["to"][v]
                    became = e[z] <= 0
                    e[z] += ans
                    if z != "w" and became and not (ask[k][3] and z in nxt):
                        nxt.append(z)
            elif what == "take":
                e[v] -= ask[k][2]
                ans = e[v]
            elif not (ask[k][2] and v in nxt):
                nxt.append(v)
            try:
                ask[k] = act[k].send(ans)
            except StopIteration:
                ask[k] = None
        key = (tuple(sorted(e.items())), tuple(sorted(cf.items())), tuple(nxt))
        return [k for k in range(len(ask)) if ask[k] is not None], key, {"e": e, "cf": cf, "list": nxt}

    stack = [()]
    while stack:
        order = stack.pop()
        live, key, st = replay(order)
        if not live:
            if key not in seen:
                seen.add(key)
                out[key] = st
        for k in live:
            stack.append(order + (k,))
    return list(out.values())


@pytest.mark.parametrize("first", ["long", "short"])
def test_a_short_rounds_list_holds_every_vertex_once(stamps, first):
    kind0 = (True, stamps(0, 0, 0)) if first == "short" else (False, False)
    states = [(dict(START, list=["u", "p"]), kind0)]
    plain = stamped = bare = 0
    for round_ in range(4):
        nxt = {}
        for st, (short, stamp) in states:
            assert len(set(st["list"])) == len(st["list"]), st
            if short and not stamp:
                assert all(st["e"][v] > 0 for v in st["list"]), st
            plain += short and not stamp
            stamped += short and stamp
            bare += any(st["e"][v] <= 0 for v in st["list"])
            for o in _outcomes(st, (lambda v: _short(v, stamp)) if short else _long):
                assert min(o["e"].values()) >= 0
                for again in (True, False) if o["list"] and not short else (True,) if o["list"] else ():
                    kind = (again, again and stamps(round_ + 1, short, stamp))     # a long round may follow too
                    nxt[(tuple(sorted(o["e"].items())), tuple(o["cf"].items()), tuple(o["list"]), kind)] = (o, kind)
                    kept = [v for v in o["list"] if o["e"][v] > 0]
                    if kind == (True, True) and kept:      # the first cluster drops the others and needs no stamps
                        k2 = dict(o, list=kept)
                        nxt[(tuple(sorted(o["e"].items())), tuple(o["cf"].items()), tuple(kept), "kept")] = (k2, (True, False))
        states = list(nxt.values())[:120]
    # the model reaches what the rule is about
    assert plain > 3 and not stamped if first == "short" else stamped > 3 and bare and plain


def test_rounds_behind_a_relabel_need_no_stamps(stamps):
    assert not any(stamps(0, a, b) for a in (0, 1) for b in (0, 1))
    assert not stamps(1, 1, 0) and stamps(1, 0, 0) and stamps(2, 1, 1)
