"""Which discharge rounds may be short ones, on the CPU.

A short round queues vertices without stamps.  The model below runs two vertices
through a round of several cycles (queued behind a stamp) and through short
rounds, over every interleaving of their accesses, and asks the header's own rule
(mf_short_may_follow, compiled here) what may come next: a short round's list
never holds a vertex twice, and never one without excess.
"""
import os
import subprocess

import pytest

from paper_2511_01235_gb300 import build_ext

PROBE = """
#include <cstdio>
#include "mf_internal.h"
int main() {
    for (int round = 0; round < 4; ++round)
        for (int last = 0; last < 2; ++last) std::printf("%d\\n", mf_short_may_follow(round, last) ? 1 : 0);
}
"""


@pytest.fixture(scope="module")
def may_follow(tmp_path_factory):
    d = tmp_path_factory.mktemp("short")
    (d / "probe.cpp").write_text(PROBE)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build_ext._nvcc())))
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", build_ext.CSRC,
                           str(d / "probe.cpp"), "-o", str(d / "probe")])
    out = subprocess.check_output([str(d / "probe")], text=True).split()
    table = {(r, k): out[2 * r + k] == "1" for r in range(4) for k in range(2)}
    return lambda round_, last_short: table[min(round_, 3), int(last_short)]


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


def _short(v):
    """One cycle on the excess read at first; queueing without a stamp."""
    eu = yield ("read", v)
    if eu <= 0:
        return
    sent = 0
    for _ in range(2):                     # the slots of the lowest neighbour
        if sent < eu:
            sent += yield ("push", v, eu - sent, False)
    if (yield ("take", v, sent)) > 0:
        yield ("queue", v, False)


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
def test_a_short_rounds_list_holds_every_vertex_once_and_with_excess(may_follow, first):
    states = [(dict(START, list=["u", "p"]), first == "short")]
    shorts = bare = 0
    for round_ in range(3):
        nxt = {}
        for st, short in states:
            if short:
                shorts += 1
                assert len(set(st["list"])) == len(st["list"]), st
                assert all(st["e"][v] > 0 for v in st["list"]), st
            else:
                bare += any(st["e"][v] <= 0 for v in st["list"])
            for o in _outcomes(st, _short if short else _long):
                assert min(o["e"].values()) >= 0
                if o["list"]:
                    # a round with short rows only: short wherever the rule lets it
                    kind = may_follow(round_ + 1, short)
                    nxt[(tuple(sorted(o["e"].items())), tuple(o["cf"].items()), tuple(o["list"]), kind)] = (o, kind)
        states = list(nxt.values())[:60]
    assert shorts > 3 if first == "short" else bare     # the model reaches what the rule is about


def test_an_iteration_may_open_with_a_short_round(may_follow):
    assert may_follow(0, 0) and may_follow(0, 1) and may_follow(2, 1)
