"""The first CTA's hand-over of its state at consecutive grid barriers, on the CPU.

Every interleaving of the first CTA (which writes its state, arrives, and waits)
and another one (which arrives, waits and reads), with as many copies as the
header declares: the reader always gets the whole state of its own barrier.
"""
import os
import subprocess

from paper_2511_01235_gb300 import build_ext

PROBE = '#include <cstdio>\n#include "mf_internal.h"\nint main() { std::printf("%d", (int)(sizeof(MfCtrl::jd) / sizeof(MfDesc))); }\n'


def _copies(tmp_path):
    (tmp_path / "probe.cpp").write_text(PROBE)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build_ext._nvcc())))
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), "-I", build_ext.CSRC,
                           str(tmp_path / "probe.cpp"), "-o", str(tmp_path / "probe")])
    return int(subprocess.check_output([str(tmp_path / "probe")], text=True))


def _torn_reads(copies, barriers=5):
    """Reads that met another barrier's words, over all interleavings; a copy is two words."""
    # first CTA: per barrier two writes, arrive, wait.  Reader: arrive, wait, two reads.
    W = [(op, k) for k in range(barriers) for op in ("w0", "w1", "arrive", "wait")]
    R = [(op, k) for k in range(barriers) for op in ("arrive", "wait", "r0", "r1")]
    bad = set()
    seen = set()
    stack = [(0, 0, 0, 0, ((-1, -1),) * copies)]
    while stack:
        st = stack.pop()
        if st in seen:
            continue
        seen.add(st)
        i, j, aw, ar, mem = st                      # places, arrivals of either, words
        if i < len(W):
            op, k = W[i]
            if op[0] == "w" and op != "wait":
                m = [list(c) for c in mem]
                m[k % copies][int(op[1])] = k
                stack.append((i + 1, j, aw, ar, tuple(map(tuple, m))))
            elif op == "arrive":
                stack.append((i + 1, j, aw + 1, ar, mem))
            elif ar > k:
                stack.append((i + 1, j, aw, ar, mem))
        if j < len(R):
            op, k = R[j]
            if op == "arrive":
                stack.append((i, j + 1, aw, ar + 1, mem))
            elif op == "wait":
                if aw > k:
                    stack.append((i, j + 1, aw, ar, mem))
            else:
                if mem[k % copies][int(op[1])] != k:
                    bad.add((k, op))
                stack.append((i, j + 1, aw, ar, mem))
    return bad


def test_every_reader_gets_the_state_of_its_own_barrier(tmp_path):
    assert _torn_reads(1)                           # one copy is overwritten under a slow reader
    assert not _torn_reads(_copies(tmp_path))
