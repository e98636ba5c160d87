"""Every order in which a few blocks can run through the barriers of a launch while a
yield request comes in: all blocks take the same decision at every barrier, none is left
waiting, and a request that is set before a barrier's first arrival stops it.  The rules
are those of the kernels (csrc/mh_barrier.h), compiled for the host.  A flag that does not
name its barrier fails the same search."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("barrier")
    src, lib = d / "rules.cpp", d / "rules.so"
    src.write_text('#include "mh_barrier.h"\n'
                   'extern "C" unsigned flag_of(unsigned a, unsigned n) { return mh::yield_flag(a, n); }\n'
                   'extern "C" int stops(unsigned f, unsigned o, unsigned n) { return mh::yield_stops(f, o, n); }\n')
    inc = os.path.join(ROOT, "paper_2603_16721_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", inc, "-o", str(lib), str(src)], check=True)
    so = ctypes.CDLL(str(lib))
    return so.flag_of, lambda f, o, n: bool(so.stops(f, o, n))


def _search(flag_of, stops, n, barriers):
    """All interleavings of n blocks; returns the first fault found, or None."""
    SAMPLE, COUNT, RAISE, ARRIVE, WAIT, READ, DONE = range(7)
    # a block: (place, barrier, what it read, stopped at or -1); then arrived, flag, request
    # set, first barrier that no block had sampled for by then
    start = (tuple((SAMPLE, 0, 0, -1) for _ in range(n)), 0, 0, False, -1)
    seen, todo = {start}, [start]
    while todo:
        state = todo.pop()
        blocks, arrived, flag, req, due = state
        nxt = [] if req else [(blocks, arrived, flag, True, max(b[1] + (b[0] != SAMPLE) for b in blocks))]
        for i, (at, k, v, end) in enumerate(blocks):
            a, f = arrived, flag
            if at == SAMPLE:
                b = (COUNT if req else ARRIVE, k, 0, end)
            elif at == COUNT:
                b = (RAISE, k, arrived, end)
            elif at == RAISE:
                f, b = flag_of(v, n), (ARRIVE, k, 0, end)
            elif at == ARRIVE:
                a, b = arrived + 1, (WAIT, k, arrived, end)
                assert arrived // n == k
            elif at == WAIT and arrived >= (k + 1) * n:
                b = (READ, k, v, end)
            elif at == READ:
                if stops(flag, v, n):
                    b = (DONE, k, 0, k)
                elif k + 1 == barriers:
                    b = (DONE, k, 0, -1)
                else:
                    b = (SAMPLE, k + 1, 0, -1)
            else:
                continue
            nxt.append((blocks[:i] + (b,) + blocks[i + 1:], a, f, req, due))
        if all(b[0] == DONE for b in blocks):
            ends = {b[3] for b in blocks}
            if len(ends) > 1:
                return "blocks stop at different barriers"
            if req and due < barriers and not 0 <= ends.pop() <= due:
                return "a request was missed"
        elif all(b[0] in (DONE, WAIT) and (b[0] == DONE or arrived < (b[1] + 1) * n) for b in blocks):
            return "a block waits for ever"
        for s in nxt:
            if s not in seen:
                seen.add(s)
                todo.append(s)
    return None


@pytest.mark.parametrize("n,barriers", [(1, 3), (2, 4), (3, 3)])
def test_all_blocks_stop_together(rules, n, barriers):
    assert _search(*rules, n, barriers) is None


def test_a_flag_without_its_barrier_does_not(rules):
    assert _search(lambda a, n: 1, lambda f, o, n: f != 0, 2, 3) == "a block waits for ever"
