"""The hand-over of scores and probabilities in the forward kernel's tensor-core attention items as a protocol of parity waits,
every interleaving walked on the CPU: a waiter that follows a barrier must not be passed by two of its phases (its wait would
then never end), nor let through a phase early.  The number of P tiles and of p_ready barriers are the kernel's own."""
import os
import re

import pytest

SRC = open(os.path.join(os.path.dirname(__file__), "..", "paper_2311_04951_b200", "csrc", "persistent.cuh")).read()


def kernel_constants(rows_padded):
    tiles = re.search(r"tc_p_tiles\(int rp\) \{ return rp == 16 \? (\d+) : (\d+); \}", SRC)
    ready = re.search(r"AB_P_READY = AB_S_FULL \+ 2,.*?AB_O_DONE(?: = AB_P_READY \+ (\d+))?\b", SRC, re.S)
    return int(tiles.group(1 if rows_padded == 16 else 2)), int(ready.group(1) or 1)


def walk(n_chunks, p_tiles, p_ready_barriers):
    """Roles: the MMA issuer, the tensor core (completes what was issued in order, at any later time) and the softmax threads
    (within a chunk of each other, so they act as one).  Returns what can go wrong, over all interleavings."""
    issuer = [("S", 0)]
    for c in range(n_chunks):
        issuer += ([("S", c + 1)] if c + 1 < n_chunks else []) + [("wait", "p", c), ("PV", c)]
    softmax = []
    for c in range(n_chunks):
        softmax += [("wait", "s", c)] + ([("wait", "o", c - p_tiles)] if c >= p_tiles else []) + [("arrive", c)]
    softmax += [("wait", "o", n_chunks - 1)]
    stride = {"s": 2, "o": 2, "p": p_ready_barriers}
    wrong, seen, stack = set(), set(), [(0, 0, 0)]  # issuer step, operations the tensor core has completed, softmax step
    while stack:
        state = stack.pop()
        if state in seen:
            continue
        seen.add(state)
        i, t, f = state
        issued = [x for x in issuer[:i] if x[0] in ("S", "PV")]
        done = {"s": [x[1] for x in issued[:t] if x[0] == "S"], "o": [x[1] for x in issued[:t] if x[0] == "PV"],
                "p": [x[1] for x in softmax[:f] if x[0] == "arrive"]}

        def passes(kind, c):  # parity wait for the phase of chunk c on barrier c % stride
            n = stride[kind]
            completed, phase = sum(k % n == c % n for k in done[kind]), c // n
            if (completed & 1) == (phase & 1):
                return False
            if completed <= phase:
                wrong.add(("early", kind, c))
            return True

        nxt = []
        if i < len(issuer) and (issuer[i][0] != "wait" or passes(*issuer[i][1:])):
            nxt.append((i + 1, t, f))
        if t < len(issued):
            nxt.append((i, t + 1, f))
        if f < len(softmax) and (softmax[f][0] != "wait" or passes(*softmax[f][1:])):
            nxt.append((i, t, f + 1))
        if not nxt and (i < len(issuer) or f < len(softmax)):
            wrong.add(("stuck", issuer[i] if i < len(issuer) else None, softmax[f] if f < len(softmax) else None))
        stack += nxt
    return wrong


@pytest.mark.parametrize("rows_padded", [16, 32])
@pytest.mark.parametrize("n_chunks", [1, 2, 3, 7])
def test_no_waiter_is_passed_by_two_phases(rows_padded, n_chunks):
    assert walk(n_chunks, *kernel_constants(rows_padded)) == set()


def test_the_walk_finds_a_barrier_that_is_one_too_few():
    assert any(w[0] == "stuck" for w in walk(3, p_tiles=2, p_ready_barriers=1))
