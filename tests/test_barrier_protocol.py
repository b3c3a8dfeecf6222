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


# ---- grid barriers whose arrivals run ahead of their waits ----
# A CTA arrives at a barrier in front of a GEMM without waiting for it (grid_arrive); the GEMM's operand issuer waits for the barrier
# named by gemm_desc's `need`, and a CTA without a share of the GEMM waits for nothing.  The counter is one sum over all
# barriers, so an arrival at barrier E + 1 must not be counted before barrier E is complete.
SEQUENTIAL_LAYER = [("gemm", 0), ("sync",), ("arrive",), ("gemm", 2), ("sync",), ("arrive",), ("gemm", 4), ("sync",), ("arrive",),
                    ("gemm", 6), ("sync",), ("arrive",)]
PARALLEL_LAYER = [("gemm", 0), ("gemm", 0), ("sync",), ("arrive",), ("gemm", 2), ("gemm", 2), ("sync",), ("arrive",)]
OVERLAPPED_ATTENTION = [("gemm", 0), ("gemm", 0), ("sync",), ("arrive",), ("signal",), ("sync",), ("arrive",)]
OVERLAPPED_OTHERS = [("gemm", 0), ("gemm", 0), ("sync",), ("arrive",), ("gemm", 2), ("gemm", 2, "signalled"), ("sync",), ("arrive",)]


def arrivals_wait_for_the_barrier_before():
    body = SRC[SRC.index("bool grid_arrive_work("):SRC.index("// Grid barrier.  Returns false")]
    wait, count = body.find("grid_poll(p, sh, epoch - 1)"), body.find("red_release_add(p.gbar")
    return 0 <= wait < count


def needs_in_the_source():
    body = SRC[SRC.index("GemmDesc gemm_desc("):SRC.index("// This CTA's contiguous share")]
    return re.findall(r"g\.need = ([^;]+);", body)


def programs(kind, layers, n_cta, idle):
    """Per CTA: the head's full barrier, the layers, a last full barrier.  `idle` CTAs have no share of any GEMM."""
    out = []
    for c in range(n_cta):
        prog, base = [("sync",)], 1
        for l in range(layers):
            layer = {"sequential": SEQUENTIAL_LAYER, "parallel": PARALLEL_LAYER,
                     "overlapped": OVERLAPPED_ATTENTION if c == 0 else OVERLAPPED_OTHERS}[kind]
            for op in layer:
                if op[0] != "gemm":
                    prog.append(op)
                elif c not in idle:
                    prog.append(("gemm", base + op[1], l + 1 if "signalled" in op else 0))  # (signals of the attention CTA before it)
            base += 8 if kind == "sequential" else 4
        out.append(prog + [("sync",)])
    return out


def walk_barriers(progs, waits_before_counting, may_give_up=()):
    """All interleavings of the CTAs' steps: announce (++epoch), [wait for the barrier before], count; a full barrier then waits for its
    own number; an operand issuer waits for `need` and reads what every CTA wrote before that barrier.  A CTA in `may_give_up` may,
    at any wait, give up: it counts no more and runs to its next full barrier, where it stops; the others' waits for it then run out.
    Returns what can go wrong."""
    n = len(progs)
    wrong, seen = set(), set()
    start = (0, 0, tuple((0, 0, 0, 0, False, False) for _ in progs))  # counted, signals; per CTA: step, stage, epoch, passed, given up, stopped
    stack = [start]
    while stack:
        state = stack.pop()
        if state in seen:
            continue
        seen.add(state)
        counted, signals, ctas = state
        hopeless = any(c[4] for c in ctas)
        moves = []

        def put(i, c, dc=0, ds=0):
            moves.append((counted + dc, signals + ds, ctas[:i] + (c,) + ctas[i + 1:]))

        def complete(i, number):  # CTA i finds `number` barriers complete
            if counted < number * n:
                return False
            if any(c[2] < number for c in ctas):
                wrong.add(("passed before all had arrived", number))
            return True

        for i, (step, stage, epoch, passed, gave_up, stopped) in enumerate(ctas):
            if stopped or step == len(progs[i]):
                continue
            op = progs[i][step]
            if gave_up:  # no work, no counting; stops at a full barrier
                put(i, (step, 0, epoch, passed, True, True) if op[0] == "sync" else (step + 1, 0, epoch, passed, True, False))
                continue
            waiting = False
            if op[0] == "signal":
                put(i, (step + 1, 0, epoch, passed, False, False), ds=1)
            elif op[0] == "gemm":
                ready = passed >= op[1] or complete(i, op[1])
                if ready and any(c[2] < op[1] for c in ctas):
                    wrong.add(("operand read before it was written", op[1]))
                if ready and signals >= op[2]:
                    put(i, (step + 1, 0, epoch, max(passed, op[1]), False, False))
                else:
                    waiting = True
            elif stage == 0:
                put(i, (step, 1, epoch + 1, passed, False, False))
            elif stage == 1:
                if not waits_before_counting or passed >= epoch - 1 or complete(i, epoch - 1):
                    put(i, (step, 2, epoch, max(passed, epoch - 1) if waits_before_counting else passed, False, False) if op[0] == "sync"
                        else (step + 1, 0, epoch, max(passed, epoch - 1) if waits_before_counting else passed, False, False), dc=1)
                else:
                    waiting = True
            elif complete(i, epoch):
                put(i, (step + 1, 0, epoch, max(passed, epoch), False, False))
            else:
                waiting = True
            if waiting and (i in may_give_up or hopeless):
                put(i, (step, 0, epoch, passed, True, False))
        if not moves and any(not c[5] and c[0] < len(progs[i]) for i, c in enumerate(ctas)):
            wrong.add(("stuck", tuple(c[0] for c in ctas)))
        stack += moves
    return wrong


def test_the_walked_needs_are_the_kernels_own():
    assert needs_in_the_source() == ["base", "base", "base + 2", "p.parallel ? base : base + 4", "p.parallel ? base + 2 : base + 6"]


@pytest.mark.parametrize("kind", ["sequential", "parallel", "overlapped"])
@pytest.mark.parametrize("n_cta,idle", [(2, ()), (2, (1,)), (3, ()), (3, (2,))])
def test_no_barrier_is_passed_before_all_have_arrived(kind, n_cta, idle):
    progs = programs(kind, 2 if n_cta == 2 else 1, n_cta, idle)
    assert walk_barriers(progs, arrivals_wait_for_the_barrier_before()) == set()


@pytest.mark.parametrize("kind", ["sequential", "parallel", "overlapped"])
@pytest.mark.parametrize("idle", [(), (1,)])
def test_a_wait_that_gives_up_ends_every_cta_and_passes_nothing_early(kind, idle):
    progs = programs(kind, 1, 2, idle)
    assert walk_barriers(progs, arrivals_wait_for_the_barrier_before(), may_give_up=(0, 1)) == set()


def test_the_walk_finds_arrivals_that_are_counted_too_early():
    """A CTA without a share of a GEMM would arrive twice where it must arrive once."""
    assert ("passed before all had arrived", 3) in walk_barriers(programs("sequential", 1, 3, (2,)), False)
