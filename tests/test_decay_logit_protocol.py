"""The hand-overs of the decay-logit kernel (csrc/decay_logit.cuh), walked on the CPU: any warp may be held up at any point while the
others go on as far as they can.  Nobody may read a value that has been overwritten or is not there yet, and no wait (which names its
phase by the parity alone) may be let through early or come when its phase is over and the next one with it."""
import os
import re
from collections import defaultdict

import pytest

SRC = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_12077_b200", "csrc", "decay_logit.cuh")).read()
NSET, WARPS = 4, 2                                           # (two of a set's four warps: one held up, one going on)
TILES = 3


def as_written():
    """(accumulators of l / d, whether the issuers of h B take turns, whether h1 and h2 have a barrier each, whether a tile's first
    product waits for the h2 before it)"""
    issuer = SRC[SRC.index("MMA issuer: sum += z A_d"):SRC.index("MMA issuers: l = h1 B_d")]
    assert int(re.search(r"constexpr int DL_NSET = (\d+);", SRC).group(1)) == NSET
    return (int(re.search(r"constexpr int DL_NACC = (\d+);", SRC).group(1)), "wait_warp(DL_TURN + 1 - odd" in SRC, "DL_H2_READY" in SRC,
            "wait_warp(DL_H2_READY, ti - 1)" in issuer)


# A warp is a generator of events: ("wait", barrier, phase), ("arrive", barrier), ("read", place, value), ("write", place, value).  A
# product reads and writes where it is issued, which is the earliest it can; its commits are arrivals after it.
def sum_issuer(S, wait_h2):
    uses = defaultdict(int)
    for t in range(TILES):
        for p in range(2):
            for s in range(S):
                n = (3 * t + p) * S + s
                if wait_h2 and t and p == 0 and s == 0:
                    yield "wait", "H2", t - 1
                yield "wait", ("OP_READY", n % NSET), uses[n % NSET]
                uses[n % NSET] += 1
                yield "read", ("OP", n % NSET), n
                if s < 2:
                    yield "write", ("SUM", s), (t, p)
                yield "arrive", ("OP_FREE", n % NSET)
                if s == S - 1:
                    yield "arrive", "SUM_FULL"


def h_issuer(S, acc, turns, two, odd):
    count, j, turn = defaultdict(int), 0, 0                  # products per set, in all, of the other issuer
    for t in range(TILES):
        first = (3 * t + 1) * S
        for p in (1, 2):
            yield ("wait", "H%d" % p, t) if two else ("wait", "H", 2 * t + p - 1)
            for n in range((3 * t + p) * S, (3 * t + p + 1) * S):
                if n % 2 == odd:
                    if n - acc >= first:
                        yield "wait", ("ACC_FREE", (n - acc) % NSET), count[(n - acc) % NSET] - 1
                    if turns and n > first:
                        yield "wait", ("TURN", 1 - odd), turn - 1
                    yield "arrive", ("TURN", odd)
                    yield "read", "H", (t, p)
                    yield "write", ("ACC", j % acc), n
                    yield "arrive", ("ACC_FULL", n % NSET)
                else:
                    turn += 1
                count[n % NSET] += 1
                j += 1
        yield "arrive", "H_FREE"


def worker(S, acc, two, me):
    op, full = 0, 0
    for t in range(TILES):
        for p in range(3):
            for n in range((3 * t + p) * S, (3 * t + p + 1) * S):
                if n % NSET != me:
                    continue
                if p:
                    yield "wait", ("ACC_FULL", me), full
                    full += 1
                    yield "read", ("ACC", (n - (t + 1) * S) % acc), n
                if p < 2:                                    # (l is handed back when half the operand is written)
                    if op:
                        yield "wait", ("OP_FREE", me), op - 1
                    op += 1
                    yield "write", ("OP", me), n
                if p:
                    yield "arrive", ("ACC_FREE", me)
                if p < 2:
                    yield "arrive", ("OP_READY", me)
            if p == 2:
                continue
            yield "wait", "SUM_FULL", 2 * t + p
            if p == 0 and t:
                yield "wait", "H_FREE", t - 1
            for half in range(min(S, 2)):
                yield "read", ("SUM", half), (t, p)
            yield "write", "H", (t, p + 1)
            yield ("arrive", "H%d" % (p + 1)) if two else ("arrive", "H")


def arrivals(barrier):
    name = barrier if isinstance(barrier, str) else barrier[0]
    return {"H": NSET * WARPS, "H1": NSET * WARPS, "H2": NSET * WARPS, "H_FREE": 2, "OP_READY": WARPS, "ACC_FREE": WARPS}.get(name, 1)


def walk(S, acc, turns, two, wait_h2, held, steps):
    """Runs warp `held` for so many steps, then only the others until they are stuck, then all.  Returns what went wrong, or None, and
    whether `held` has more steps."""
    warps = [sum_issuer(S, wait_h2), h_issuer(S, acc, turns, two, 0), h_issuer(S, acc, turns, two, 1)]
    warps += [worker(S, acc, two, s) for s in range(NSET) for _ in range(WARPS)]
    nxt = [next(w, None) for w in warps]
    arrived, memory, done = defaultdict(int), {}, [0] * len(warps)

    def step(i):
        """One event of warp i: False if it has to wait, a text if that is a fault."""
        kind, what, *rest = nxt[i]
        if kind == "wait":
            complete, phase = arrived[what] // arrivals(what), rest[0]
            if complete % 2 == phase % 2:
                return "%s: phase %d is over, and %d" % (what, phase, phase + 1) if complete > phase else False
            if complete != phase + 1:
                return "%s: let through to phase %d, %d complete" % (what, phase, complete)
        elif kind == "arrive":
            arrived[what] += 1
        elif kind == "read":
            if memory.get(what) != rest[0]:
                return "%s: holds %s, not %s" % (what, memory.get(what), rest[0])
        else:
            memory[what] = rest[0]
        nxt[i] = next(warps[i], None)
        done[i] += 1
        return True

    def run(who, until=lambda: False):
        moved = True
        while moved and not until():
            moved = False
            for i in who:
                while nxt[i] is not None and not until():
                    r = step(i)
                    if r is not True:
                        if r:
                            return r
                        break
                    moved = True
        return None

    everyone, others = list(range(len(warps))), [i for i in range(len(warps)) if i != held]
    fault = run([held] + others, lambda: done[held] >= steps) or run(others) or run(everyone)
    if not fault and any(n is not None for n in nxt):
        fault = "stuck: %s" % [n for n in nxt if n is not None]
    return fault, done[held] > steps


def faults(S, *form):
    found = set()
    for held in [0, 1, 2] + [3 + WARPS * s for s in range(NSET)]:
        steps, more = 0, True
        while more:
            fault, more = walk(S, *form, held, steps)
            if fault:
                found.add(fault)
            steps += 1
    return found


@pytest.mark.parametrize("S", range(1, 10))
def test_every_hand_over_holds_whoever_is_late(S):
    assert faults(S, *as_written()) == set()


def test_the_walk_sees_what_it_is_for():
    # one barrier for h1 and h2, and nothing between a late reader of a tile's second sum and the next tile's first product
    for S in (1, 2, 3):
        assert any("SUM" in f for f in faults(S, 3, True, False, False)), S
    assert faults(4, 3, True, False, False) == set()
    # ... an issuer without a slice is not held within a phase of it
    assert any(f.startswith("H:") for f in faults(1, 3, True, False, False))
    assert any("SUM" in f for f in faults(3, 3, True, True, False))
    # three accumulators for four sets: without turns an issuer may look for a set's slice when its next has been read as well
    assert any("ACC_FREE" in f for f in faults(8, 3, False, True, True))
