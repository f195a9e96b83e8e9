"""The load ring of the chunked prefill, explored on the CPU: two sets of warps take alternate chunks of a ring whose depth is
odd, and a wait names its phase by the parity alone.  Whatever the order in which copies land, no set may be let through to a
chunk whose copy has not landed, and none may wait for a phase that has passed."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_12077_b200", "csrc")
CHUNKS = 14


def constant(name, default=None):
    m = re.search(r"constexpr int %s = (\d+);" % name, open(os.path.join(CSRC, "wkv6_chunked.cuh")).read())
    return int(m.group(1)) if m else default


def walk(depth, sets, barrier, before, start):
    """Explores every order of events.  barrier(c): the barrier chunk c's copy completes a phase of; before[b]: the phases of it
    completed at the start; start(c): the parity chunk c's set waits for there.  Chunk c is requested once chunk c - depth has
    been released (scaled, and all before it: the products run in order).  Returns a chunk that was started before its copy had
    landed, -1 if all chunks can stay unscaled for good, or None."""
    seen, todo, finished = set(), [(0, tuple(range(sets)))], False      # copies landed (bits), each set's next chunk
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        landed, at = state
        finished |= min(at) >= CHUNKS
        requested, more = min(CHUNKS, min(at) + depth), False
        for c in range(requested):
            if not landed >> c & 1:
                todo.append((landed | 1 << c, at))
                more = True
        for e, c in enumerate(at):
            if c >= CHUNKS:
                continue
            done = before.get(barrier(c), 0) + sum(landed >> i & 1 for i in range(CHUNKS) if barrier(i) == barrier(c))
            if (done & 1) != start(c):
                if not landed >> c & 1:
                    return c
                todo.append((landed, at[:e] + (c + sets,) + at[e + 1:]))
                more = True
        if not more and min(at) < CHUNKS:
            return -1
    return None if finished else -1


def one_barrier_per_stage(depth, sets):
    return walk(depth, sets, lambda c: c % depth, {}, lambda c: c // depth & 1)


def test_the_model_sees_a_stale_phase():
    # one barrier per stage: a late first copy lets a set read the stage it is still landing in
    assert one_barrier_per_stage(5, 2) is not None
    assert one_barrier_per_stage(4, 2) is None               # an even depth gives every set stages of its own


def test_no_set_is_let_through_early():
    depth, sets, step = constant("NS"), constant("N_ESET"), constant("STAGE_STEP")
    if step is None:
        assert one_barrier_per_stage(depth, sets) is None
        return
    parity = {}                                              # as a set's loop counts: the next stage each time, a flip at the wrap
    for e in range(sets):
        s, ph = step * e, 0
        for c in range(e, CHUNKS, sets):
            assert s == step * c % depth
            assert ph == ((c >> 1) + (c & 1) * step) // depth & 1        # (as the producer counts when it leaves)
            parity[c] = ph
            s += 1
            if s == depth:
                s, ph = 0, ph ^ 1
    ahead = {(1, s): 1 for s in range(step)}
    assert walk(depth, sets, lambda c: (c % sets, step * c % depth), ahead, parity.get) is None
    assert walk(depth, sets, lambda c: (c % sets, step * c % depth), {}, parity.get) is not None        # (they have to be ahead)
