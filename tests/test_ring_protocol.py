"""The load ring of the chunked prefill, explored on the CPU: two sets of warps take alternate chunks of a ring whose depth is
odd, so a set meets only every other phase of a stage's barrier, and a wait names its phase by the parity alone.  Whatever
the order in which copies land, no set may be let through to a chunk whose copy has not landed."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_12077_b200", "csrc")


def constant(name, default=None):
    m = re.search(r"constexpr int %s = (\d+);" % name, open(os.path.join(CSRC, "wkv6_chunked.cuh")).read())
    return int(m.group(1)) if m else default


def let_through_early(depth, sets, ahead, chunks=13):
    """A chunk that a set starts before its copy has landed, in some order of events; None if there is none.  Chunk c is
    requested once chunk c - depth has been released (scaled, and all before it: the products run in order) and the copy of
    chunk c - ahead has landed."""
    seen, todo = set(), [(0, tuple(range(sets)))]            # copies landed (bits), each set's next chunk
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        landed, at = state
        released = min(at)                                   # chunks below this one have been scaled
        requested = 0
        while requested < chunks and requested < released + depth and (requested < ahead or landed >> (requested - ahead) & 1):
            requested += 1
        for c in range(requested):
            if not landed >> c & 1:
                todo.append((landed | 1 << c, at))
        for e, c in enumerate(at):
            if c >= chunks:
                continue
            done = sum(landed >> i & 1 for i in range(c % depth, chunks, depth))       # phases of the stage's barrier completed
            if (done & 1) != (c // depth & 1):               # the wait for parity (c / depth) & 1 returns
                if not landed >> c & 1:
                    return c
                todo.append((landed, at[:e] + (c + sets,) + at[e + 1:]))
    return None


def test_the_model_sees_a_stale_phase():
    # without a limit on how far copies run ahead, a late first copy lets a set read the stage it is still landing in
    assert let_through_early(5, 2, 5) is not None
    assert let_through_early(4, 2, 4) is None                # an even depth gives every set stages of its own


def test_no_set_is_let_through_early():
    depth, sets = constant("NS"), constant("N_ESET")
    assert let_through_early(depth, sets, constant("LOAD_AHEAD", depth)) is None
