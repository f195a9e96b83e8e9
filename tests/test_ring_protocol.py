"""The load ring of the chunked prefill, explored on the CPU: two sets of warps take alternate chunks of a ring whose depth is
odd, and a wait names its phase by the parity alone.  Whatever the order in which copies land, no set may be let through to a
chunk whose copy has not landed."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_12077_b200", "csrc")


def constants():
    src = open(os.path.join(CSRC, "wkv6_chunked.cuh")).read()
    depth, sets = (int(re.search(r"constexpr int %s = (\d+);" % n, src).group(1)) for n in ("NS", "N_ESET"))
    per_set = re.search(r"constexpr int N_FULL = NS % N_ESET \? N_ESET \* NS : NS;", src) is not None
    return depth, sets, sets * depth if per_set and depth % sets else depth


def let_through_early(depth, sets, barriers, chunks=13):
    """A chunk that a set starts before its copy has landed, in some order of events; None if there is none.  Chunk c completes
    phase c / barriers of barrier c % barriers, and is requested once chunk c - depth has been released (scaled, and all before
    it: the products run in order)."""
    seen, todo = set(), [(0, tuple(range(sets)))]            # copies landed (bits), each set's next chunk
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        landed, at = state
        for c in range(min(chunks, min(at) + depth)):        # requested
            if not landed >> c & 1:
                todo.append((landed | 1 << c, at))
        for e, c in enumerate(at):
            if c >= chunks:
                continue
            done = sum(landed >> i & 1 for i in range(c % barriers, chunks, barriers))     # phases of the barrier completed
            if (done & 1) != (c // barriers & 1):            # the wait for parity (c / barriers) & 1 returns
                if not landed >> c & 1:
                    return c
                todo.append((landed, at[:e] + (c + sets,) + at[e + 1:]))
    return None


def test_the_model_sees_a_stale_phase():
    # one barrier per stage: a late first copy lets a set read the stage it is still landing in
    assert let_through_early(5, 2, 5) is not None
    assert let_through_early(4, 2, 4) is None                # an even depth gives every set stages of its own


def test_no_set_is_let_through_early():
    assert let_through_early(*constants()) is None
