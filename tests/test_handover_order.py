"""The two barriers over which a slot's four softmax warps hand P to the MMA thread: p_part (P of the first 96 keys; awaited in
tiles with both 64-key halves) and p_full (all of P; awaited in every tile).  A parity wait only tells a barrier's current phase
from the one before, so at no point may the MMA thread wait for a phase that the barrier is more than one completion away from.
All interleavings of a slot's warps with the MMA thread are walked through, with the order of the arrivals as the kernel has it."""
import itertools
import os
import re

import pytest

import paper_2510_25600_b200

KERNEL = os.path.join(os.path.dirname(paper_2510_25600_b200.__file__), "csrc", "prefill_tc.cu")
WARPS = 4
FULL, HALF, EXACT = "full", "half", "exact"  # tile with both halves; with one; with both, redone against its maximum


def arrivals_of_the_kernel():
    """Kind of tile -> the barriers a warp arrives on, in program order."""
    text = open(KERNEL).read()
    fast = text[text.index("bool exact = false;"):text.index("if (exact) {")]
    end = text[text.index("l_sum += l_tile;"):]
    end = end[:end.index("++t;")]
    in_both = re.findall(r"mbar_arrive\((part|full)_bar\)", fast)  # a tile with both halves, on the way
    at_end = []
    for m in re.finditer(r"(if \([^;{]*?\) )?mbar_arrive\((part|full)_bar\)", end):
        at_end.append((m.group(2), bool(m.group(1))))  # (barrier, only in the other kinds of tile)
    assert in_both == ["part"] and sorted(b for b, _ in at_end) == ["full", "part"], "the hand-over is not where it was"
    rest = [b for b, _ in at_end]
    return {FULL: ["part"] + [b for b, only in at_end if not only], HALF: rest, EXACT: rest}


def first_fault(tiles, order):
    """A description of the first wait of the MMA thread that falls through, over all interleavings; None if there is none."""
    n = len(tiles)
    program = [(t, b) for t, kind in enumerate(tiles) for b in order[kind]]             # of a warp
    waits = [(t, b) for t, kind in enumerate(tiles) for b in (["full"] if kind == HALF else ["part", "full"])]  # of the MMA thread
    seen, todo = set(), [((0,) * WARPS, 0)]
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        pcs, w = state
        done = {b: sum(sum(x == b for _, x in program[:pc]) for pc in pcs) for b in ("part", "full")}
        for i, pc in enumerate(pcs):
            # S of tile t is issued behind P V of tile t - 1, that is behind all of the MMA thread's waits for it
            if pc < len(program) and all(t >= program[pc][0] for t, _ in waits[w:]):
                todo.append((tuple(sorted(pcs[:i] + (pc + 1,) + pcs[i + 1:])), w))
        if w < len(waits):
            t, b = waits[w]
            phase = done[b] // WARPS  # the barrier's current phase; the wait returns when its parity is not t's
            if phase % 2 != t % 2:
                if phase <= t:
                    return f"tile {t} ({tiles[t]}): the wait for {b} falls through in phase {phase}"
                if phase > t + 1:
                    return f"tile {t}: {b} has run ahead"
                if not all(any(p == (t, b) for p in program[:pc]) for pc in pcs):
                    return f"tile {t}: {b} completed without every warp"
                todo.append((pcs, w + 1))
    return None


@pytest.mark.parametrize("tiles", list(itertools.product([FULL, HALF, EXACT], repeat=4)), ids="-".join)
def test_every_wait_for_p_is_for_its_own_tile(tiles):
    assert first_fault(tiles, arrivals_of_the_kernel()) is None


def test_the_walk_sees_an_arrival_that_comes_too_late():
    late = {FULL: ["part", "full"], HALF: ["full", "part"], EXACT: ["part", "full"]}
    assert first_fault((HALF, FULL), late) is not None
