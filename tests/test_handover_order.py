"""The two barriers over which a slot's four softmax warps hand P to the MMA thread: p_part (P of the first 96 keys; awaited in
tiles with both 64-key halves) and p_full (all of P; awaited in every tile).  A parity wait only tells a barrier's current phase
from the one before, so at no point may the MMA thread wait for a phase that the barrier is more than one completion away from.
All interleavings of a slot's warps with the MMA thread are walked through, with the order of the arrivals as the kernel has it.
The same for the barriers over which the slots hand whole output tiles to the thread that copies them out."""
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


# ---- the output's hand-over: a slot leaves a whole query tile in the stage of its unit's last key tile and says so; one thread
# copies the tiles out, unit by unit and slot by slot, and gives the stages back.  K's stage is slot 0's, V's is slot 1's.
STAGES = 2


def staged_barriers_of_the_kernel():
    """'stage' if every stage of a slot's has a barrier of its own, 'slot' if a slot has one barrier."""
    text = open(KERNEL).read()
    uses = re.findall(r"bars\.o_staged\[sl\](\[[^\]]*\])?", text)
    declared = re.search(r"uint64_t o_staged\[2\](\[ST\])?;", text)
    assert declared and len(uses) == 3, "the hand-over is not where it was"  # initialised, awaited, arrived on
    if not declared.group(1):
        return "slot"
    init, wait, arrive = uses
    assert init == "[s]" and wait == "[s]" and arrive == "[(it - 1u) % ST]" and "const uint32_t s = (it - 1u) % ST;" in text
    return "stage"


def first_staging_fault(units, barriers):
    """`units` is a list of (key tiles, slots that work, whether the output is staged).  Walks all interleavings of the MMA thread,
    the slots and the storing thread; loads are made as soon as their stage is free.  A description of the first wait that the
    storing thread could enter with its barrier a phase too far, or of a standstill; None if there is neither."""
    tiles = [(u, n == 0, n == count - 1) for u, (count, _, _) in enumerate(units) for n in range(count)]
    end, works, staged = [sum(c for c, _, _ in units[:u + 1]) for u in range(len(units))], [w for _, w, _ in units], [s for _, _, s in units]
    mma = []  # in program order: ("s" or "pv", tile, slot)
    at = 0
    for count, slots, _ in units:
        mma += [("s", at, sl) for sl in range(slots)]
        for i in range(at, at + count):
            for sl in range(slots):
                mma.append(("pv", i, sl))
                if i + 1 < at + count:
                    mma.append(("s", i + 1, sl))
        at += count
    done_at = {x: n for n, x in enumerate(mma)}  # an instruction is complete once the thread's count is beyond it
    slot_of = [[("p", i) if kind == "p" else ("out", u) for u in range(len(units)) if works[u] > sl
                for kind, i in [("p", i) for i in range(end[u] - units[u][0], end[u])] + ([("out", 0)] if staged[u] else [])] for sl in range(2)]
    store = [(u, sl) for u in range(len(units)) if staged[u] for sl in range(works[u])]
    barrier_of = lambda u, sl: (sl, (end[u] - 1) % STAGES if barriers == "stage" else 0)
    arrivals = [{}, {}]  # per slot: unit -> its place in the slot's program
    for sl in range(2):
        for n, (kind, u) in enumerate(slot_of[sl]):
            if kind == "out":
                arrivals[sl][u] = n

    def released(i, which, m, copied):
        """Whether tile i's K (0) or V (1) stage has been given back."""
        u, _, last = tiles[i]
        if last and staged[u] and which < works[u]:
            return store.index((u, which)) < copied
        return m > max(done_at["s" if which == 0 else "pv", i, sl] for sl in range(works[u]))

    def successors(state):
        m, slots, copied = state
        if m < len(mma):
            kind, i, sl = mma[m]
            free = i < STAGES or released(i - STAGES, 0 if kind == "s" else 1, m, copied)
            if free and (kind == "s" or ("p", i) in slot_of[sl][:slots[sl]]):
                yield m + 1, slots, copied
        for sl in range(2):
            if slots[sl] < len(slot_of[sl]):
                kind, x = slot_of[sl][slots[sl]]
                if m > done_at[("s", x, sl) if kind == "p" else ("pv", end[x] - 1, sl)]:
                    yield m, (slots[0] + (sl == 0), slots[1] + (sl == 1)), copied
        if copied < len(store):
            u, sl = store[copied]
            if slots[sl] > arrivals[sl][u]:
                yield m, slots, copied + 1

    seen, todo = set(), [(0, (0, 0), 0)]
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        m, slots, copied = state
        if copied < len(store):
            u, sl = store[copied]
            mine = [x for x in arrivals[sl] if barrier_of(x, sl) == barrier_of(u, sl)]
            if sum(slots[sl] > arrivals[sl][x] for x in mine) > mine.index(u) + 1:
                return f"unit {u}: the barrier of slot {sl} has run a phase ahead of the storing thread"
        following = list(successors(state))
        if not following and (m < len(mma) or copied < len(store)):
            return f"standstill after {copied} of {len(store)} copies"
        todo += following
    return None


@pytest.mark.parametrize("lengths", [(3, 1, 3), (2, 1, 1, 1, 2), (1, 1, 1, 1, 1), (2, 2, 2), (1, 2, 3, 1), (3, 3, 1, 1, 3)], ids=str)
def test_every_output_tile_is_copied_for_its_own_unit(lengths):
    order = staged_barriers_of_the_kernel()
    for kinds in itertools.product([(2, True), (1, True), (2, False)], repeat=len(lengths)):  # a pair, a single head, a cut tile
        units = [(n, *kind) for n, kind in zip(lengths, kinds)]
        assert first_staging_fault(units, order) is None, units


def test_the_walk_sees_a_slot_that_runs_ahead_of_the_copies():
    assert first_staging_fault([(3, 2, True), (1, 2, True), (3, 2, True)], "slot") is not None
    assert first_staging_fault([(2, 2, True)] * 4, "slot") is None
