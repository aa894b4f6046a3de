"""Slot rings shared by several consumer groups, on the CPU: an exhaustive
model of the ring that hands the states of one pulse after the other to the
updating warps of the digit-sliced batches (csrc/dig.cuh).

A slot's barrier counts phases; a waiter names only the parity of the phase it
wants, so a wait returns whenever the barrier's current phase has the other
parity: rightly when the phase it wants has just completed, wrongly when that
phase is still two behind.  The copies of several slots are in flight at once
and may land in any order."""
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DIG = open(os.path.join(ROOT, "paper_1201_6062_gb300", "csrc", "dig.cuh")).read()


def constant(name):
    return int(re.search(r"\b%s = (\d+)" % name, DIG).group(1))


def explore(slots, groups, tiles, first=None):
    """Every interleaving of a producer, copies in flight and `groups` consumers that take the items of a
    tile in turn (item p of a tile: group p % groups) and start a tile when all have finished the one
    before.  Returns the set of faults met: "early" (a wait returned although the copies of its item had
    not landed), "stuck" (nothing can move before all items are consumed) and "drain": had the kernel given
    up here, waiting for items first(issued) to issued - 1 would miss copies in flight, or not return once
    they have landed."""
    bounds = [0]
    for n in tiles:
        bounds.append(bounds[-1] + n)
    owner = {}
    for t, n in enumerate(tiles):
        for p in range(n):
            owner[bounds[t] + p] = (t, p % groups)
    items = [[i for i in range(bounds[-1]) if owner[i][1] == g] for g in range(groups)]
    faults, seen = set(), set()
    start = (0, frozenset(), (0,) * slots, (0,) * slots, (0,) * groups)
    todo = [start]
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        # issued items; items in flight; completed `full` and `empty` phases per slot; items taken per group
        issued, flight, full, empty, taken = state
        moves = []
        if first is not None:
            landed = list(full)
            for i in flight:
                landed[i % slots] += 1
            drained = range(first(issued), issued)
            if any(i not in drained for i in flight) or any(landed[q % slots] % 2 == q // slots % 2 for q in drained):
                faults.add("drain")
        if issued < bounds[-1]:
            s, k = issued % slots, issued // slots
            if k == 0 or empty[s] % 2 != (k - 1) % 2:           # parity wait for the release of item issued - slots
                moves.append((issued + 1, flight | {issued}, full, empty, taken))
        for i in flight:
            f = list(full)
            f[i % slots] += 1
            moves.append((issued, flight - {i}, tuple(f), empty, taken))
        done = [items[g][:taken[g]] for g in range(groups)]
        for g in range(groups):
            if taken[g] == len(items[g]):
                continue
            i = items[g][taken[g]]
            t = owner[i][0]
            if any(owner[j][0] < t and j not in done[h] for h in range(groups) for j in items[h]):
                continue                                        # the tile before is not handed over
            s, k = i % slots, i // slots
            if full[s] % 2 == k % 2:
                continue                                        # the wait goes on
            if full[s] != k + 1:
                faults.add("early")
                continue
            e = list(empty)
            e[s] += 1
            moves.append((issued, flight, full, tuple(e), tuple(v + (h == g) for h, v in enumerate(taken))))
        if not moves and sum(taken) < bounds[-1]:
            faults.add("stuck")
        todo += moves
    return faults


@pytest.mark.parametrize("tiles", [(13,), (5, 6, 3), (1, 1, 7), (2, 3, 4)])
def test_no_wait_of_the_state_slots_returns_early(tiles):
    assert explore(constant("DIG_NSU"), constant("DIG_UPD_GROUPS"), tiles) == set()


def test_the_model_sees_a_slot_that_changes_hands():
    assert "early" in explore(5, 2, (13,))
    assert explore(5, 1, (13,)) == set()
    assert explore(4, 2, (13,)) == set()


def test_the_drain_after_giving_up_ends_with_the_last_copies():
    S, G = constant("DIG_NSU"), constant("DIG_UPD_GROUPS")
    assert re.search(r"for \(int q = max\(st_issued - DIG_NSU, 0\); q < st_issued; \+\+q\)", DIG)
    assert explore(S, G, (5, 6, 3), lambda issued: max(issued - S, 0)) == set()
    # from the start of the tile on, waits for copies that landed long ago would run into their limit
    assert "drain" in explore(S, G, (13,), lambda issued: 0)
