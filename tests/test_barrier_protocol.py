"""Barrier protocols that no run can be made to break on purpose, checked on the CPU: every order in which the roles of a CTA can
get ahead of one another is walked through on a model of the barriers."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24899_b200", "csrc")


def _enum(text, prefix):
    """Values of the enum whose members start with `prefix` (plain numbers)."""
    body = next(m.group(1) for m in re.finditer(r"enum \{([^}]*)\};", text) if prefix in m.group(1))
    return {k: int(v) for k, v in re.findall(r"(\w+) = (\d+)", body)}


def _stuck_state(roles, counts):
    """First state found in which some role is not through and none can move, or None.

    A role is a list of steps: ("wait", barrier, parity), ("arrive", barrier) or ("commit", barrier); commits complete in the order
    in which they were made, at any later time.  A barrier's phase completes after counts[barrier] arrivals, and a wait for a
    parity passes when the phase in progress has the other one.  A wait may name the phase it is meant for as well
    ("wait", barrier, parity, phase): one that passes before that phase is over is returned like a state where all are stuck."""
    names = sorted(counts)
    start = (tuple(0 for _ in roles), tuple((0, 0) for _ in names), ())
    seen, todo = {start}, [start]
    while todo:
        pos, bars, queue = todo.pop()
        moves = []

        def arrived(b):
            i = names.index(b)
            phase, n = bars[i]
            new = (phase + 1, 0) if n + 1 == counts[b] else (phase, n + 1)
            return bars[:i] + (new,) + bars[i + 1:]

        for r, steps in enumerate(roles):
            if pos[r] == len(steps):
                continue
            step = steps[pos[r]]
            ahead = pos[:r] + (pos[r] + 1,) + pos[r + 1:]
            if step[0] == "wait":
                if (bars[names.index(step[1])][0] & 1) != step[2]:
                    if len(step) > 3 and bars[names.index(step[1])][0] <= step[3]:
                        return pos, bars
                    moves.append((ahead, bars, queue))
            elif step[0] == "arrive":
                moves.append((ahead, arrived(step[1]), queue))
            else:
                moves.append((ahead, bars, queue + (step[1],)))
        if queue:
            moves.append((pos, arrived(queue[0]), queue[1:]))
        if not moves and any(p < len(s) for p, s in zip(pos, roles)):
            return pos, bars
        for m in moves:
            if m not in seen:
                seen.add(m)
                todo.append(m)
    return None


@pytest.mark.parametrize("tiles", [1, 2, 3, 6])
def test_key_side_gradient_at_d64_finishes_in_every_order(tiles):
    """bsk_kernel: two compute threads stand for the 512, the issuing lane's steps as in its loop (the loads are taken to be there)."""
    with open(os.path.join(CSRC, "backward_tensor_d64.cu")) as f:
        e = _enum(f.read(), "K_XRDY")
    slots = e["K_DONE"] - e["K_XRDY"]
    assert e["K_BARS"] - e["K_DONE"] == 2 and e["K_XRDY"] - e["K_AT"] == 2

    def ready(t):
        return "x%d" % (t % slots), (t // slots) & 1

    thread, lane = [], [("commit", "at0")]
    for t in range(tiles):
        thread.append(("wait", "at%d" % (t & 1), (t >> 1) & 1))
        if t > 1:
            thread.append(("wait", "done%d" % (t & 1), ((t - 2) >> 1) & 1))
        thread.append(("arrive", ready(t)[0]))
        if t + 1 < tiles:
            lane.append(("commit", "at%d" % ((t + 1) & 1)))
        if t > 0 and t + 2 < tiles:
            lane.append(("wait", "done%d" % ((t - 1) & 1), ((t - 1) >> 1) & 1))
        lane.append(("wait",) + ready(t))
        lane.append(("commit", "done%d" % (t & 1)))
    for t in range(max(0, tiles - 2), tiles):
        thread.append(("wait", "done%d" % (t & 1), (t >> 1) & 1))
    counts = {"at0": 1, "at1": 1, "done0": 1, "done1": 1, **{"x%d" % i: 2 for i in range(slots)}}
    assert _stuck_state([thread, thread, lane], counts) is None


def test_dependents_are_let_in_only_by_ctas_that_own_their_tensor_memory():
    """In every kernel that allocates tensor memory the allocating warp alone calls griddep_launch, behind the allocation (a dependent
    CTA that took the columns first would wait for this kernel while this one waits for the columns, without a limit)."""
    checked = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, name)) as f:
            kernels = re.split(r"\b__global__\b", re.sub(r"//[^\n]*", "", f.read()))[1:]
        for body in kernels:
            if "griddep_launch()" not in body or "tmem_alloc(" not in body:
                continue
            assert body.count("griddep_launch()") == 1 and body.count("tmem_alloc(") == 1, (name, body[:120])
            assert re.search(r"tmem_alloc\([^;]*\); tmem_relinquish\(\); griddep_launch\(\);", body), (name, body[:120])
            checked += 1
    assert checked >= 8


def _query_stage(tiles, chunks, groups, shared, threads, ring, units=1, own_tail=True):
    """The query stage with a one-layer map, unit after unit (the last one of `groups` groups, the others of two): compute threads (one or
    two stand for a group's), the warp that issues what writes the score columns (shared by the groups at d = 128, with `own_tail` only
    in the key loop),
    the warp that issues what accumulates into O and, with `ring`, the loads."""
    n, counts = tiles + chunks, {}
    compute, score, accum, load = [[], []], [], [], []
    # ring items of a unit in the order they are loaded: K_0, then K_j+1 and V_j; W_0, the last V; then W_c+1 and S_c
    order = ([("k", 0)] if tiles else []) + [x for j in range(tiles - 1) for x in (("k", j + 1), ("v", j))]
    order += [("k", tiles)] * (chunks > 0) + [("v", tiles - 1)] * (tiles > 0)
    order += [x for c in range(chunks - 1) for x in (("k", tiles + c + 1), ("v", tiles + c))] + [("v", n - 1)] * (chunks > 0)
    assert sorted(order) == sorted([(x, i) for x in "kv" for i in range(n)])
    for u in range(units):
        ng = groups if u + 1 == units else 2

        def at(x, i):
            return u * 2 * n + order.index((x, i))

        def full(x, i):
            return [("wait", "full%d" % (at(x, i) % 3), (at(x, i) // 3) & 1, at(x, i) // 3)] if ring else []

        def release(x, i):
            return [("commit", "empty%d" % (at(x, i) % 3))] if ring else []

        def wait(b, g, phase):
            return [("wait", "%s%d" % (b, g), phase & 1, phase)] if phase >= 0 else []

        for i in range(n):
            ph = u * n + i
            for g in range(ng):
                # the threads
                steps = compute[g]
                steps += wait("s", g, ph)
                if i > tiles:                              # feature rows: the tile they go to is free first, then the columns are read
                    steps += wait("pf", g, ph - 1)
                steps.append(("arrive", "sf%d" % g))
                if i <= tiles:
                    steps += wait("pf", g, ph - 1)
                steps.append(("arrive", "p%d" % g))
                if i + 1 == n:
                    steps += wait("o", g, u)
                # what writes the score columns
                score += full("k", i) if g == 0 else []
                if not shared or (own_tail and (i > tiles or tiles == 0)):
                    score += wait("sf", g, ph - 1)
                elif g == 1:
                    score += wait("sf", 0, ph) if i < tiles or not own_tail else wait("pl", 0, u)
                else:
                    score += wait("sf", 0, ph - 1) if i == 0 and own_tail else []
                    score += wait("sf", 1 if ng == 2 or i == 0 else 0, ph - 1)
                score.append(("commit", "s%d" % g))
                # what accumulates
                accum += full("v", i) if g == 0 else []
                accum += wait("p", g, ph) + [("commit", "pf%d" % g)] + ([("commit", "o%d" % g)] if i + 1 == n else [])
                accum += [("commit", "pl0")] if shared and own_tail and chunks and g == 1 and i + 1 == tiles else []
            score += release("k", i)
            accum += release("v", i)
    for g in range(2 if units > 1 else groups):
        counts.update({"s%d" % g: 1, "sf%d" % g: threads, "p%d" % g: threads, "pf%d" % g: 1, "o%d" % g: 1, "pl0": 1})
    if ring:
        counts.update({"%s%d" % (x, s): 1 for x in ("full", "empty") for s in range(3)})
        for item in range(2 * n * units):
            load += ([("wait", "empty%d" % (item % 3), (item // 3 + 1) & 1)] if item >= 3 else []) + [("arrive", "full%d" % (item % 3))]
    roles = [steps for g in range(2) for steps in [compute[g]] * threads if steps] + [score, accum]
    return roles + ([load] if ring else []), counts


@pytest.mark.parametrize("tiles,chunks,units", [(1, 0, 1), (3, 0, 1), (0, 1, 1), (0, 3, 1), (1, 1, 1), (2, 1, 1), (3, 2, 1), (1, 0, 3), (2, 0, 2), (0, 1, 3),
                                                (1, 1, 3), (2, 1, 2), (1, 2, 2)])
@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("shared,own_tail", [(False, True), (True, True), (True, False)])
@pytest.mark.parametrize("threads,ring", [(2, False), (1, True)])
def test_query_stage_finishes_in_every_order(tiles, chunks, units, groups, shared, own_tail, threads, ring):
    assert _stuck_state(*_query_stage(tiles, chunks, groups, shared, threads, ring, units, own_tail)) is None


def test_the_model_finds_what_it_is_there_for():
    """Feature rows handed over without a look at whether the last tile's product has completed; group 1's feature columns taken with a look
    at the last phase of a barrier whose phases were not all looked at."""
    roles, counts = _query_stage(2, 1, 1, False, 2, False)
    late = [i for i, step in enumerate(roles[0]) if step[:2] == ("wait", "pf0")][-1]
    roles[:2] = [roles[0][:late] + roles[0][late + 1:]] * 2
    assert _stuck_state(roles, counts) is not None
    roles, counts = _query_stage(3, 1, 2, True, 1, False)
    at = [i for i, step in enumerate(roles[-2]) if step[1] == "pl0"][0]
    roles[-2][at] = ("wait", "pf1", 0, 2)
    assert _stuck_state(roles, counts) is not None
