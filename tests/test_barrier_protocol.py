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
    parity passes when the phase in progress has the other one."""
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
