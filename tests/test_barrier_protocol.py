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
    ("wait", barrier, parity, phase): one that passes before that phase is over is returned like a state where all are stuck.  So may an
    arrival or a commit ("arrive", barrier, phase): one that counts for another phase is returned.  ("copy", barrier, phase) arrives at any
    later time, copies in any order."""
    names = sorted(counts)
    start = (tuple(0 for _ in roles), tuple((0, 0) for _ in names), (), ())
    seen, todo = {start}, [start]
    while todo:
        pos, bars, queue, flying = todo.pop()
        moves = []

        def arrived(b, meant=None):
            i = names.index(b)
            phase, n = bars[i]
            if meant not in (None, phase):
                return None
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
                    moves.append((ahead, bars, queue, flying))
            elif step[0] == "arrive":
                moves.append((ahead, arrived(*step[1:]), queue, flying))
            elif step[0] == "copy":
                moves.append((ahead, bars, queue, tuple(sorted(flying + (step[1:],)))))
            else:
                moves.append((ahead, bars, queue + (step[1:],), flying))
        if queue:
            moves.append((pos, arrived(*queue[0]), queue[1:], flying))
        for i, copy in enumerate(flying):
            moves.append((pos, arrived(*copy), queue, flying[:i] + flying[i + 1:]))
        if any(m[1] is None for m in moves):
            return pos, bars
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


def _ring(kinds):
    """Slot, barrier and phase of the ring items of a CTA in the order they are loaded, "k" for what the one issuing warp uses, "v" for the other's."""
    items, phases = [], {}
    for i, kind in enumerate(kinds):
        name = "%sfull%d" % (kind, i % 3)
        phases[name] = phases.get(name, -1) + 1
        items.append((i % 3, name, phases[name]))
    return items


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
    items = _ring([x for x, _ in order] * units)
    for u in range(units):
        ng = groups if u + 1 == units else 2

        def full(x, i):
            _, name, phase = items[u * 2 * n + order.index((x, i))]
            return [("wait", name, phase & 1, phase)] if ring else []

        def release(x, i):
            slot = items[u * 2 * n + order.index((x, i))][0]
            return [("commit", "empty%d" % slot)] if ring else []

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
        counts.update({"%s%d" % (x, s): 1 for x in ("kfull", "vfull", "empty") for s in range(3)})
        for item, (slot, name, phase) in enumerate(items):
            load += ([("wait", "empty%d" % slot, (item // 3 + 1) & 1)] if item >= 3 else []) + [("copy", name, phase)]
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


def _without_memory(roles):
    """What `_stuck_state` takes of the steps of `_race`."""
    keep = {"wait": lambda s: [("wait", s[1], s[2] & 1, s[2])], "arrive": lambda s: [s], "commit": lambda s: [s], "load": lambda s: [("copy",) + s[2:]]}
    return [[x for s in steps for x in keep.get(s[0], lambda s: [])(s)] for steps in roles]


def _race(roles):
    """Two steps that use the same memory with nothing between them that orders them, or None (after `_stuck_state` has found that every arrival
    counts for the phase it is meant for: then the order that the barriers give does not depend on who is ahead).

    Steps: ("wait", barrier, phase), ("arrive", barrier, phase); ("read", cell) and ("write", cell) of a thread; ("mma", reads, writes), a product,
    at work from its issue to some later time; ("commit", barrier, phase), which arrives once the role's products before it are
    done; ("load", cell, barrier, phase), a copy in; ("store", cell), a copy out, and ("drain",), the wait for the role's copies out.  A role's asynchronous work is
    done in order; a product may follow one of its own role over the same cells."""
    before, uses, arrivals, waits = [], [], {}, []               # before[e]: events directly before e

    def event(*after):
        before.append([a for a in after if a is not None])
        return len(before) - 1

    for r, steps in enumerate(roles):
        here = pipe = None                                       # the role's latest event, its asynchronous work's latest end
        for step in steps:
            here = event(here)
            if step[0] == "wait":
                waits.append((here, step[1:3]))
            elif step[0] == "drain":
                before[here] += [] if pipe is None else [pipe]
            elif step[0] == "arrive":
                arrivals.setdefault(step[1:3], []).append(here)
            elif step[0] in ("read", "write"):
                uses.append((here, here, r, step[0] == "write", step[1], step))
            else:
                pipe = event(here, pipe)
                if step[0] in ("commit", "load"):
                    arrivals.setdefault(step[-2:], []).append(pipe)
                cells = {"mma": lambda: [(c, False) for c in step[1]] + [(c, True) for c in step[2]], "load": lambda: [(step[1], True)],
                         "store": lambda: [(step[1], False)], "commit": lambda: []}[step[0]]()
                uses += [(here, pipe, r if step[0] == "mma" else None, write, cell, step) for cell, write in cells]
    for e, (barrier, phase) in waits:
        before[e] += [a for p in range(phase + 1) for a in arrivals.get((barrier, p), [])]
    past, todo = {}, list(range(len(before)))                    # events that every event comes after, as bits
    while todo:
        e = todo.pop()
        if e not in past:
            missing = [a for a in before[e] if a not in past]
            if missing:
                todo += [e] + missing
            else:
                past[e] = 0
                for a in before[e]:
                    past[e] |= past[a] | 1 << a
    for i, (from_a, to_a, role_a, write_a, cell, a) in enumerate(uses):
        for from_b, to_b, role_b, write_b, cell_b, b in uses[:i]:
            if cell == cell_b and (write_a or write_b) and not (role_a == role_b is not None):
                if not (past[from_a] >> to_b & 1 or past[from_b] >> to_a & 1):
                    return cell, b, a
    return None


def _query_unit_stage(tiles, slices, chunks, groups, threads, units, shared):
    """The query stage with its memory: `tiles` key tiles, `slices` of the hidden width (none: a one-layer map), `chunks` of features; units, groups
    and threads as in `_query_stage`.  `shared`: d = 128, one set of score columns in the key loop, and in a tail of several products group 1's over
    both P's."""
    n_s, n_p, n_pf, rows = tiles + slices + chunks, tiles + chunks, tiles + (1 if slices else chunks), range(threads)
    own = not shared or slices > 0 or chunks > 1
    # ring items of a unit in the order they are loaded
    order = ([("k", 0)] if tiles else []) + [x for j in range(tiles - 1) for x in (("k", j + 1), ("v", j))]
    if slices:
        order += [("w1", 0)] + [("v", tiles - 1)] * (tiles > 0) + [("w1", j) for j in range(1, slices)]
        order += [("w2", c, j) for c in range(chunks) for j in range(slices)] + [("s", c) for c in range(chunks)]
    else:
        order += [("w", 0)] * (chunks > 0) + [("v", tiles - 1)] * (tiles > 0)
        order += [x for c in range(1, chunks) for x in (("w", c), ("s", c - 1))] + [("s", chunks - 1)] * (chunks > 0)
    compute, score, accum, load = [[[] for _ in rows] for _ in range(2)], [], [], []
    counts = {"%s%d" % (x, s): 1 for x in ("kfull", "vfull", "empty") for s in range(3)}
    counts["pl"] = 1
    items = _ring(["v" if item[0] in ("v", "s") else "k" for item in order] * units)
    for g in range(2):
        counts.update({"%s%d" % (x, g): 1 for x in ("s", "pf", "o", "qf")})
        counts.update({"sf%d" % g: threads, "p%d" % g: threads, "q%d" % g: threads, "h%d" % g: threads * max(slices, 1)})
    for u in range(units):
        ng = groups if u + 1 == units else 2

        def at(item):
            return u * len(order) + order.index(item)

        def ring(item):
            return "ring%d" % (at(item) % 3)

        def full(g, item):
            return [("wait",) + items[at(item)][1:]] if g == 0 else []

        def release(g, item):
            return [("commit", "empty%d" % (at(item) % 3), at(item) // 3)] if g == ng - 1 else []

        def wait(b, g, phase):
            return [("wait", "%s%d" % (b, g), phase)] if phase >= 0 else []

        def all_rows(cell, g):
            return [(cell, g, t) for t in rows]

        def columns(g, i):                                       # where product i of the unit lands
            if not shared:
                return all_rows("scores", g)
            return all_rows("scores", 0) if i < tiles or g == 0 or not own else all_rows("P", 0) + all_rows("P", 1)

        def s_free(g, i):
            ph = u * n_s + i
            if not shared or (own and (i > tiles or tiles == 0)):
                return wait("sf", g, ph - 1)
            if g == 1:
                return wait("sf", 0, ph) if i < tiles or not own else [("wait", "pl", u)]
            return (wait("sf", 0, ph - 1) if i == 0 and own else []) + wait("sf", 1 if ng == 2 or i == 0 else 0, ph - 1)

        for g in range(ng):
            for t in rows:
                c, ps, pp, ppf = compute[g][t], u * n_s, u * n_p, u * n_pf

                def landed(i):
                    return wait("s", g, ps + i)

                def read(i):
                    return [("read", x) for x in columns(g, i) if x[2] == t] + [("arrive", "sf%d" % g, ps + i)]

                for j in range(tiles):
                    c += landed(j) + read(j) + wait("pf", g, ppf + j - 1)
                    c += [("write", ("O", g, t))] * (j > 0) + [("write", ("P", g, t)), ("arrive", "p%d" % g, pp + j)]
                for j in range(slices):
                    c += landed(tiles + j) + ([("drain",)] if j == 0 else [])
                    c += [("write", ("tile" if j == 0 else "Q", g, t))] + read(tiles + j) + [("arrive", "h%d" % g, u)]
                for ch in range(0 if slices else chunks):
                    c += landed(tiles + ch) + [("drain",)] + (wait("pf", g, ppf + tiles + ch - 1) if ch else []) + [("write", ("tile", g, t))]
                    c += read(tiles + ch) + (wait("pf", g, ppf + tiles - 1) if ch == 0 else []) + [("arrive", "p%d" % g, pp + tiles + ch)]
                if slices:
                    c += wait("pf", g, ppf + tiles - 1) + landed(tiles + slices) + read(tiles + slices)
                    c += (landed(n_s - 1) if chunks == 2 else []) + [("write", ("tile", g, t)), ("arrive", "p%d" % g, pp + tiles)]
                if slices and chunks == 2:
                    c += read(n_s - 1) + [("write", ("Q", g, t))] + wait("pf", g, ppf + tiles) + [("arrive", "p%d" % g, pp + tiles + 1)]
                c += wait("o", g, u) + ([("drain",)] if chunks == 0 else []) + [("read", ("O", g, t)), ("write", ("tile", g, t)), ("store", ("tile", g, t))]
        for i in range(n_s):
            for g in range(ng):
                ph, ch = u * n_s + i, i - tiles - slices
                if ch < 0 or not slices:
                    item = ("k", i) if i < tiles else ("w1" if slices else "w", i - tiles)
                    parts = [(item, all_rows("Q", g))]
                    score += full(g, item) if 0 < i < tiles else []
                else:
                    parts = [(("w2", ch, j), all_rows("Q" if j else "tile", g)) for j in range(slices)]
                score += s_free(g, i) + (wait("h", g, u) if slices and ch == 0 else [])
                score += (full(g, parts[0][0]) if i == 0 and tiles else []) + (wait("q", g, u) if i == 0 else [])
                for n, (item, a) in enumerate(parts):
                    score += (full(g, item) if i >= tiles else []) + [("mma", a + [ring(item)], columns(g, i))]
                    if n + 1 == len(parts):
                        score.append(("commit", "s%d" % g, ph))
                        last_of_q = i == n_s - 1 if not slices else chunks == 1 and (i == tiles if slices == 1 else ch == 0)
                        score += [("commit", "qf%d" % g, u)] * last_of_q
                    score += release(g, item)
        for i in range(n_p):
            item, ch = (("v", i), -1) if i < tiles else (("s", i - tiles), i - tiles)
            for g in range(ng):
                in_q = slices > 0 and ch == 1
                a = all_rows("P" if ch < 0 else ("Q" if in_q else "tile"), g)
                accum += full(g, item) + wait("p", g, u * n_p + i) + [("mma", a + [ring(item)], all_rows("O", g))]
                accum += [("commit", "pf%d" % g, u * n_pf + i)] * (not in_q) + [("commit", "o%d" % g, u)] * (i + 1 == n_p)
                accum += [("commit", "qf%d" % g, u)] * in_q
                accum += [("commit", "pl", u)] * (shared and own and chunks > 0 and g == 1 and i + 1 == tiles)
                accum += release(g, item)
        for n, item in enumerate(order):
            if n == (tiles > 0):
                for g in range(ng):                              # (the copy arrives for all rows at once)
                    load += wait("qf", g, u - 1) + [("load", ("Q", g, t), "q%d" % g, u) for t in rows]
            gi = at(item)
            load += wait("empty", gi % 3, gi // 3 - 1) + [("load", ring(item)) + items[gi][1:]]
    return [c for g in range(2) for c in compute[g] if c] + [score, accum, load], counts


def _query_unit_fault(*shape, without=None):
    roles, counts = _query_unit_stage(*shape)
    if without is not None:
        roles = [[s for s in steps if s != without] for steps in roles]
    return _stuck_state(_without_memory(roles), counts) or _race(roles)


# no tail; one layer of F = 128, 256, 384; slices of the hidden width, chunks of features: 128 / 128, 256 / 128, 128 / 256, 256 / 256 at d = 128; 64 / 64 at d = 64
@pytest.mark.parametrize("slices,chunks,shared", [(0, 0, True), (0, 1, True), (0, 2, True), (0, 3, True), (0, 0, False), (0, 1, False), (0, 2, False), (1, 1, True),
                                                  (2, 1, True), (1, 2, True), (2, 2, True), (1, 1, False)])
@pytest.mark.parametrize("tiles,groups,threads,units", [(0, 1, 2, 1), (1, 1, 2, 1), (2, 1, 2, 1), (0, 2, 1, 2), (1, 2, 1, 2), (5, 2, 1, 1), (1, 1, 1, 2),
                                                        (2, 1, 1, 3)])
def test_query_stage_with_its_memory(tiles, slices, chunks, groups, threads, units, shared):
    """Nobody waits for good, no wait passes early, no arrival counts for another phase, and nothing is written while it is in use, in any order."""
    if tiles or (chunks and (slices or not shared)):         # (without a key loop and with one layer it is the kernel with columns for each group)
        assert _query_unit_fault(tiles, slices, chunks, groups, threads, units, shared) is None


@pytest.mark.parametrize("tiles,chunks,units", [(5, 0, 1), (6, 1, 1), (4, 3, 1), (4, 1, 2)])
@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("shared", [False, True])
def test_query_stage_with_the_ring_round_more_than_once(tiles, chunks, units, groups, shared):
    assert _stuck_state(*_query_stage(tiles, chunks, groups, shared, 1, True, units, chunks > 1)) is None


@pytest.mark.parametrize("shape,without", [
    ((1, 2, 2, 1, 2, 1, True), ("wait", "pf0", 1)),          # the second chunk's features handed over, the first one's product not looked at
    ((1, 1, 1, 2, 1, 1, True), ("wait", "pl", 0)),           # group 1's hidden slice over P's that are still being read
    ((2, 0, 2, 2, 1, 1, True), ("wait", "pl", 0)),           # group 1's features over P's that are still being read
    ((1, 0, 0, 1, 1, 2, True), ("drain",)),                  # output rows over those that are still being copied out
    ((1, 1, 1, 1, 1, 2, True), ("drain",)),                  # hidden activations over output rows that are still being copied out
    ((2, 1, 1, 2, 1, 1, True), ("wait", "sf0", 1)),          # group 1's scores over those that group 0 is reading
])
def test_the_model_with_memory_finds_what_it_is_there_for(shape, without):
    assert _query_unit_fault(*shape, without=without) is not None


def test_one_barrier_for_both_users_of_the_ring_would_not_do(monkeypatch):
    """Each warp would look at some of its phases only: with copies that land in any order its wait passes early."""
    both = _ring
    monkeypatch.setitem(globals(), "_ring", lambda kinds: both(["k"] * len(kinds)))
    assert _stuck_state(*_query_stage(4, 0, 2, True, 1, True)) is not None
    assert _query_unit_fault(1, 2, 2, 2, 1, 1, True) is not None
