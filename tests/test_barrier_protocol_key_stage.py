"""The barrier protocols of the key stage, of the first layer of the keys in runs of tiles, and of the query stage's units whose key loops are in parts, walked
through in every order and looked through for races by the model in test_barrier_protocol.py."""
import pytest

from test_barrier_protocol import _race, _stuck_state, _without_memory


def _fault(roles, counts, without=None):
    """`without`: (role, step) pairs to leave out."""
    if without is not None:
        roles = [[s for s in steps if not without(r, s)] for r, steps in enumerate(roles)]
    return _stuck_state(_without_memory(roles), counts) or _race(roles)


class _Phases:
    """Phases in order: the n-th arrival's phase of a barrier that `per` arrivals complete."""

    def __init__(self):
        self.n = {}

    def next(self, b, per=1):
        self.n[b] = self.n.get(b, 0) + 1
        return (self.n[b] - 1) // per


# ---------------------------------------------------------------- key stage
def _key_stage(tiles, x_items, slots, gathers, threads=2):
    """kpass_kernel: `x_items` ring items a tile feed the features (K, or the hidden slices of two layers), one is V; two issuing warps, `threads` stand for the
    feature warps, one for the gather warps."""
    two, items = x_items > 1, []
    ph = _Phases()
    for t in range(tiles):
        for i in range(x_items + 1):
            slot = (t * (x_items + 1) + i) % slots
            name = "%s%d" % ("v" if i == x_items else "x", slot)
            items.append((slot, name, ph.next(name)))
    features, gather, load, phi, acc = [[] for _ in range(threads)], [], [], [], []
    counts = {"w": 1, "done": 1, "ring_idle": threads + (1 if gathers else 0)}
    for s in range(slots):
        counts.update({"x%d" % s: 1, "v%d" % s: 1, "e%d" % s: 2 if gathers else 1})
    for b in range(2):
        counts.update({"d1%d" % b: 1, "pk%d" % b: threads, "sd%d" % b: 1})

    def use(t, i):
        return items[t * (x_items + 1) + i]

    load.append(("load", "W", "w", 0))
    for n, (slot, name, phase) in enumerate(items):
        if n == x_items + 1:
            load.append(("wait", "x0", 0))                    # the first tile has the memory system to itself
        load += [("wait", "e%d" % slot, n // slots - 1)] * (n >= slots) + [("load", ("ring", slot), name, phase)]
    phi.append(("wait", "w", 0))
    for t in range(tiles):
        b = t & 1
        phi += [("wait", "pk%d" % b, (t - 2) >> 1)] * (t >= 2)
        for i in range(x_items):
            slot, name, phase = use(t, i)
            phi += [("wait", name, phase), ("mma", ["W", ("ring", slot)], [("D1", b, th) for th in range(threads)]), ("commit", "e%d" % slot, (t * (x_items + 1) + i) // slots)]
            phi += [("commit", "d1%d" % b, t >> 1)] * (i + 1 == x_items)
        slot, name, phase = use(t, x_items)
        acc += [("wait", name, phase), ("wait", "pk%d" % b, t >> 1), ("mma", [("P", b, th) for th in range(threads)] + [("ring", slot)], ["S"]),
                ("commit", "e%d" % slot, (t * (x_items + 1) + x_items) // slots), ("commit", "sd%d" % b, t >> 1)] + [("commit", "done", 0)] * (t + 1 == tiles)
        for th in range(threads):
            features[th] += [("wait", "d1%d" % b, t >> 1), ("read", ("D1", b, th))] + [("wait", "sd%d" % b, (t - 2) >> 1)] * (t >= 2)
            features[th] += [("write", ("P", b, th)), ("arrive", "pk%d" % b, t >> 1)]
        for i in range(x_items + 1):
            slot, name, phase = use(t, i)
            gather += [("wait", name, phase)] + [("arrive", "e%d" % slot, (t * (x_items + 1) + i) // slots)] * (two and i < x_items)
        for i in range(x_items if two else 0, x_items + 1):
            gather.append(("read", ("ring", use(t, i)[0])))
        for i in range(x_items if two else 0, x_items + 1):
            gather.append(("arrive", "e%d" % use(t, i)[0], (t * (x_items + 1) + i) // slots))
    gather.append(("arrive", "ring_idle", 0))
    for th in range(threads):                                 # the partial state goes through the ring
        features[th] += [("wait", "done", 0), ("arrive", "ring_idle", 0), ("wait", "ring_idle", 0), ("read", "S")]
        features[th] += [("write", ("ring", s)) for s in range(slots) if s % threads == th]
    return features + ([gather] if gathers else []) + [load, phi, acc], counts


@pytest.mark.parametrize("tiles,x_items,slots,gathers", [(1, 1, 4, True), (3, 1, 4, True), (4, 1, 3, False), (5, 1, 6, False), (2, 2, 5, True), (3, 2, 5, False), (4, 1, 4, True)])
def test_key_stage(tiles, x_items, slots, gathers):
    assert _fault(*_key_stage(tiles, x_items, slots, gathers, threads=1 if tiles > 3 else 2)) is None


@pytest.mark.parametrize("what", ["sd", "pk", "ring_idle", "e"])
def test_the_key_stage_model_finds_what_it_is_there_for(what):
    """Features over those that a product reads; Phi^T over what is being read; the partial state over rows that are being gathered; a ring slot loaded over what is in use."""
    roles, counts = _key_stage(4, 1, 4, True, threads=1)
    features, gather, load, phi = 0, 1, 2, 3
    role = {"sd": features, "pk": phi, "ring_idle": features, "e": load}[what]
    assert _fault(roles, counts, lambda r, s: r == role and s[0] == "wait" and s[1].startswith(what)) is not None


# ---------------------------------------------------------------- first layer of the keys in runs of tiles
def _run_of_tiles(heads, gathers, threads=2):
    """phi1_run_kernel: the head of each tile of the run; three tiles in the ring, two sets of accumulators of two slices, weights that change with the head."""
    n, roles, load, mma = len(heads), [[] for _ in range(threads)], [], []
    counts = {"wfree": 1, "meet": threads}
    for s in range(3):
        counts.update({"x%d" % s: 1, "xe%d" % s: 1 + (threads if gathers else 0)})
    for j in range(2):
        counts.update({"w%d" % j: 1, "free%d" % j: threads, "done0%d" % j: 1, "done1%d" % j: 1})
    n_w = met = 0
    for i, h in enumerate(heads):
        s, b, first = i % 3, i & 1, i == 0 or heads[i - 1] != h
        last = i + 1 < n and heads[i + 1] != h
        load += [("wait", "xe%d" % s, i // 3 - 1)] * (i >= 3) + [("load", ("ring", s), "x%d" % s, i // 3)]
        if first:
            load += [("wait", "wfree", n_w - 1)] * (i > 0) + [("load", ("W", j), "w%d" % j, n_w) for j in range(2)]
        mma += [("wait", "free%d" % b, (i >> 1) - 1)] * (i >= 2) + [("wait", "x%d" % s, i // 3)]
        for j in range(2):
            mma += [("wait", "w%d" % j, n_w)] * first + [("mma", [("ring", s), ("W", j)], [("A", b, j, th) for th in range(threads)]), ("commit", "done%d%d" % (b, j), i >> 1)]
        mma += [("commit", "xe%d" % s, i // 3)] * (i + 3 < n) + [("commit", "wfree", n_w + first - 1)] * last
        n_w += first
        for th in range(threads):
            c, m = roles[th], met
            if gathers:
                c += [("wait", "x%d" % s, i // 3), ("read", ("ring", s)), ("arrive", "xe%d" % s, i // 3)]
            for j in range(2):
                # thread 0 drains its copies out (the model's: all of them) ahead of the barrier behind which all write
                c += [("wait", "done%d%d" % (b, j), i >> 1)] + [("drain",)] * (th == 0) + [("arrive", "meet", m), ("wait", "meet", m)]
                c += [("read", ("A", b, j, th)), ("write", ("out", j, th))] + [("arrive", "free%d" % b, i >> 1)] * (j == 1)
                c += [("arrive", "meet", m + 1), ("wait", "meet", m + 1)] + [("store", ("out", j, x)) for x in range(threads)] * (th == 0)
                m += 2
        met += 4
    return roles + [load, mma], counts


@pytest.mark.parametrize("heads", [(0,), (0, 0, 0, 0), (0, 1), (0, 0, 1, 1), (0, 1, 2), (0, 0, 0, 0, 1)])
@pytest.mark.parametrize("gathers", [False, True])
def test_first_layer_in_runs_of_tiles(heads, gathers):
    assert _fault(*_run_of_tiles(heads, gathers, threads=1 if len(heads) > 2 else 2)) is None


@pytest.mark.parametrize("what,role", [("free", "mma"), ("xe", "load"), ("wfree", "load"), ("meet", "row"), ("drain", "row")])
def test_the_run_model_finds_what_it_is_there_for(what, role):
    """Products over rows that are being read; a tile of K over one in use; weights over those in use; rows stored before all are written, and written over those being stored."""
    roles, counts = _run_of_tiles((0, 0, 0, 0, 1) if what != "meet" else (0, 0), True, threads=1 if what != "meet" else 2)
    which = {"mma": len(roles) - 1, "load": len(roles) - 2, "row": 0}[role]
    assert _fault(roles, counts, lambda r, s: r == which and (s[0] == "drain" if what == "drain" else s[0] == "wait" and s[1].startswith(what))) is not None


# ---------------------------------------------------------------- units with key loops in parts
def _units_in_parts(units, shared, threads=1):
    """The query stage with a one-layer map over units (key tiles, feature chunks, "whole", "leaves" or "merges"): one that leaves its sum has no tail; one that merges adds to O
    behind its last product.  What comes before a unit is counted on, as the plan's offsets are."""
    wide = max(c for _, c, _ in units) > 1
    own = shared and wide
    compute, score, accum, load = [[[] for _ in range(threads)] for _ in range(2)], [], [], []
    counts = {"pl": 1}
    for g in range(2):
        counts.update({"%s%d" % (x, g): 1 for x in ("s", "pf", "o", "qf")})
        counts.update({"%s%d" % (x, g): threads for x in ("sf", "p", "q")})
    for s in range(3):
        counts.update({"%s%d" % (x, s): 1 for x in ("k", "v", "e")})
    ph, ring, ps, tail = _Phases(), 0, 0, 0

    def rows(cell, g):
        return [(cell, g, t) for t in range(threads)]

    for u, (tiles, chunks, kind) in enumerate(units):
        chunks = 0 if kind == "leaves" else chunks
        n = tiles + chunks
        order = [("k", 0)] + [x for j in range(tiles - 1) for x in (("k", j + 1), ("v", j))] + [("k", tiles)] * (chunks > 0) + [("v", tiles - 1)]
        order += [x for c in range(chunks - 1) for x in (("k", tiles + c + 1), ("v", tiles + c))] + [("v", n - 1)] * (chunks > 0)
        place = {}
        for m, (kind_of, i) in enumerate(order):
            slot = (ring + m) % 3
            name = "%s%d" % (kind_of, slot)
            place[kind_of, i] = (slot, name, ph.next(name), (ring + m) // 3)
            if m == 1:
                for g in range(2):
                    load += [("wait", "qf%d" % g, u - 1)] * (u > 0) + [("load", x, "q%d" % g, u) for x in rows("Q", g)]
            load += [("wait", "e%d" % slot, (ring + m) // 3 - 1)] * (ring + m >= 3) + [("load", ("ring", slot), name, place[kind_of, i][2])]
        ring += len(order)

        def columns(g, i):
            if not shared:
                return rows("scores", g)
            return rows("scores", 0) if i < tiles or g == 0 or not own else rows("P", 0) + rows("P", 1)

        def s_free(g, i):
            p = ps + i
            if not shared or (own and i > tiles):
                return [("wait", "sf%d" % g, p - 1)] * (p > 0)
            if g == 1:
                return [("wait", "sf0", p)] if not own or i < tiles else [("wait", "pl", tail)]
            return [("wait", "sf0", p - 1)] * (own and i == 0 and p > 0) + [("wait", "sf1", p - 1)] * (p > 0)

        for i in range(n):
            slot, name, phase, release = place["k", i]
            for g in range(2):
                score += [("wait", name, phase)] * (g == 0 and 0 < i < tiles) + s_free(g, i) + [("wait", name, phase)] * (g == 0 and (i == 0 or i >= tiles))
                score += [("wait", "q%d" % g, u)] * (i == 0)
                score += [("mma", rows("Q", g) + [("ring", slot)], columns(g, i)), ("commit", "s%d" % g, ps + i)] + [("commit", "qf%d" % g, u)] * (i + 1 == n)
                score += [("commit", "e%d" % slot, release)] * (g == 1)
            slot, name, phase, release = place["v", i]
            for g in range(2):
                accum += [("wait", name, phase)] * (g == 0) + [("wait", "p%d" % g, ps + i), ("mma", rows("P" if i < tiles else "tile", g) + [("ring", slot)], rows("O", g)),
                                                              ("commit", "pf%d" % g, ps + i)]
                accum += [("commit", "o%d" % g, u)] * (i + 1 == n) + [("commit", "pl", tail)] * (own and chunks > 0 and g == 1 and i + 1 == tiles)
                accum += [("commit", "e%d" % slot, release)] * (g == 1)
        for g in range(2):
            for t in range(threads):
                c = compute[g][t]
                for i in range(n):
                    c += [("wait", "s%d" % g, ps + i)]
                    mine = [("read", x) for x in columns(g, i) if x[2] == t]
                    if i < tiles:
                        c += mine + [("arrive", "sf%d" % g, ps + i)] + [("wait", "pf%d" % g, ps + i - 1)] * (ps + i > 0)
                        c += [("write", ("O", g, t))] * (i > 0) + [("write", ("P", g, t)), ("arrive", "p%d" % g, ps + i)]
                        if i + 1 == tiles and kind == "merges":
                            c += [("wait", "pf%d" % g, ps + i), ("write", ("O", g, t))]
                    else:
                        c += [("drain",)] + [("wait", "pf%d" % g, ps + i - 1)] * (i > tiles) + [("write", ("tile", g, t))] + mine + [("arrive", "sf%d" % g, ps + i)]
                        c += [("wait", "pf%d" % g, ps + i - 1)] * (i == tiles) + [("arrive", "p%d" % g, ps + i)]
                c += [("wait", "o%d" % g, u), ("read", ("O", g, t))]
                if kind != "leaves":
                    c += [("drain",)] * (chunks == 0) + [("write", ("tile", g, t)), ("store", ("tile", g, t))]
        ps, tail = ps + n, tail + (chunks > 0)
    return [c for g in range(2) for c in compute[g]] + [score, accum, load], counts


@pytest.mark.parametrize("units", [((2, 1, "leaves"), (1, 1, "merges")), ((1, 2, "leaves"), (2, 2, "merges")), ((1, 1, "whole"), (2, 1, "leaves"), (1, 1, "merges")),
                                   ((1, 2, "whole"), (1, 2, "leaves"), (2, 2, "merges")), ((3, 0, "leaves"), (2, 0, "merges")), ((1, 1, "whole"), (3, 1, "merges"))])
@pytest.mark.parametrize("shared", [False, True])
def test_units_in_parts(units, shared):
    assert _fault(*_units_in_parts(units, shared)) is None


@pytest.mark.parametrize("what", ["merge", "tail"])
def test_the_parts_model_finds_what_it_is_there_for(what):
    """O added to while the last product writes it; group 1's features taken to be behind the tail of a unit that has none."""
    units = ((1, 2, "whole"), (1, 2, "leaves"), (2, 2, "merges"))
    roles, counts = _units_in_parts(units, True)
    if what == "merge":
        at = [i for i, s in enumerate(roles[0]) if s == ("write", ("O", 0, 0))][-1]
        assert roles[0][at - 1][:2] == ("wait", "pf0")
        roles[0] = roles[0][:at - 1] + roles[0][at:]
    else:                                                     # a unit's index in place of the number of tails before it
        roles[2] = [("wait", "pl", 2) if s == ("wait", "pl", 1) else s for s in roles[2]]
    assert _fault(roles, counts) is not None
