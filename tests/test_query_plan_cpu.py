"""The query stage's plan as it is compiled: every tile of every unit once, each part for one reader, ring items and phases that go on where the CTA's units
before have ended, and key loops in parts only where they were measured to be no slower."""
import random

import pytest

from _query_plan import deal, plan


@pytest.mark.parametrize("sms", [148, 132, 20, 7])
@pytest.mark.parametrize("lin,fc,slices", [(0, 1, 0), (1, 1, 0), (1, 3, 0), (1, 1, 1), (1, 2, 2)])
def test_every_key_tile_once_every_part_read_once_and_phases_that_go_on(sms, lin, fc, slices):
    rng = random.Random(sms)
    # a whole unit's ring items, score-column products, hand-overs of P, products that have read one
    whole = (lambda k: (2 * k + (slices + fc * slices + fc if slices else 2 * fc), k + slices + fc, k + fc, k + (1 if slices else fc))) if lin else (lambda k: (2 * k, k, k, k))
    for _ in range(120):
        left, nkv, rounds = rng.randint(1, sms - 1), rng.randint(2, 300), rng.choice([0, 0, 1, 5])
        share = max(2, -(-left * nkv // sms))
        if share >= nkv:
            continue
        ctas = sms if rounds else -(-left * nkv // share)
        dealt = [deal(rounds * ctas + left, rounds, share, nkv, lin, fc, slices, ctas, c) for c in range(ctas)]
        owner, leaves, read = {}, {}, set()
        for c, parts in enumerate(dealt):
            assert bool(parts) == (c < -(-left * nkv // share))
            assert len(parts) <= 2 and [p[3] for p in parts] in ([], [1], [0], [1, 0])
            at = tuple(rounds * x for x in whole(nkv))
            for unit, k0, k1, left_over, _, *before in parts:
                assert 0 <= unit < left and 0 <= k0 < k1 <= nkv and left_over == (k1 < nkv)
                assert tuple(before) == at + (rounds,)
                at = tuple(a + x * (k1 - k0) for a, x in zip(at, (2, 1, 1, 1)))     # of a part that is left: its key tiles, no tail
                for k in range(k0, k1):
                    assert (unit, k) not in owner
                    owner[unit, k] = c
                if left_over:
                    leaves[c] = unit
        assert len(owner) == left * nkv
        for c, parts in enumerate(dealt):
            for unit, k0, k1, left_over, merges, *_ in parts:
                if not left_over:
                    before = set(range(c - merges, c))
                    assert {owner[unit, k] for k in range(k0)} == before and all(leaves[x] == unit for x in before) and not before & read
                    read |= before
        assert read == set(leaves)


# (heads, N, one softmax token in, d, F, hidden, biases): whole calls in parts against whole units, on 148 SMs (us)
SLOWER_IN_PARTS = [(1, 6803, 2, 128, 128, 0, False),         # 52.0 for 49.3
                   (7, 8689, 3, 128, 128, 0, False),         # 117.5 for 112.4
                   (10, 6079, 2, 128, 128, 0, False),        # 122.2 for 118.5
                   (8, 11813, 4, 128, 128, 0, False),        # 169.2 for 166.7
                   (7, 8319, 3, 128, 128, 0, True),          # 122.3 for 114.9
                   (12, 9837, 2, 128, 128, 0, True),         # 308.1 for 302.8
                   (5, 11654, 4, 128, 256, 0, False),        # 122.0 for 120.5
                   (5, 11890, 4, 128, 128, 128, False)]      # 136.0 for 133.3
FASTER_IN_PARTS = [(1, 8000, 1, 64, 64, 0, False), (5, 9467, 1, 64, 64, 0, False), (8, 7121, 2, 64, 64, 64, False), (2, 10000, 1, 128, 128, 0, False),
                   (5, 9072, 2, 128, 128, 0, False), (3, 7069, 2, 128, 128, 0, False), (2, 10726, 2, 128, 128, 0, True), (3, 6772, 2, 128, 256, 0, False),
                   (5, 11324, 2, 128, 128, 128, False)]


@pytest.mark.parametrize("layer", SLOWER_IN_PARTS)
def test_units_stay_whole_where_parts_are_slower(layer):
    H, N, rate, d, F, hidden, biases = layer
    assert not plan(N, H, rate, d, F, hidden, biases)["parts"]


@pytest.mark.parametrize("layer", FASTER_IN_PARTS)
def test_key_loops_go_in_parts_where_that_is_faster(layer):
    H, N, rate, d, F, hidden, biases = layer
    assert plan(N, H, rate, d, F, hidden, biases)["parts"]
