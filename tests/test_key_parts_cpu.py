"""How the key tiles of a last round of units are dealt out to the CTAs (the arithmetic of the query stage's q_parts, written down once more): every tile of
every unit once, at most two parts to a CTA, the one that it leaves to another first and only one such, and whoever finishes a unit finds what the CTAs
right before it have left of it, each for one reader."""
import random

import pytest


def _parts(cta, left, nkv, share):
    """(unit, first key tile, end, whether it is left, CTAs to add up) of a CTA, in its order."""
    r0, r1 = cta * share, min(left * nkv, (cta + 1) * share)
    if r0 >= r1:
        return []
    unit = r0 // nkv
    k0, over = r0 - unit * nkv, r1 - (unit + 1) * nkv

    def part(u, a, b):
        return u, a, b, b < nkv, 0 if b < nkv or a == 0 else cta - u * nkv // share

    return ([part(unit + 1, 0, over)] if over > 0 else []) + [part(unit, k0, nkv if over > 0 else r1 - unit * nkv)]


@pytest.mark.parametrize("sms", [148, 132, 20, 7])
def test_every_key_tile_once_and_every_part_read_once(sms):
    rng = random.Random(sms)
    for _ in range(400):
        left, nkv = rng.randint(1, sms - 1), rng.randint(2, 300)
        share = max(2, -(-left * nkv // sms))
        if share >= nkv:
            continue
        dealt = [_parts(c, left, nkv, share) for c in range(sms)]
        assert all(bool(ps) == (c < -(-left * nkv // share)) for c, ps in enumerate(dealt))
        owner, leaves, read = {}, {}, set()
        for c, ps in enumerate(dealt):
            assert len(ps) <= 2 and [p[3] for p in ps] in ([], [True], [False], [True, False])
            for unit, a, b, left_over, _ in ps:
                assert 0 <= unit < left and 0 <= a < b <= nkv
                for k in range(a, b):
                    assert (unit, k) not in owner
                    owner[unit, k] = c
                if left_over:
                    leaves[c] = unit
        assert len(owner) == left * nkv
        for c, ps in enumerate(dealt):
            for unit, a, b, left_over, merges in ps:
                if not left_over:
                    before = set(range(c - merges, c))
                    assert {owner[unit, k] for k in range(a)} == before and all(leaves[x] == unit for x in before) and not before & read
                    read |= before
        assert read == set(leaves)
