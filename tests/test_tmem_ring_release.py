"""A CPU model of how a unit of the tensor-memory RowSel kernel (rowsel_tmem.cu)
releases its ring entry: its k-chunks are copied from the ring in order into a
few shared-memory slots, the copies land in any order, and the two converter
sets (even and odd k-chunks) see only their own landings. The entry may be
overwritten once its release count is reached, so no copy may still be reading
it then. Counting every landed k-chunk keeps that; counting the unit once, at
its last k-chunk, does not."""

import random

import pytest


def release_is_safe(kch, slots, per_chunk, seed):
    rng = random.Random(seed)
    issued, landed, seen = 0, set(), set()   # copies issued, landed, converted
    count = 0
    while True:
        acts = []
        if issued < kch and (issued < slots or issued - slots in seen):
            acts.append(("issue", issued))
        acts += [("land", c) for c in range(issued) if c not in landed]
        for cs in (0, 1):                    # a set takes its k-chunks in order
            nxt = next((c for c in range(cs, kch, 2) if c not in seen), None)
            if nxt is not None and nxt in landed:
                acts.append(("convert", nxt))
        act, c = rng.choice(acts)
        if act == "issue":
            issued += 1
        elif act == "land":
            landed.add(c)
        else:
            seen.add(c)
            count += 1 if per_chunk or c == kch - 1 else 0
            if count == (kch if per_chunk else 1):
                return len(landed) == kch


@pytest.mark.parametrize("kch,slots", [(1, 4), (2, 4), (5, 4), (16, 4), (16, 6)])
def test_every_chunk_counted_releases_after_the_last_read(kch, slots):
    assert all(release_is_safe(kch, slots, True, s) for s in range(300))


def test_one_count_at_the_last_chunk_can_release_early():
    assert not all(release_is_safe(16, 4, False, s) for s in range(300))
