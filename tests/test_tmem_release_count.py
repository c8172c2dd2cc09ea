"""A CPU model of how the units of the tensor-memory RowSel kernel
(rowsel_tmem.cu) count a ring entry as read: several CTAs copy the entry's
k-chunks, unit by unit, into a few shared-memory slots each; copies land in any
order; of a CTA's two converter sets one takes the even and one the odd
k-chunks of its running sequence (so a unit of an odd number of k-chunks swaps
their parts), each in order. The producer tags a k-chunk with what its set adds
to the entry's count: nothing before the set's last k-chunk of the unit, there
the number of the set's k-chunks. The entry may be overwritten once its count
reaches units x k-chunks. Adding the whole unit's k-chunks at its last one is
the rule that released entries early."""

import random

import pytest


def adds(kc, kch):
    return kc // 2 + 1 if kc + 2 >= kch else 0


def counts(kch, units, slots, ctas, by_set, seed):
    """The entry's count at each step with whether every copy of it had landed."""
    rng = random.Random(seed)
    work = [[] for _ in range(ctas)]
    for u in range(units):
        work[u % ctas] += [(u, kc) for kc in range(kch)]
    issued, landed, seen = [0] * ctas, [set() for _ in range(ctas)], [set() for _ in range(ctas)]
    count, out = 0, []
    while True:
        acts = []
        for i in range(ctas):
            if issued[i] < len(work[i]) and (issued[i] < slots or issued[i] - slots in seen[i]):
                acts.append(("issue", i, 0))
            acts += [("land", i, c) for c in range(issued[i]) if c not in landed[i]]
            for cs in (0, 1):
                nxt = next((c for c in range(cs, len(work[i]), 2) if c not in seen[i]), None)
                if nxt is not None and nxt in landed[i]:
                    acts.append(("convert", i, nxt))
        if not acts:
            return count, out
        act, i, c = rng.choice(acts)
        if act == "issue":
            issued[i] += 1
        elif act == "land":
            landed[i].add(c)
        else:
            seen[i].add(c)
            kc = work[i][c][1]
            n = adds(kc, kch) if by_set else (kch if kc == kch - 1 else 0)
            count += n
            if n:
                out.append((count, all(len(landed[k]) == len(work[k]) for k in range(ctas))))


CASES = [(1, 3, 4, 2), (2, 2, 4, 1), (3, 4, 4, 2), (5, 3, 4, 3), (8, 2, 4, 2), (16, 2, 4, 1), (17, 2, 6, 2)]


@pytest.mark.parametrize("kch", list(range(1, 40)))
def test_a_units_counts_add_up(kch):
    assert sum(adds(kc, kch) for kc in range(kch)) == kch
    assert sum(adds(kc, kch) > 0 for kc in range(kch)) == min(kch, 2)


@pytest.mark.parametrize("kch,units,slots,ctas", CASES)
def test_the_count_is_reached_when_every_copy_has_landed(kch, units, slots, ctas):
    for s in range(200):
        total, out = counts(kch, units, slots, ctas, True, s)
        assert total == units * kch   # nothing is lost: the entry is released
        assert all(landed for n, landed in out if n == units * kch)


def test_counting_a_unit_at_its_last_chunk_can_release_early():
    assert any(not landed for s in range(300) for n, landed in counts(16, 1, 4, 1, False, s)[1] if n == 16)
