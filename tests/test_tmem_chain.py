"""A CPU model of the chain ciphertexts -> ring -> shared-memory slots -> tensor
memory -> MMAs of the tensor-memory RowSel kernel (rowsel_tmem.cu) with the
release rules it runs, under random interleavings; single-CTA and SM-pair forms.

  - an ingest group claims tasks (entry, k-chunk) in order and writes ring entry
    E % R once the count of entry E - R has reached units x k-chunks, and at most
    `la` entries ahead of the units claimed;
  - a producer claims units in order and, once its entry is ready, copies its
    k-chunks one by one into ring slot i % RS (after rempty) and the database's
    part into B stage i % NS (after empty). Copies land in any order and read
    their source when they land;
  - converter set c takes k-chunks i = c, c + 2, ...: waits rfull, reads the
    words, adds to the entry's count what the producer tagged (at the set's last
    k-chunk of the unit its number of k-chunks there, else nothing), waits aempty
    and full, stores to the A buffer, and only then hands back the ring slot
    (rempty) and signals the buffer (afull);
  - the MMA warp issues k-chunks in order; they run later, in order, and their
    commits arrive on empty and aempty (of both CTAs in the pair); accumulators
    are double buffered and drained by the epilogue.
Checked: no deadlock; no copy reads another entry's data; every MMA reads its
own k-chunk's words and B part."""

import random

import pytest

from tests.test_tmem_protocol import Bar, _kernel_cfg


class Cta:
    def __init__(self, ns, rs, nbuf, afull):
        self.full, self.empty = [Bar(1) for _ in range(ns)], [Bar(1) for _ in range(ns)]
        self.rfull, self.rempty = [Bar(1) for _ in range(rs)], [Bar(2) for _ in range(rs)]
        self.afull, self.aempty = [Bar(afull) for _ in range(nbuf)], [Bar(1) for _ in range(nbuf)]
        self.slot, self.slot_tag = [None] * rs, [None] * rs
        self.stage, self.stage_tag = [None] * ns, [None] * ns
        self.abuf = {}


def run(pair, ns, rs, kpb, entries, upe, kch, R, la, clusters, seed, bug=None, land=0.25):
    rng = random.Random(seed)
    nbuf, C = 4 // kpb, 2 if pair else 1
    n_units = entries // C * upe
    ring, ready, count = [[None] * kch for _ in range(R)], [0] * entries, [0] * entries
    ctr = {"unit": 0, "task": 0}
    copies, done = [], []

    def wait(bar, parity):
        while not bar.done(parity):
            yield

    def ingest():
        while ctr["task"] < entries * kch:
            E, kc = divmod(ctr["task"], kch)
            ctr["task"] += 1
            yield
            while (E >= la and ctr["unit"] < (E - la) // C * upe) or (E >= R and count[E - R] < upe * kch):
                yield
            assert not any(c[2] == ("ring", E - R, kc) for c in copies), "a copy in flight is overwritten"
            ring[E % R][kc] = E
            ready[E] += 1
            yield

    def producer(cl, r):
        me, i, n = cl["ctas"][r], 0, 0
        while True:
            if r == 0:
                cl["units"].append(ctr["unit"] if ctr["unit"] < n_units else None)
                ctr["unit"] += 1
            while len(cl["units"]) <= n:
                yield
            u = cl["units"][n]
            n += 1
            for kc in range(kch) if u is not None else range(2):
                sl, st = i % rs, i % ns
                if u is None:
                    yield from wait(me.empty[st], (i // ns) & 1 ^ 1)
                    me.stage_tag[st] = None
                    yield from wait(me.rempty[sl], (i // rs) & 1 ^ 1)
                    me.slot_tag[sl] = None
                    me.rfull[sl].arrive()
                    i += 1
                    continue
                E = u // upe * C + r
                while ready[E] < kch:
                    yield
                yield from wait(me.rempty[sl], (i // rs) & 1 ^ 1)
                n_set = kc // 2 + 1 if kc + 2 >= kch else 0
                if bug == "count_unit_at_last":
                    n_set = kch if kc == kch - 1 else 0
                me.slot_tag[sl] = (u, kc, E, n_set)
                me.rfull[sl].arrive(tx=1)
                copies.append((me, sl, ("ring", E, kc), (u, kc)))
                yield from wait(me.empty[st], (i // ns) & 1 ^ 1)
                me.stage_tag[st] = (u, kc)
                me.full[st].arrive(tx=1)
                copies.append((me, st, ("b",), (u, kc)))
                i += 1
                yield
            if u is None:
                return

    def converter(cl, r, cs):
        me, i = cl["ctas"][r], cs
        while True:
            sl, st, bi = i % rs, i % ns, i // kpb
            ab, aph = bi % nbuf, (bi // nbuf) & 1
            yield from wait(me.rfull[sl], (i // rs) & 1)
            tag = me.slot_tag[sl]
            if tag is None:
                yield from wait(me.aempty[ab], aph ^ 1)
                cl["ctas"][0].afull[ab].arrive()
                return
            count[tag[2]] += tag[3]
            if bug == "slot_before_store":
                me.rempty[sl].arrive(2)
            yield
            yield from wait(me.aempty[ab], aph ^ 1)
            yield from wait(me.full[st], (i // ns) & 1)
            assert me.slot[sl] == tag[:2], "a ring slot was refilled before its words were used"
            me.abuf[ab, i % kpb] = tag[:2]
            yield
            if bug != "slot_before_store":
                me.rempty[sl].arrive(2)
            cl["ctas"][0].afull[ab].arrive()
            i += 2

    def mma(cl):
        me, i = cl["ctas"][0], 0
        while True:
            if i % kpb == 0:
                yield from wait(me.afull[i // kpb % nbuf], (i // kpb // nbuf) & 1)
            tag = me.stage_tag[i % ns]
            if tag is None:
                return
            while cl["acc"] == 2:            # both accumulators full or in use
                yield
            cl["acc"] += 1
            for kc in range(kch):
                if kc and i % kpb == 0:
                    yield from wait(me.afull[i // kpb % nbuf], (i // kpb // nbuf) & 1)
                cl["engine"].append((i, (tag[0], kc), kc == kch - 1))
                i += 1
                yield

    def engine_step(cl):
        i, want, last = cl["engine"].pop(0)
        ab, part = i // kpb % nbuf, i % kpb
        for c in cl["ctas"]:
            assert c.stage[i % ns] == want and c.abuf[ab, part] == want, "an MMA read another k-chunk's operands"
            c.empty[i % ns].arrive()
            if part == kpb - 1:
                c.aempty[ab].arrive()
        if last:
            done.append(want[0])
            cl["drain"] += 1

    cls = [{"ctas": [Cta(ns, rs, nbuf, kpb * (C if r == 0 else 1)) for r in range(C)], "units": [], "engine": [],
            "acc": 0, "drain": 0} for _ in range(clusters)]
    actors = []
    for cl in cls:
        actors.append(mma(cl))
        for r in range(C):
            actors += [producer(cl, r), converter(cl, r, 0), converter(cl, r, 1), ingest()]
    idle = 0
    while actors or copies or any(cl["engine"] for cl in cls):
        k = rng.random()
        busy = [cl for cl in cls if cl["engine"]]
        draining = [cl for cl in cls if cl["drain"]]
        if copies and k < land:
            me, at, src, tag = copies.pop(rng.randrange(len(copies)))
            if src[0] == "ring":
                assert ring[src[1] % R][src[2]] == src[1], "a copy read another entry's data"
                me.slot[at] = tag
                me.rfull[at].complete_tx(1)
            else:
                me.stage[at] = tag
                me.full[at].complete_tx(1)
            idle = 0
        elif busy and k < 0.4:
            engine_step(rng.choice(busy))
            idle = 0
        elif draining and k < 0.5:
            cl = rng.choice(draining)
            cl["drain"] -= 1
            cl["acc"] -= 1
            idle = 0
        elif actors:
            a = rng.choice(actors)
            before = (ctr["unit"], ctr["task"], sum(ready), sum(count), len(copies), sum(len(c["engine"]) for c in cls))
            try:
                next(a)
            except StopIteration:
                actors.remove(a)
                idle = 0
                continue
            after = (ctr["unit"], ctr["task"], sum(ready), sum(count), len(copies), sum(len(c["engine"]) for c in cls))
            idle = 0 if before != after or copies or busy or draining else idle + 1
            assert idle < 400 * len(actors), "deadlock"
    assert sorted(done) == list(range(n_units)), "a unit was lost or run twice"


SHAPES = [  # entries, units per entry, k-chunks, ring entries, lookahead, clusters
    (4, 2, 1, 2, 2, 1),
    (6, 2, 3, 2, 2, 2),      # the smallest ring
    (6, 1, 8, 4, 2, 3),
    (4, 4, 5, 2, 2, 2),
]


@pytest.mark.parametrize("pair", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_the_shipped_rules_progress_and_read_their_own_data(pair, shape):
    ns, rs, kpb = _kernel_cfg()[pair]
    for seed in range(25):
        run(pair, ns, rs, kpb, *shape, seed)


@pytest.mark.parametrize("bug,text,shape,land", [
    ("count_unit_at_last", "copy", (8, 1, 2, 2, 4, 2), 0.04),       # slow copies
    ("slot_before_store", "refilled", (8, 1, 12, 4, 4, 1), 0.5),    # fast ones
])
def test_the_unsafe_rules_are_caught(bug, text, shape, land):
    ns, rs, kpb = _kernel_cfg()[False]
    caught = 0
    for seed in range(120):
        try:
            run(False, ns, rs, kpb, *shape, seed, bug, land)
        except AssertionError as e:
            assert text in str(e), e
            caught += 1
    assert caught
