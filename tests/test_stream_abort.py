"""A CPU model of how the epilogue warps of the streaming RowSel kernel
(rowsel_stream.cu) leave it after an expired wait, under random interleavings.

Per unit each of the warps waits for the accumulators of the unit's slots in
turn, then all of them meet at a barrier (bar.sync / bar.red: it has no time
limit, and completes only when every warp has arrived), write the unit and meet
again. A wait looks at the accumulator first and at the abort flag after it, so
an accumulator that arrives around an abort is seen by some warps and not by
others. A warp that leaves goes to the CTA's last barrier and waits there for
the others. Agreeing at the first barrier lets every warp leave; leaving before
it (the rule without agreement) can strand the others."""

import random

import pytest

WARPS, SLOTS, UNITS = 8, 8, 3


def all_leave(agree, seed):
    rng = random.Random(seed)
    total = UNITS * SLOTS
    ready, aborted = 0, False             # accumulators that have arrived; the abort flag
    stop = rng.randrange(total + 1)       # none arrives after this many
    state = [["wait", 0, True] for _ in range(WARPS)]   # phase, accumulators taken, ok
    # a poll in progress: the accumulator was looked at and not there, the flag comes next
    looked = [False] * WARPS
    for _ in range(100000):
        acts = [("abort",)] if not aborted else []
        if ready < stop:
            acts.append(("arrive",))
        acts += [("warp", w) for w in range(WARPS) if state[w][0] == "wait"]
        for where in ("meet", "meet2"):
            if all(s[0] == where for s in state):
                acts = [("pass", where)]
        if all(s[0] == "gone" for s in state):
            return True
        if not acts:
            return False                   # no step left: a warp waits for one that has gone
        act = rng.choice(acts)
        if act[0] == "abort":
            aborted = ready >= stop or rng.random() < 0.1
        elif act[0] == "arrive":
            ready += 1
        elif act[0] == "pass":
            ok = all(s[2] for s in state)
            for s in state:
                if act[1] == "meet":
                    s[0] = "meet2" if ok else "gone"
                else:
                    s[0] = "wait" if s[1] < total else "gone"
        else:
            w = act[1]
            s = state[w]
            if looked[w]:
                looked[w] = False
                if aborted:
                    s[2] = False
                    s[0] = "meet" if agree else "gone"
            elif ready > s[1]:
                s[1] += 1
                if s[1] % SLOTS == 0:
                    s[0] = "meet"
            else:
                looked[w] = True
        if not agree and any(s[0] == "gone" for s in state) and any(s[0] in ("meet", "meet2") for s in state):
            return False                   # that barrier can never complete
    return False


def test_warps_that_agree_all_leave():
    assert all(all_leave(True, s) for s in range(400))


def test_leaving_before_the_barrier_strands_the_others():
    assert not all(all_leave(False, s) for s in range(400))
