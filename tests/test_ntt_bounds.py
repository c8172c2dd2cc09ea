"""A CPU model of the tree kernels' transforms as csrc/ntt.cuh runs them: the
compile-time value bounds (forward below 16q, inverse 16/8/4/4/2/2/2/2 within a
round), the buffer layout x + 4 (x >> 9) with 16-byte accesses in the
bit-reversed rounds, the scaling folded into the last inverse level, the digit
fields with their per-prime addends and the two-quotient 64-bit reduction, all
in exact 32-bit arithmetic against the oracle."""

import numpy as np
import pytest

import oracle
import synth
from tests.test_ntt_schedule import M32, brev, csub, middle_levels, set_of, tables

TOP = (1 << 28) - 57   # not a prime: the largest modulus the bounds must hold for


def pad(x):
    return x + 4 * (x >> 9)


def shoup(a, w, q):
    assert 0 <= a <= M32 and 0 <= w < q
    r = (a * w - ((a * ((w << 32) // q)) >> 32) * q) & M32
    assert r < 2 * q
    return r


def fwd_bound(l):
    b = 2
    for _ in range(l):
        b = 10 if b + 2 > 16 else b + 2
    return b


def inv_bound(k, r):
    if r == 0:
        return 2
    bit = 1 << (r - 1)
    return 2 if k & bit else inv_bound(k, r - 1) + inv_bound(k | bit, r - 1)


def fwd_levels(v, R, lvl, tw, q):
    for r in range(R):
        span = 1 << (R - 1 - r)
        assert all(x < fwd_bound(lvl + r) * q for x in v)
        for k in range(1 << R):
            if not k & span:
                t = shoup(v[k + span], tw(r, k), q)
                u = csub(v[k], 8 * q) if fwd_bound(lvl + r) + 2 > 16 else v[k]
                assert u + t <= M32 and u - t + 2 * q >= 0
                v[k], v[k + span] = u + t, u - t + 2 * q


def inv_levels(v, R, tw, q):
    assert all(x < 2 * q for x in v)
    for r in range(R):
        span = 1 << r
        for k in range(1 << R):
            if not k & span:
                x, y = v[k], v[k + span]
                assert x < inv_bound(k, r) * q and y < inv_bound(k + span, r) * q and x + y <= M32
                off = inv_bound(k + span, r) * q
                assert x - y + off <= M32
                v[k], v[k + span] = x + y, shoup(x - y + off, tw(r, k), q)


def settle(v, R, q):
    for k in range(1 << R):
        b = inv_bound(k, R)
        v[k] = shoup(v[k], 1, q) if b > 4 else csub(v[k], 2 * q) if b > 2 else v[k]
        assert v[k] < 2 * q


class Buf:
    """Word accesses per round: (thread, first word, words) triples."""

    def __init__(self, N):
        self.w, self.rounds = {}, []

    def round(self):
        self.rounds.append([])

    def note(self, b, addrs, width):
        assert all(a % width == 0 for a in addrs[::width])
        self.rounds[-1].append((b, [addrs[i] for i in range(0, len(addrs), width)], width))

    def worst(self):
        """Largest number of passes over the banks beyond the least one access needs."""
        worst = 1
        for rnd in self.rounds:
            per = 32 // rnd[0][2]      # threads served together
            for t0 in range(0, len(rnd), per):
                for i in range(len(rnd[t0][1])):
                    banks = {}
                    for _, addrs, width in rnd[t0:t0 + per]:
                        for a in range(addrs[i], addrs[i] + width):
                            banks.setdefault(a % 32, set()).add(a)
                    worst = max(worst, max(len(s) for s in banks.values()))
        return worst


def middle(buf, N, R, step, levels):
    S = N // 8
    buf.round()
    for b in range(S):
        for sb in range(b, N >> R, S):
            i, o = set_of(sb, step, R, N)
            base = (i << R) * step + o
            addrs = [pad(base) + pad(k * step) for k in range(1 << R)]
            assert addrs == [pad(base + k * step) for k in range(1 << R)]
            v = [buf.w[a] for a in addrs]
            levels(v, i)
            for a, x in zip(addrs, v):
                buf.w[a] = x
            if sb == b:
                buf.note(b, addrs, 1)


def forward(coef, q, N, T, buf):
    fw, _, fwl, _ = T
    logn, S, out = N.bit_length() - 1, N // 8, [None] * N
    buf.round()
    for b in range(S):
        v = [coef[b + k * S] for k in range(8)]
        fwd_levels(v, 3, 0, lambda r, k: fw[(1 << r) + (k >> (3 - r))][0], q)
        addrs = [pad(b) + pad(k * S) for k in range(8)]
        buf.w.update(zip(addrs, v))
        buf.note(b, addrs, 1)
    end, lvl = (logn - 3 if logn >= 6 else logn), 3
    while lvl < end:
        R, m0 = middle_levels(end - lvl), 1 << lvl
        middle(buf, N, R, N >> (lvl + R), lambda v, i: fwd_levels(
            v, R, lvl, lambda r, k: fw[(m0 << r) + (i << r) + (k >> (R - r))][0], q))
        lvl += R
    buf.round()
    for b in range(S):
        if logn < 6:
            for e in range(8):
                out[b + e * S] = buf.w[pad(brev(b + e * S, logn))]
            buf.note(b, [pad(brev(b, logn))], 1)
            continue
        addrs = [pad(8 * brev(b, logn - 3)) + k for k in range(8)]
        buf.note(b, addrs, 4)
        w = [buf.w[a] for a in addrs]
        t = fwl[b]
        tw = {(0, 0): t[0], (1, 0): t[1], (1, 4): t[2], (2, 0): t[4], (2, 2): t[5], (2, 4): t[6], (2, 6): t[7]}
        fwd_levels(w, 3, logn - 3, lambda r, k: tw[(r, k & ~((1 << (3 - r)) - 1))][0], q)
        for e, k in enumerate([0, 4, 2, 6, 1, 5, 3, 7]):
            out[b + e * S] = w[k]
    return out


def inverse(slots, q, N, T, buf):
    _, iv, _, ivf = T
    logn, S, out = N.bit_length() - 1, N // 8, [None] * N
    ninv = pow(N, q - 2, q)
    buf.round()
    for b in range(S):
        i = brev(b, logn - 3)
        v = [slots[b + e * S] for e in (0, 4, 2, 6, 1, 5, 3, 7)]
        if logn >= 6:
            t = ivf[b]
            tw = {(0, 0): t[0], (0, 2): t[1], (0, 4): t[2], (0, 6): t[3], (1, 0): t[4], (1, 4): t[5], (2, 0): t[6]}
            inv_levels(v, 3, lambda r, k: tw[(r, k & ~((2 << r) - 1))][0], q)
        else:
            inv_levels(v, 3, lambda r, k: iv[((N // 2) >> r) + (i << (2 - r)) + (k >> (r + 1))][0], q)
        settle(v, 3, q)
        addrs = [pad(8 * i) + k for k in range(8)]
        buf.w.update(zip(addrs, v))
        buf.note(b, addrs, 4)
    end, g = (logn - 3 if logn >= 6 else logn), 3
    while g < end:
        R, t0 = middle_levels(end - g), 1 << g

        def levels(v, i):
            inv_levels(v, R, lambda r, k: iv[((N // (2 * t0)) >> r) + (i << (R - 1 - r)) + (k >> (r + 1))][0], q)
            settle(v, R, q)
        middle(buf, N, R, t0, levels)
        g += R
    buf.round()
    for b in range(S):
        addrs = [pad(b) + pad(k * S) for k in range(8)]
        buf.note(b, addrs, 1)
        w = [buf.w[a] for a in addrs]
        if logn >= 6:
            inv_levels(w, 3, lambda r, k: iv[(4 >> r) + (k >> (r + 1))][0] if r < 2 else iv[1][0] * ninv % q, q)
            w = [csub(shoup(x, ninv, q) if k < 4 else x, q) for k, x in enumerate(w)]
        else:
            w = [csub(shoup(x, ninv, q), q) for x in w]
        for k in range(8):
            out[b + k * S] = w[k]
    return out


@pytest.mark.parametrize("logn", list(range(4, 13)))
def test_transforms_match_the_oracle_within_their_bounds(logn):
    N = 1 << logn
    rng = np.random.default_rng(100 + logn)
    for q in synth.PRIMES_28:
        T = tables(q, N)
        a = [int(x) for x in rng.integers(0, q, N)]
        want = [int(x) for x in oracle.ntt_negacyclic(a, q, oracle.psi_2n(q, N))]
        fb, ib = Buf(N), Buf(N)
        got = forward([x + q if i % 3 == 0 else x for i, x in enumerate(a)], q, N, T, fb)
        assert all(x < 16 * q for x in got) and [x % q for x in got] == want
        assert inverse([x + q if i % 3 == 0 else x for i, x in enumerate(want)], q, N, T, ib) == a
        if N == 4096:
            assert fb.worst() == 1 and ib.worst() == 1


def test_bounds_hold_for_the_largest_modulus():
    assert 16 * TOP <= 1 << 32
    assert all(fwd_bound(l) <= 16 for l in range(13))
    assert [inv_bound(k, 3) for k in range(8)] == [16, 8, 4, 4, 2, 2, 2, 2]


@pytest.mark.parametrize("primes", [synth.PRIMES_28, synth.PRIMES_28[:1], synth.PRIMES_28[::-1], (97, 193), (193, 97),
                                    (97,), (268369921, 97)], ids=str)
def test_digit_fields_match_the_oracle(primes):
    """Garner with a multiple of q1 in place of a conditional subtraction, the offset value from two constants, and
    each masked field plus its addend: nonnegative, congruent to the balanced digit, below 2q for 28-bit primes."""
    z, Q = 1 << 22, int(np.prod([int(q) for q in primes], dtype=object))
    ell = max(1, oracle.gadget_digits(primes))
    off = sum((z // 2) << (22 * k) for k in range(ell - 1))
    rng = np.random.default_rng(7)
    xs = [int(v) for v in rng.integers(0, Q, 3000)] + [0, 1, Q - 1, Q // 2, Q // 2 + 1]
    for x in xs:
        y0 = x % primes[0]
        if len(primes) == 2:
            q0, q1 = primes
            add = -(-q0 // q1) * q1
            v = x % q1 + add - y0
            assert 0 <= v <= M32
            k = csub(shoup(v, pow(q0, -1, q1), q1), q1)
            assert y0 + q0 * k == x
        y = x + (off - Q if x > Q // 2 else off)
        want = oracle.balanced_digits(x - Q if x > Q // 2 else x, z, ell)
        for i in range(ell):
            top = i + 1 == ell
            f = ((y >> (22 * i)) & M32) & (M32 if top else z - 1)
            for q in primes:
                up = -(-(z // 2 + 1) // q) * q
                d = (f + (up if top else up - z // 2)) & M32
                assert d % q == want[i] % q and d < max(2 * q, 1 << 24)


def test_two_quotient_reduction():
    """hi 2^32 + lo below 4q for any 64-bit value, and the tree sums fit 64 bits."""
    rng = np.random.default_rng(9)
    for q in list(synth.PRIMES_28) + [97, TOP]:
        r32, one = (1 << 32) % q, (1 << 32) // q
        xs = [0, q - 1, q, M32, (1 << 64) - 1, ((1 << 64) // q) * q - 1]
        xs += [int(v) for v in rng.integers(0, (1 << 64) - 1, 2000, dtype=np.uint64)]
        for x in xs:
            hi, lo = x >> 32, x & M32
            r = (hi * r32 + lo - (((hi * ((r32 << 32) // q)) >> 32) + ((lo * one) >> 32)) * q) & M32
            assert r < 4 * q and r % q == x % q
    assert 3 * (16 * TOP) * TOP + (4 + 1) * TOP < 1 << 64
