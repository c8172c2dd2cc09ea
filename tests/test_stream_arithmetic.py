"""CPU model of the streaming kernel's arithmetic (csrc/rowsel_stream.cu): the
database's 7-bit fields, the ciphertexts' offset base-2^10 digits, fp32 sums of
256 rows in any order, the weights and the column correction, against exact
integers, at the largest digits as well as random ones."""

import numpy as np
import pytest

import synth

OFF = 512 + 512 * (1 << 10) + 128 * (1 << 20)


def _model(ct, db, q, corr_of=lambda s, q: OFF % q * s % q):
    """ct [M][K], db [K][n] -> ct @ db mod q by the kernel's steps."""
    M, K = ct.shape
    f = [(db >> (7 * u)) & 127 for u in range(4)]
    d = [((ct >> (10 * v)) & 1023) - (512, 512, 128)[v] for v in range(3)]
    assert max(int(x.max()) for x in d) <= 511 and min(int(x.min()) for x in d) >= -512
    total = np.zeros((M, db.shape[1]), dtype=object)
    for k0 in range(0, K, 256):
        k = slice(k0, min(K, k0 + 256))
        for u in range(4):
            for v in range(3):
                a, b = d[v][:, k].astype(np.float16), f[u][k].astype(np.float16)
                acc = np.zeros((M, db.shape[1]), dtype=np.float32)
                for i in np.random.default_rng(k0 + u).permutation(a.shape[1]):   # any order of additions
                    acc = acc + a[:, i, None].astype(np.float32) * b[None, i].astype(np.float32)
                assert np.abs(acc).max() <= 1 << 24 and (acc == np.rint(acc)).all()
                w = pow(2, 7 * u + 10 * v, q)
                total += acc.astype(np.int64).astype(object) * w
    s = db.astype(object).sum(axis=0) % q
    corr = np.array([corr_of(int(x), q) for x in s], dtype=object)
    return (total + corr[None, :]) % q


@pytest.mark.parametrize("K", [1, 63, 256, 300])
@pytest.mark.parametrize("q", list(synth.PRIMES_28))
@pytest.mark.parametrize("kind", ["random", "largest", "zero"])
def test_digits_sums_and_correction(K, q, kind):
    rng = np.random.default_rng(K + q % 97)
    ct, db = rng.integers(0, q, (4, K)), rng.integers(0, q, (K, 5))
    if kind == "largest":   # every field and digit at a bound
        ct[0], ct[1], ct[2] = q - 1, (1 << 20) - 1, 1023
        db[:] = min(q - 1, (127 << 14) | (127 << 7) | 127)
    elif kind == "zero":
        ct[:2], db[:, :2] = 0, 0
    want = (ct.astype(object) @ db.astype(object)) % q
    assert (_model(ct, db, q) == want).all()


def test_a_missing_correction_shows():
    q = synth.PRIMES_28[0]
    rng = np.random.default_rng(5)
    ct, db = rng.integers(0, q, (2, 40)), rng.integers(1, q, (40, 3))
    want = (ct.astype(object) @ db.astype(object)) % q
    assert (_model(ct, db, q, lambda s, q: 0) != want).any()
