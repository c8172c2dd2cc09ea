"""The tensor-memory kernel (tile variant 8, csrc/rowsel_tmem.cu) on either side
of its rule for the second store warp (units of fewer than 7 k-chunks of 64
rows), against the oracle: partial row steps and column halves, one job and
several whose rows lie on both sides, guarded outputs."""

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu

L, N, PRIMES = 2, 32, synth.PRIMES_28[:2]


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


def _jobs(g, shapes):
    from tests.gpu_util import DbHandle, make_problem, to_dev
    out = []
    for B, D0, D1 in shapes:
        ct, db = make_problem(17 * B + D0 + D1, B, D0, D1, L, N, PRIMES)
        h = DbHandle(g, db, N, PRIMES)
        g.gpir_set_variant(h.h, B, g.GPIR_PATH_TC, 8)
        want = oracle.rowsel(ct, db, list(PRIMES))
        buf = torch.full((want.size + 64,), -1, dtype=torch.int32, device="cuda")
        out.append((h, B, to_dev(ct), buf, want))
    return out


def _check(jobs):
    from tests.gpu_util import to_host
    for _, _, _, buf, want in jobs:
        got = to_host(buf)
        assert np.array_equal(got[:want.size].reshape(want.shape), want)
        assert (got[want.size:] == 0xFFFFFFFF).all()


@pytest.mark.parametrize("B", [9, 16, 19, 34])
@pytest.mark.parametrize("D0,D1", [(384, 33), (385, 33), (448, 64), (449, 95), (513, 1), (1025, 70)])
def test_one_job(g, B, D0, D1):
    jobs = _jobs(g, [(B, D0, D1)])
    try:
        for h, b, ct, buf, want in jobs:
            h.rowsel(ct, b, g.GPIR_PATH_TC, out=buf[:want.size].view(want.shape))
        _check(jobs)
    finally:
        for j in jobs:
            j[0].close()


@pytest.mark.parametrize("shapes", [
    [(9, 64, 33), (17, 384, 20)],                  # all short
    [(16, 40, 33), (11, 500, 65), (20, 130, 7)],   # one long
    [(10, 449, 64), (18, 700, 31)],                # all long
], ids=["short", "mixed", "long"])
def test_several_jobs(g, shapes):
    jobs = _jobs(g, shapes)
    try:
        g.gpir_rowsel_multi([(h.h, b, ct, buf[:want.size].view(want.shape)) for h, b, ct, buf, want in jobs],
                            g.GPIR_PATH_TC)
        g.gpir_sync(None, 20000)
        _check(jobs)
    finally:
        for j in jobs:
            j[0].close()
