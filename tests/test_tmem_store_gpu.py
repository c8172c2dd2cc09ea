"""Output rows of the tensor-memory kernel (tile variant 8,
csrc/rowsel_tmem.cu) against the oracle: the store warps take rows in steps of
four, alternately, so batches whose last row block ends inside a step and
column blocks that end inside a half of 32 are written to a buffer with a
guard behind it."""

import numpy as np
import pytest
import torch

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


@pytest.mark.parametrize("B", [9, 16, 17, 18, 20, 31])
@pytest.mark.parametrize("D0,D1", [(65, 33), (64, 1), (130, 95)])
def test_partial_row_steps(g, B, D0, D1):
    from tests.gpu_util import DbHandle, make_problem, to_dev, to_host
    L, N, primes = 2, 32, synth.PRIMES_28[:2]
    ct, db = make_problem(31 * B + D1, B, D0, D1, L, N, primes)
    want = oracle.rowsel(ct, db, list(primes))
    size = want.size
    buf = torch.full((size + 64,), -1, dtype=torch.int32, device="cuda")
    h = DbHandle(g, db, N, primes)
    try:
        g.gpir_set_variant(h.h, B, g.GPIR_PATH_TC, 8)
        h.rowsel(to_dev(ct), B, g.GPIR_PATH_TC, out=buf[:size].view(want.shape))
    finally:
        h.close()
    got = to_host(buf)
    assert np.array_equal(got[:size].reshape(want.shape), want)
    assert (got[size:] == 0xFFFFFFFF).all()
