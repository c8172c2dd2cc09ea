"""The streaming tensor-core kernel (tile variant 12, csrc/rowsel_stream.cu)
against the oracle: edges of its tiles (8 slots, 16 rows, 32 columns, 64-row
steps, 256-row exact groups), digits at their bounds, several jobs in one
launch, and the calls that choose it by themselves."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

STREAM = 12
P28 = synth.PRIMES_28


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


def _run(g, ct, db, N, primes, variant=STREAM, path=4):
    from tests.gpu_util import DbHandle, to_dev, to_host
    h = DbHandle(g, db, N, primes, path_mask=0)
    try:
        if variant is not None:
            g.gpir_set_variant(h.h, ct.shape[0], g.GPIR_PATH_TC, variant)
        return to_host(h.rowsel(to_dev(ct), ct.shape[0], path))
    finally:
        h.close()


SHAPES = [
    # (B, D0, D1, L, N)
    (1, 1, 1, 1, 4),        # half a slot group, one of everything
    (4, 64, 32, 2, 8),      # exactly one box, one step, one column block
    (5, 65, 33, 2, 16),     # one past each
    (8, 256, 31, 1, 64),    # a full row block, a full exact group
    (9, 257, 64, 2, 32),    # two row blocks, a second group of one row
    (17, 63, 90, 2, 16),    # three row blocks, three column blocks, one short step
    (12, 600, 5, 1, 128),   # three groups
    (3, 40, 70, 2, 2048),   # more units than SMs
]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "B%d_%dx%d_L%d_N%d" % s)
def test_against_the_oracle(g, shape):
    from tests.gpu_util import make_problem
    B, D0, D1, L, N = shape
    primes = P28[:L]
    ct, db = make_problem(3000 + D0 + B, B, D0, D1, L, N, primes)
    assert np.array_equal(_run(g, ct, db, N, primes), oracle.rowsel(ct, db, list(primes)))


def test_digits_at_their_bounds(g):
    """Database fields of 127 against ciphertext digits of -512 and 511 over full 256-row groups: the partial sums
    reach 127 * 512 * 256, just below 2^24, and neighbouring integers must stay apart."""
    B, D0, D1, L, N = 8, 512, 32, 1, 8
    q = P28[0]
    db = np.full((D0, D1, L, N), 0xFFEFFFF, dtype=np.uint32)   # fields 127, 127, 123, 127
    db[:, 1::3] = 0x7F
    db[5, ::2] = 0xFFEFFFE
    ct = np.zeros((B, D0, 2, L, N), dtype=np.uint32)           # digits -512, -512, -128
    ct[1::2] = 0x00FFFFF                                       # digits 511, 511, -128
    ct[2, :, 1] = 0xFF003FF
    ct[:, 300:, :, :, 3] = q - 1
    assert int(ct.max()) < q and int(db.max()) < q
    assert np.array_equal(_run(g, ct, db, N, P28[:1]), oracle.rowsel(ct, db, [q]))


def test_several_jobs_in_one_launch(g):
    """Nine jobs of uneven shapes (two launches) through gpir_rowsel_multi, twice, equal to the oracle."""
    import torch
    from tests.gpu_util import DbHandle, make_problem, to_dev, to_host
    L, N = 2, 1024
    shapes = [(9, 70, 33), (16, 130, 20), (8, 300, 64), (12, 64, 32), (10, 20, 90), (8, 257, 7), (11, 65, 65), (17, 40, 40),
              (9, 10, 10)]
    hs, jobs, want = [], [], []
    try:
        for k, (B, D0, D1) in enumerate(shapes):
            ct, db = make_problem(3100 + k, B, D0, D1, L, N, P28)
            h = DbHandle(g, db, N, P28, path_mask=0)
            g.gpir_set_variant(h.h, B, g.GPIR_PATH_TC, STREAM)
            out = torch.full((B, D1, 2, L, N), -1, dtype=torch.int32, device="cuda")
            hs.append(h)
            jobs.append((h.h, B, to_dev(ct), out))
            want.append(oracle.rowsel(ct, db, list(P28)))
        for path in (g.GPIR_PATH_TC, g.GPIR_PATH_AUTO):
            for j in jobs:
                j[3].fill_(-1)
            g.gpir_rowsel_multi(jobs, path)
            g.gpir_sync(None, 20000)
            for (_, _, _, out), w in zip(jobs, want):
                assert np.array_equal(to_host(out), w)
    finally:
        for h in hs:
            h.close()


@pytest.mark.parametrize("nth", [4, 5])
def test_upload_without_room_for_its_tiles(g, nth):
    """A database whose streaming tiles cannot be allocated (the fourth and
    fifth allocation of an upload) is served by the other kernels, by itself,
    in a multi-job call and where the streaming variant is asked for."""
    import torch
    from tests.gpu_util import to_dev, to_host
    B, D0, D1, L, N = 4, 40, 24, 2, 2048
    ct = synth.ct_tensor(77, B, D0, L, N, P28)
    db = synth.db_tensor(77, D0, D1, L, N, P28)
    want = oracle.rowsel(ct, db, list(P28))
    params = g.gpir_params_create(N, list(P28))
    h = None
    try:
        g.gpir_set_fail_alloc(nth)
        h = g.gpir_db_upload(params, D0, D1, to_dev(db), True, 0)
        assert g.gpir_set_fail_alloc(0) == 0
        ctd, out = to_dev(ct), torch.empty((B, D1, 2, L, N), dtype=torch.int32, device="cuda")
        for path in (g.GPIR_PATH_AUTO, g.GPIR_PATH_TC):
            out.fill_(-1)
            g.gpir_rowsel_batch(h, B, ctd, out, path)
            g.gpir_sync(None, 20000)
            assert np.array_equal(to_host(out), want)
        g.gpir_set_variant(h, B, g.GPIR_PATH_TC, STREAM)
        out.fill_(-1)
        g.gpir_rowsel_multi([(h, B, ctd, out)], g.GPIR_PATH_TC)
        g.gpir_sync(None, 20000)
        assert np.array_equal(to_host(out), want)
    finally:
        g.gpir_set_fail_alloc(0)
        if h is not None:
            g.gpir_db_free(h)
        g.gpir_params_destroy(params)
