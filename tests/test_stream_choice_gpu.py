"""Which path untuned batches of up to 8 clients take by themselves
(GPIR_PATH_AUTO) on either side of the rule between the CUDA cores and the
streaming kernel, and that the answers are the oracle's on both."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

CC, TC = 1, 4


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


def _db(g, N, L, D0, D1):
    """A database of that shape from the device-side fill (no host copy), with its parameter set."""
    import torch
    primes = synth.PRIMES_28[:L]
    params = g.gpir_params_create(N, list(primes))
    buf = torch.empty(D0 * D1 * L * N, dtype=torch.int32, device="cuda")
    g.gpir_fill_uniform(buf, buf.numel(), 0, 5, 6, params, N)
    return params, g.gpir_db_upload(params, D0, D1, buf, True, 0)


# (N, L, D0, D1): path of 1 to 8 clients. The sizes are clear of the rule's line on any GPU of 140 to 160 SMs.
CHOICES = [
    ((4096, 2, 256, 64), [CC] + [TC] * 7),
    ((4096, 2, 192, 32), [CC] * 4 + [TC] * 4),            # 2 to 4 clients: above 192 rows only
    ((4096, 2, 208, 32), [CC] + [TC] * 7),
    ((4096, 1, 16, 8), [CC] * 7 + [TC]),                  # few rows: one padded step
    ((2048, 1, 32, 48), [CC] * 7 + [TC]),
    ((4096, 1, 100, 8), [CC] * 4 + [TC] * 4),
    ((2048, 1, 257, 33), [CC] * 4 + [TC] * 4),            # four streaming waves for one, a group of one row
    ((256, 1, 257, 192), [CC] + [TC] * 7),                # two full waves: worth it
    ((256, 1, 1024, 32), [CC] * 7 + [TC]),                # fewer units than SMs
]


@pytest.mark.parametrize("shape,want", CHOICES, ids=["N%d_L%d_%dx%d" % c[0] for c in CHOICES])
def test_path_of_untuned_batches(g, shape, want):
    import torch
    if not 140 <= torch.cuda.get_device_properties(0).multi_processor_count <= 160:
        pytest.skip("the sizes are those of a GB300's SM count")
    params, h = _db(g, *shape)
    try:
        assert [g.gpir_selected_path(h, b) for b in range(1, 9)] == want
        assert all(g.gpir_selected_variant(h, b, TC) == -1 for b in range(1, 9))   # none forced
    finally:
        g.gpir_db_free(h)
        g.gpir_params_destroy(params)


@pytest.mark.parametrize("N,L,D0,D1", [(2048, 1, 16, 20), (1024, 2, 66, 20), (2048, 1, 258, 20)])
@pytest.mark.parametrize("B", [1, 2, 4, 5, 7, 8])
def test_untuned_batches_against_the_oracle(g, N, L, D0, D1, B):
    from tests.gpu_util import DbHandle, make_problem, to_dev, to_host
    primes = synth.PRIMES_28[:L]
    ct, db = make_problem(4000 + D0 + B, B, D0, D1, L, N, primes)
    h = DbHandle(g, db, N, primes)
    try:
        assert np.array_equal(to_host(h.rowsel(to_dev(ct), B, g.GPIR_PATH_AUTO)), oracle.rowsel(ct, db, list(primes)))
    finally:
        h.close()
