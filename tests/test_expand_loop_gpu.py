"""ExpandQuery stages of more nodes than resident clusters, where each cluster
of the persistent kernel runs several nodes in turn (reusing its shared memory,
with the next node's input copied ahead), and buffers off a 16-byte boundary,
which are read with plain loads instead of bulk copies, in both stage kernels.
Against the oracle, bit-exact."""

import numpy as np
import pytest

import oracle
import synth
from tests import expand_util as eu

pytestmark = pytest.mark.gpu

P28 = synth.PRIMES_28


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


def _clients(J, n_out, L, N):
    """Clients whose last stage has a little over two nodes for every resident cluster."""
    import torch
    threads = N // 8 if N >= 256 else 32
    resident = torch.cuda.get_device_properties(0).multi_processor_count * min(16, 1024 // threads) // L
    return (2 * resident + 7) // min(1 << (J - 1), n_out) + 1


def _check(g, B, J, n_out, L, N, off_query, off_out, seed):
    import torch
    from tests.gpu_util import to_dev, to_host
    primes = P28[:L]
    ell, kinds = oracle.gadget_digits(primes), 2 if N > 2048 else 3   # clients c, c + kinds, ... have the same inputs
    query = synth.uniform_residues(seed, eu.TAG_QUERY, (kinds, 2, L, N), primes, limb_axis=2)
    evk = synth.uniform_residues(seed + 1, eu.TAG_EVK, (kinds, J, ell, 2, L, N), primes, limb_axis=4)
    of = torch.arange(B, device="cuda") % kinds
    q = torch.empty(B * 2 * L * N + off_query, dtype=torch.int32, device="cuda")[off_query:]
    q.copy_(to_dev(query)[of].view(-1))
    size = B * n_out * 2 * L * N
    buf = torch.full((size + off_out + 64,), -1, dtype=torch.int32, device="cuda")
    out = buf[off_out:off_out + size]
    assert (q.data_ptr() % 16 == 0) == (off_query == 0) and (out.data_ptr() % 16 == 0) == (off_out == 0)
    params = g.gpir_params_create(N, list(primes))
    try:
        g.gpir_expand_query(params, B, J, n_out, q, to_dev(evk)[of], out)
        g.gpir_sync(None, 20000)
    finally:
        g.gpir_params_destroy(params)
    assert bool((buf[:off_out] == -1).all()) and bool((buf[off_out + size:] == -1).all())
    got = to_host(out).reshape(B, n_out, 2, L, N)
    for k in range(kinds):
        want = oracle.expand_query(query[k], evk[k], primes, n_out)
        for c in range(k, B, kinds):
            assert np.array_equal(got[c], want), "client %d of %d" % (c, B)


@pytest.mark.parametrize("J,n_out,L,N", [(5, 32, 1, 32), (5, 27, 2, 32), (4, 16, 1, 16), (3, 7, 1, 512), (1, 2, 1, 4096),
                                         (1, 2, 2, 4096)])
def test_clusters_run_several_nodes(g, J, n_out, L, N):
    _check(g, _clients(J, n_out, L, N), J, n_out, L, N, 0, 0, 7000 + N + L)


@pytest.mark.parametrize("off_query,off_out", [(1, 0), (0, 2)])
@pytest.mark.parametrize("J,n_out,L,N,loop", [(3, 7, 2, 64, False), (1, 2, 1, 1024, False), (5, 32, 1, 32, True),
                                              (2, 4, 2, 1024, True)])
def test_buffers_off_a_16_byte_boundary(g, J, n_out, L, N, loop, off_query, off_out):
    B = _clients(J, n_out, L, N) if loop else 3
    _check(g, B, J, n_out, L, N, off_query, off_out, 7100 + N + L)
