"""Tree stages that start while the stage before them finishes: calls queued
one after another on one stream, whose inputs the host side of the stream
changes in between, against the oracle. The sizes cross the rule for ColTor's
overlapping stages (a stage whose CTAs the chip holds at once) and both of
ExpandQuery's forms."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

P28 = synth.PRIMES_28


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


@pytest.mark.parametrize("B,D1,L,N", [(20, 16, 2, 64), (1, 8, 2, 4096), (3, 32, 1, 128)])
def test_coltor_calls_in_a_row(g, B, D1, L, N):
    import torch
    from tests.gpu_util import to_dev, to_host
    primes = P28[:L]
    ell, stages, calls = oracle.gadget_digits(primes), D1.bit_length() - 1, 3
    cts = [synth.uniform_residues(40 + i, synth.TAG_COLTOR, (B, D1, 2, L, N), primes, limb_axis=3) for i in range(calls)]
    rgsw = synth.uniform_residues(47, synth.TAG_RGSW, (B, stages, 2 * ell, 2, L, N), primes, limb_axis=4)
    params = g.gpir_params_create(N, list(primes))
    try:
        dev, key = [to_dev(x) for x in cts], to_dev(rgsw)
        ct = torch.empty_like(dev[0])
        outs = [torch.full((B, 2, L, N), -1, dtype=torch.int32, device="cuda") for _ in range(calls)]
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for x, out in zip(dev, outs):
                ct.copy_(x)
                g.gpir_coltor(params, B, D1, ct, key, out, s)
        s.synchronize()
        for x, out in zip(cts, outs):
            got = to_host(out)
            for c in range(0, B, max(1, B // 3)):
                assert np.array_equal(got[c], oracle.coltor(x[c], rgsw[c], primes))
    finally:
        g.gpir_params_destroy(params)


@pytest.mark.parametrize("B,J,n_out,L,N", [(20, 4, 13, 2, 64), (2, 3, 8, 2, 2048), (40, 3, 7, 1, 128)])
def test_expand_calls_in_a_row(g, B, J, n_out, L, N):
    import torch
    from tests.gpu_util import to_dev, to_host
    primes = P28[:L]
    ell, calls = oracle.gadget_digits(primes), 3
    qs = [synth.uniform_residues(60 + i, synth.TAG_COLTOR, (B, 2, L, N), primes, limb_axis=2) for i in range(calls)]
    evk = synth.uniform_residues(67, synth.TAG_RGSW, (B, J, ell, 2, L, N), primes, limb_axis=4)
    params = g.gpir_params_create(N, list(primes))
    try:
        dev, key = [to_dev(x) for x in qs], to_dev(evk)
        q = torch.empty_like(dev[0])
        outs = [torch.full((B, n_out, 2, L, N), -1, dtype=torch.int32, device="cuda") for _ in range(calls)]
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for x, out in zip(dev, outs):
                q.copy_(x)
                g.gpir_expand_query(params, B, J, n_out, q, key, out, s)
        s.synchronize()
        for x, out in zip(qs, outs):
            got = to_host(out)
            for c in range(0, B, max(1, B // 3)):
                assert np.array_equal(got[c], oracle.expand_query(x[c], evk[c], primes, n_out))
    finally:
        g.gpir_params_destroy(params)
