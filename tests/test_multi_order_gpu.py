"""A call over several databases whose tensor-memory jobs cannot have their
workspace returns GPIR_ENOMEM and has launched nothing: the outputs of the jobs
that need none (streaming kernel, CUDA cores) are untouched. The same call then
succeeds, equal to the oracle."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


@pytest.mark.parametrize("auto", [False, True], ids=["tc", "auto"])
def test_nothing_runs_without_the_workspace(g, auto):
    import torch
    from tests.gpu_util import DbHandle, make_problem, to_dev, to_host
    L, N, primes = 2, 1024, synth.PRIMES_28
    hs, jobs, want = [], [], []
    stream = torch.cuda.Stream()                     # has no workspace yet
    try:
        # the streaming kernel's, the tensor-memory kernel's and (auto) the CUDA cores'
        for k, (B, D0, D1, variant) in enumerate([(5, 70, 20, 12), (16, 65, 33, 8), (1, 40, 30, None)][:3 if auto else 2]):
            ct, db = make_problem(5100 + k, B, D0, D1, L, N, primes)
            h = DbHandle(g, db, N, primes)
            hs.append(h)
            if variant is not None:
                g.gpir_set_variant(h.h, B, g.GPIR_PATH_TC, variant)
            out = torch.full((B, D1, 2, L, N), -1, dtype=torch.int32, device="cuda")
            jobs.append((h.h, B, to_dev(ct), out))
            want.append(oracle.rowsel(ct, db, list(primes)))
        torch.cuda.synchronize()
        path = g.GPIR_PATH_AUTO if auto else g.GPIR_PATH_TC
        g.gpir_set_fail_alloc(1)
        with pytest.raises(g.GpirError) as ei:
            g.gpir_rowsel_multi(jobs, path, stream)
        assert ei.value.code == g.GPIR_ENOMEM
        assert g.gpir_set_fail_alloc(0) == 0
        stream.synchronize()
        for _, _, _, out in jobs:
            assert bool((out == -1).all())
        g.gpir_rowsel_multi(jobs, path, stream)
        stream.synchronize()
        for (_, _, _, out), w in zip(jobs, want):
            assert np.array_equal(to_host(out), w)
    finally:
        g.gpir_set_fail_alloc(0)
        for h in hs:
            h.close()
