"""The streaming kernel's tiles are optional device memory: an upload takes them
only where an eighth of the device stays free, and they are given back when a
later allocation of the library finds the device full, unless a captured launch
refers to them. The device is filled up to a gibibyte or more, never to the end."""

import pytest

import synth

pytestmark = pytest.mark.gpu

GIB = 1 << 30
N, L, PRIMES = 4096, 2, synth.PRIMES_28
B = 4
STREAM = 12


@pytest.fixture(scope="module")
def g():
    from tests import gpu_util
    return gpu_util.lib()


@pytest.fixture
def params(g):
    import torch
    p = g.gpir_params_create(N, list(PRIMES))
    yield p
    g.gpir_params_destroy(p)
    torch.cuda.empty_cache()


def _residues(g, params, words, seed):
    import torch
    t = torch.empty(words, dtype=torch.int32, device="cuda")
    g.gpir_fill_uniform(t, words, 0, seed, 3, params, N)
    return t


def _fill(leave):
    """Device memory held so that about `leave` bytes stay free."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    while True:
        n = min(8 * GIB, torch.cuda.mem_get_info()[0] - leave) >> 21 << 21
        if n < 1 << 25:
            return held
        held.append(torch.empty(n, dtype=torch.uint8, device="cuda"))


def _without_tiles(D0, D1):
    return D0 * D1 * L * N * (4 + 8 + 6)   # whole tiles of 64 x 64


def _answer(g, h, D1, ct, path):
    import torch
    out = torch.full((B * D1 * 2 * L * N,), -1, dtype=torch.int32, device="cuda")
    g.gpir_rowsel_batch(h, B, ct, out, path)
    g.gpir_sync(None, 20000)
    return out


def test_an_eighth_of_the_device_stays_free(g, params):
    import torch
    D0, D1 = 256, 64
    db, ct = _residues(g, params, D0 * D1 * L * N, 1), _residues(g, params, B * D0 * 2 * L * N, 2)
    answers = []
    for spare, tiles in ((GIB // 4, False), (GIB, True)):   # the tiles take half a gibibyte
        held = _fill(torch.cuda.mem_get_info()[1] // 8 + _without_tiles(D0, D1) + spare)
        h = g.gpir_db_upload(params, D0, D1, db, True, 0)
        del held
        try:
            assert (g.gpir_db_device_bytes(h) > _without_tiles(D0, D1)) == tiles
            answers += [_answer(g, h, D1, ct, path) for path in (g.GPIR_PATH_AUTO, g.GPIR_PATH_TC)]
        finally:
            g.gpir_db_free(h)
    assert all(torch.equal(a, answers[0]) for a in answers)


@pytest.mark.parametrize("captured", [False, True], ids=["idle", "captured"])
def test_tiles_are_given_back_when_the_device_is_full(g, params, captured):
    import torch
    D0, D1 = 512, 64                                       # 1 GiB, its tiles another
    db, ct = _residues(g, params, D0 * D1 * L * N, 3), _residues(g, params, B * D0 * 2 * L * N, 4)
    h = h2 = graph = None
    stream = torch.cuda.Stream()
    try:
        h = g.gpir_db_upload(params, D0, D1, db, True, 0)
        with_tiles = g.gpir_db_device_bytes(h)
        assert with_tiles > _without_tiles(D0, D1)
        g.gpir_set_variant(h, B, g.GPIR_PATH_TC, STREAM)
        want = _answer(g, h, D1, ct, g.GPIR_PATH_TC)
        if captured:
            out = torch.full_like(want, -1)
            torch.cuda.synchronize()
            graph = g.gpir_graph_create([(h, B, ct, out)], g.GPIR_PATH_TC, stream)
        half = db[:db.numel() // 2].clone()                # a database of half the rows: 2.25 GiB
        del db
        held = _fill(3 * GIB // 2)
        if captured:
            with pytest.raises(g.GpirError) as ei:
                g.gpir_db_upload(params, D0 // 2, D1, half, True, 0)
            assert ei.value.code == g.GPIR_ENOMEM
            assert g.gpir_db_device_bytes(h) == with_tiles
            out.fill_(-1)
            torch.cuda.synchronize()
            g.gpir_graph_launch(graph, stream)
            g.gpir_sync(stream, 20000)
            assert torch.equal(out, want)
        else:
            h2 = g.gpir_db_upload(params, D0 // 2, D1, half, True, 0)
            assert g.gpir_db_device_bytes(h) == _without_tiles(D0, D1)
        del held
        torch.cuda.empty_cache()
        for path in (g.GPIR_PATH_AUTO, g.GPIR_PATH_TC):
            assert torch.equal(_answer(g, h, D1, ct, path), want)
    finally:
        if graph is not None:
            g.gpir_graph_destroy(graph)
        for x in (h, h2):
            if x is not None:
                g.gpir_db_free(x)
