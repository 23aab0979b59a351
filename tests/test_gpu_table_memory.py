"""Device memory of freed join tables is kept for the next one: reuse leaves
no trace in a table's contents, the amount kept is bounded, contexts with a
budget take no part, threads share it safely, and it is given back with the
last context."""
import gc
import threading

import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _join(ctx, n, seed, load=0.0):
    b = datagen.join_build(n, "mult14", seed=seed)
    p = datagen.join_probe(20_000, b, 0.5, "uniform", seed=seed)
    t = ctx.join_build(torch.from_numpy(b.keys).cuda(), None, load)
    got = ctx.join_probe(t, p.keys).astype(np.uint64)
    t.free()
    np.testing.assert_array_equal(np.sort((got[:, 0] << np.uint64(32)) | got[:, 1]), oracle.join(b.keys, p.keys))


def _free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_reuse_bounds_and_return():
    gc.collect()
    torch.cuda.empty_cache()                   # what other tests left cached is not counted
    with olap.Context(0) as warm:
        _join(warm, 1000, 1)
    torch.cuda.empty_cache()
    before = _free_bytes()
    with olap.Context(0) as ctx:
        for i, n in enumerate((200_000, 190_000, 1000, 200_000, 150_000, 300_000)):     # larger, smaller, reused
            _join(ctx, n, 30 + i, (0.5, 0.7, 0.9)[i % 3])
        keys = torch.randint(-(1 << 62), 1 << 62, (1 << 24,), device="cuda")
        tables = [ctx.join_build(keys) for _ in range(4)]                               # a gigabyte each
        for t in tables:
            t.free()
        assert before - _free_bytes() < (3 << 30) + keys.numel() * 8                    # two of the four kept at most
        del keys, tables
        torch.cuda.empty_cache()
    assert abs(before - _free_bytes()) < (64 << 20)


def test_budgeted_contexts_free_at_once():
    with olap.Context(0, mem_budget_bytes=1 << 30) as ctx:
        _join(ctx, 1000, 2)
        before = _free_bytes()
        _join(ctx, 400_000, 3)
        assert before - _free_bytes() < (24 << 20)                                      # scratch of the calls, no table


def test_threads():
    errors = []

    def work(seed):
        try:
            with olap.Context(0) as ctx:
                for i in range(6):
                    _join(ctx, 50_000 + 7000 * ((seed + i) % 3), 100 + seed * 10 + i)
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)
    ts = [threading.Thread(target=work, args=(s,)) for s in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors[0]
