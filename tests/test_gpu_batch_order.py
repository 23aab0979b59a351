"""Batches whose Top-K and probe items share memory that one of them writes
run every probe first, against the CPU oracle: a Top-K over the pairs a probe
appends, and a probe of keys that a Top-K then overwrites, over several runs."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = olap.Context(0)
    yield c
    c.close()


def _top(keys, k, order, ok=None):
    ok = torch.empty(k, dtype=torch.int64, device="cuda") if ok is None else ok
    orow = torch.empty(k, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    return olap.topk_item(keys, k, order, ok, orow, cnt), (ok, orow, cnt)


@pytest.mark.parametrize("n", [1000, 200_003])
def test_topk_over_a_probes_pairs(ctx, n):
    build = datagen.splitmix64(1, 5000).view(np.int64)
    t = ctx.join_build(torch.from_numpy(build).cuda())
    other = torch.from_numpy(datagen.splitmix64(3, 300_000).view(np.int64).copy()).cuda()
    probe = torch.zeros(n, dtype=torch.int64, device="cuda")
    pairs = torch.full((n, 2), -7, dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    item, (ok, orow, _) = _top(pairs.view(torch.int64).view(-1), 100, olap.ASC)
    busy, _held = _top(other, 1000, olap.DESC)
    b = ctx.batch([busy, item, olap.probe_item(t, probe, pairs, n, cnt)])
    for seed in range(3):
        pk = build[(datagen.splitmix64(10 + seed, n) % np.uint64(5000)).astype(np.int64)]
        probe.copy_(torch.from_numpy(pk))
        b.run()
        ctx.sync()
        assert int(cnt.item()) == n
        got = pairs.view(torch.int64).view(-1).cpu().numpy()
        np.testing.assert_array_equal(np.sort(got.view(np.uint64)), np.sort(
            ((oracle.join(build, pk) & np.uint64(0xFFFFFFFF)) << np.uint64(32)) | (oracle.join(build, pk) >> np.uint64(32))))
        wk, wr = oracle.topk(got, 100, olap.ASC)
        np.testing.assert_array_equal(ok.cpu().numpy(), wk)
        np.testing.assert_array_equal(orow.cpu().numpy().view(np.uint32), wr)
    b.free()
    t.free()


def test_probe_of_keys_a_topk_overwrites(ctx):
    k = 4096
    keys = datagen.splitmix64(5, 400_000).view(np.int64)
    wk, _ = oracle.topk(keys, k, olap.DESC)
    t = ctx.join_build(torch.from_numpy(wk[::2].copy()).cuda())
    dk = torch.from_numpy(keys).cuda()
    mid = torch.zeros(k, dtype=torch.int64, device="cuda")       # Top-K results, probed by the next run
    pairs = torch.empty((k, 2), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    item, _held = _top(dk, k, olap.DESC, mid)
    b = ctx.batch([item, olap.probe_item(t, mid, pairs, k, cnt)])
    for run in range(3):
        b.run()
        ctx.sync()
        assert int(cnt.item()) == (0 if run == 0 else k // 2)
        np.testing.assert_array_equal(mid.cpu().numpy(), wk)
    b.free()
    t.free()
