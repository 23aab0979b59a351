"""GPU parity of the partition passes of a probe against the CPU oracle: row
counts around a tile and a wave of tiles, one, two and eight partitions a lane,
all rows in one partition, and calls in a row on one context (the partitions'
counts are left at zero for the next one)."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILE = 320 * 7


def packed(pairs):
    p = np.asarray(pairs, dtype=np.uint64)
    return np.sort(p[:, 0] << np.uint64(32) | p[:, 1])


@pytest.fixture(scope="module")
def ctxs():
    cs = {p: olap.Context(0, join_partitions=p) for p in (2, 32, 64, 128, 256)}
    yield cs
    for c in cs.values():
        c.close()


@pytest.mark.parametrize("parts", [2, 32, 64, 128, 256])
@pytest.mark.parametrize("n", [1, 31, TILE - 1, TILE, TILE + 1, 3 * TILE + 17, 608 * TILE + 5])
def test_sizes(ctxs, parts, n):
    c = ctxs[parts]
    b = datagen.join_build(20_000, "mult14", seed=parts)
    t = c.join_build(torch.from_numpy(b.keys).cuda())
    p = datagen.join_probe(n, b, 0.5, "uniform", seed=n)
    rid = np.random.default_rng(n).permutation(n).astype(np.uint32)
    want = oracle.join(b.keys, p.keys)
    want_rid = oracle.join(b.keys, p.keys, None, rid)
    out = torch.empty((want.shape[0] + 1, 2), dtype=torch.int32, device="cuda")
    dk, dr = torch.from_numpy(p.keys).cuda(), torch.from_numpy(rid.view(np.int32)).cuda()
    for rows, w in ((None, want), (dr, want_rid), (None, want)):
        got = c.join_probe(t, dk, rowids=rows, out=out)
        assert c.join_probe_info()["parts"] == parts
        np.testing.assert_array_equal(packed(got.cpu().numpy().view(np.uint32)), w)
    t.free()


@pytest.mark.parametrize("parts", [2, 32, 64, 256])
def test_one_partition(ctxs, parts):
    """Every row has the same key, or one of two."""
    c = ctxs[parts]
    bk = datagen.splitmix64(3, 5000).view(np.int64)
    t = c.join_build(torch.from_numpy(bk).cuda())
    for n in (TILE, 50_001):
        for keys in (np.full(n, bk[17]), np.where(np.arange(n) % 3 == 0, bk[4], bk[4000])):
            keys = np.ascontiguousarray(keys)
            out = torch.empty((n, 2), dtype=torch.int32, device="cuda")
            got = c.join_probe(t, torch.from_numpy(keys).cuda(), out=out)
            np.testing.assert_array_equal(packed(got.cpu().numpy().view(np.uint32)), oracle.join(bk, keys))
    t.free()


@pytest.mark.parametrize("hit", [0.02, 0.5])
def test_pre_probe_leaves_few_rows(hit):
    """Rows enough to partition, but the pre-probe leaves fewer (0.02) or still
    enough of them (0.5; a quarter of 2^23 buckets is 2.1 * 10^6 rows)."""
    c = olap.Context(0)
    b = datagen.join_build(1 << 22, "unique", seed=8)
    t = c.join_build(torch.from_numpy(b.keys).cuda())
    n = 5_000_011
    assert c.join_probe_partitions(t, n) > 1
    p = datagen.join_probe(n, b, hit, "uniform", seed=8)
    want = oracle.join(b.keys, p.keys)
    out = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
    for _ in range(2):
        got = c.join_probe(t, torch.from_numpy(p.keys).cuda(), out=out)
        info = c.join_probe_info()
        assert info["prefiltered"] and (info["parts"] == 1) == (hit < 0.1)
        np.testing.assert_array_equal(packed(got.cpu().numpy().view(np.uint32)), want)
    t.free()
    c.close()


def test_large_build_between_replays_of_a_captured_probe(ctxs):
    """A large build orders its rows in scratch of its own: the scratch that a
    captured probe uses neither moves nor changes."""
    c = ctxs[32]
    b = datagen.join_build(20_000, "unique", seed=4)
    t = c.join_build(torch.from_numpy(b.keys).cuda())
    p = datagen.join_probe(100_003, b, 0.5, "uniform", seed=4)
    want = oracle.join(b.keys, p.keys)
    dk = torch.from_numpy(p.keys).cuda()
    out = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    c.join_probe_async(t, dk, out, want.shape[0], cnt)
    c.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.join_probe_async(t, dk, out, want.shape[0], cnt, stream=torch.cuda.current_stream().cuda_stream)
    keys = torch.randint(-(1 << 62), 1 << 62, ((1 << 23) + 11,), device="cuda")
    for _ in range(2):
        c.join_build(keys).free()
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert int(cnt.item()) == want.shape[0]
        np.testing.assert_array_equal(packed(out.cpu().numpy().view(np.uint32)), want)
    t.free()
