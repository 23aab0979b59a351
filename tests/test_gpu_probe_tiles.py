"""GPU parity of the tiled probe (tiles of 128 rows per warp, probes walking
on past their home bucket compacted 32 at a time, 640 pairs staged per warp)
at the sizes where tiles, chunks and stages end, against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EDGES = [1, 31, 32, 33, 127, 128, 129, 511, 512, 513, 16383, 16385]


def packed(pairs):
    p = np.asarray(pairs, dtype=np.uint32).reshape(-1, 2).astype(np.uint64)
    return np.sort((p[:, 0] << np.uint64(32)) | p[:, 1])


@pytest.fixture(scope="module")
def sides():
    """A crowded table (load 0.9): every third key in 1 to 40 copies, and
    empty-marker keys (-1) on both sides."""
    rng = np.random.default_rng(8)
    distinct = datagen.splitmix64(8, 1200).view(np.int64)
    reps = np.where(np.arange(1200) % 3 == 0, rng.integers(1, 41, 1200), 1)
    bk = np.concatenate([np.repeat(distinct, reps), np.full(70, -1, dtype=np.int64)])
    bk = bk[rng.permutation(bk.shape[0])]
    pk = np.concatenate([bk, datagen.splitmix64(9, 5000).view(np.int64)])
    pk = pk[rng.integers(0, pk.shape[0], max(EDGES))]
    br = (datagen.splitmix64(1, bk.shape[0]) >> np.uint64(33)).astype(np.uint32)
    pr = (datagen.splitmix64(2, pk.shape[0]) >> np.uint64(33)).astype(np.uint32)
    return bk, pk, br, pr


@pytest.mark.parametrize("n", EDGES)
@pytest.mark.parametrize("rowids", [False, True])
def test_probe_edges(sides, n, rowids):
    bk, pk, br, pr = sides
    p, r = np.ascontiguousarray(pk[:n]), np.ascontiguousarray(pr[:n]) if rowids else None
    want = oracle.join(bk, p, br, r)
    with olap.Context(0) as ctx:
        t = ctx.join_build(torch.from_numpy(bk).cuda(), torch.from_numpy(br.view(np.int32)).cuda(), 0.9)
        dk = torch.from_numpy(p).cuda()
        dr = None if r is None else torch.from_numpy(r.view(np.int32)).cuda()
        out = torch.full((want.shape[0] + 1, 2), 7, dtype=torch.int32, device="cuda")
        got = ctx.join_probe(t, dk, dr, out=out)
        np.testing.assert_array_equal(packed(got.cpu().numpy().view(np.uint32)), want)
        assert out[-1].tolist() == [7, 7]                  # nothing past the pairs
        # the same rows as one batch item, cut into chunks
        cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
        bout = torch.empty((max(1, want.shape[0]), 2), dtype=torch.int32, device="cuda")
        b = ctx.batch([olap.probe_item(t, dk, bout, want.shape[0], cnt, d_rowids=dr)])
        b.run()
        ctx.sync()
        assert int(cnt.item()) == want.shape[0]
        np.testing.assert_array_equal(packed(bout.cpu().numpy().view(np.uint32)[: want.shape[0]]), want)
        b.free()
        # a capacity in the middle of a flush: exact count, nothing written past it
        cap = want.shape[0] // 2
        small = torch.full((cap + 64, 2), 7, dtype=torch.int32, device="cuda")
        if cap:
            with pytest.raises(olap.OlapError, match=f"need {want.shape[0]} pairs"):
                ctx.join_probe(t, dk, dr, out=small, capacity=cap)
            assert bool((small[cap:] == 7).all())
        t.free()
