"""GPU parity of the block-wise join build against the CPU oracle where many
copies of keys share a block (their runs of slots are long, pass the block's
last slot or fill the block but for one slot), in tables of one bucket to
several blocks, and a block that is just too full, which the general build
takes.  Reading the number of launches shows which build ran."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
M64 = (1 << 64) - 1


@pytest.fixture(scope="module")
def ctx():
    c = olap.Context(0, join_prefilter=olap.PREFILTER_ON)
    yield c
    c.close()


def _fmix64(keys):
    h = keys.astype(np.uint64).copy()
    for c in (0xff51afd7ed558ccd, 0xc4ceb9fe1a85ec53):
        h ^= h >> np.uint64(33)
        h *= np.uint64(c)
    return h ^ (h >> np.uint64(33))


def _check(ctx, bk, load=0.5, launches=None):
    rng = np.random.default_rng(bk.shape[0])
    bk = np.ascontiguousarray(bk[rng.permutation(bk.shape[0])])
    pk = np.concatenate([bk[:: max(1, bk.shape[0] // 37)], datagen.splitmix64(77, 500).view(np.int64)])
    want = oracle.join(bk, pk)
    before = ctx.launches()
    t = ctx.join_build(torch.from_numpy(bk).cuda(), None, load)
    if launches:
        assert ctx.launches() - before == launches
    out = torch.empty((max(1, want.shape[0]), 2), dtype=torch.int32, device="cuda")
    got = ctx.join_probe(t, torch.from_numpy(pk).cuda(), out=out).cpu().numpy().view(np.uint32).astype(np.uint64)
    np.testing.assert_array_equal(np.sort((got[:, 0] << np.uint64(32)) | got[:, 1]), want)
    t.free()


@pytest.mark.parametrize("copies", [2, 3, 17, 64, 500])
@pytest.mark.parametrize("load", [0.5, 0.9])
def test_every_key_repeats(ctx, copies, load):
    for n in (1, 2, 5, 30, 900, 1800, 20_000):
        _check(ctx, np.repeat(datagen.splitmix64(copies, max(1, n // copies)).view(np.int64), copies)[:n], load)


@pytest.mark.parametrize("n", [100_000, (1 << 22) + 5])
def test_one_heavy_key(ctx, n):
    """1100 copies fit their block (about 781 or 1024 other rows at most)."""
    bk = datagen.splitmix64(9, n).view(np.int64).copy()
    bk[:1000] = 5
    _check(ctx, bk, launches=4 if n > 1 << 22 else 2)


def _keys_of_block(block, blocks, count, homes=None):
    """Distinct keys whose home bucket is in `block` of `blocks` * 1024 buckets
    (within the block, in `homes`)."""
    out = []
    for s in range(1, 400):
        k = datagen.splitmix64(s, 1 << 16)
        b = _fmix64(k) & np.uint64(blocks * 1024 - 1)
        keep = (b >> np.uint64(10)) == np.uint64(block)
        if homes is not None:
            keep &= np.isin(b & np.uint64(1023), np.asarray(homes, dtype=np.uint64))
        out.append(k[keep])
        if sum(map(len, out)) >= count:
            break
    return np.concatenate(out)[:count].view(np.int64)


@pytest.mark.parametrize("rows,launches", [(2046, 2), (2047, 2), (2048, 2 + 3)])
def test_full_block(ctx, rows, launches):
    """All rows of one block of four: one slot fewer, all but one, too many."""
    _check(ctx, _keys_of_block(2, 4, rows), 0.26, launches)


@pytest.mark.parametrize("homes", [[1023], [1020, 1021, 1022, 1023], [0, 1023], [511, 512]])
def test_runs_past_the_end(ctx, homes):
    """Home buckets at the block's end (their runs wrap) beside ones at its
    start, each key twice."""
    distinct = _keys_of_block(0, 2, 150, homes)
    other = _keys_of_block(0, 2, 600)
    _check(ctx, np.concatenate([np.repeat(distinct, 2), np.repeat(distinct[:40], 6), other]), 0.3)
