"""GPU parity of the split and finish of a larger K (above 8192 survivors)
against the CPU oracle: selected rows in one dense run (a warp's stage fills
and empties) or spread thin, every row selected, row counts that leave warps
and steps ragged, bins around the sizes that one or two threads an entry (256,
512) and one CTA (2048) rank, and tied keys around the most that splitters
take (2^18 below the K-th entry's bin)."""
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


def _check(ctx, keys, k, order, rowids=None):
    dr = None if rowids is None else torch.from_numpy(rowids.view(np.int32)).cuda()
    gk, gr = ctx.topk(torch.from_numpy(keys).cuda(), k, order, rowids=dr)
    wk, wr = oracle.topk(keys, k, order, rowids)
    np.testing.assert_array_equal(gr, wr)
    np.testing.assert_array_equal(gk.view(np.uint8), wk.view(np.uint8))


@pytest.mark.parametrize("n", [12_301, 40_000, 622_595, 1_300_001])
@pytest.mark.parametrize("kt", [np.int64, np.float32])
def test_dense_and_sparse(ctx, n, kt):
    asc = np.arange(n).astype(kt)
    mixed = asc[np.random.default_rng(n).permutation(n)]
    rowids = np.random.default_rng(n + 1).permutation(n).astype(np.uint32)
    for k in (8400, min(n // 2, 9000 + n // 40), n - 1, n):
        for keys in (asc, mixed):
            _check(ctx, keys, k, olap.ASC)
        _check(ctx, asc, k, olap.DESC, rowids)


@pytest.mark.parametrize("m", [255, 256, 257, 511, 512, 513, 2047, 2048, 2049])
def test_bin_sizes(ctx, m):
    n = 60_000
    keys = (np.arange(n, dtype=np.int64) // m) * (1 << 42) + np.arange(n, dtype=np.int64) % m
    keys[7] = 1 << 62
    keys = keys[np.random.default_rng(m).permutation(n)]
    for k in (9000, 40_000, n):
        _check(ctx, keys, k, olap.ASC)


@pytest.mark.parametrize("k", [(1 << 18) - 5000, (1 << 18) - 1, 1 << 18, (1 << 18) + 1, (1 << 18) + 5000])
def test_ties_around_the_splitters_limit(ctx, k):
    keys = (datagen.splitmix64(8, 700_001) % np.uint64(11)).astype(np.int64) << 50
    _check(ctx, keys, k, olap.DESC)
    _check(ctx, keys, k, olap.ASC, (datagen.splitmix64(9, keys.shape[0]) % np.uint64(50_000)).astype(np.uint32))


@pytest.mark.parametrize("m", [1023, 1024, 1025])
def test_bin_sizes_past_the_splitters_limit(ctx, m):
    """With more entries than splitters take, bins end at 1024."""
    n = 300_000
    keys = (np.arange(n, dtype=np.int64) // m) * (1 << 42) + np.arange(n, dtype=np.int64) % m
    keys[7] = 1 << 62
    keys = keys[np.random.default_rng(m).permutation(n)]
    for k in (270_000, n):
        _check(ctx, keys, k, olap.ASC)
