"""GPU parity of the larger-K finish (K above 8192: bins of the spanned
interval, else gaps between sorted splitters, else a merge sort) against the
CPU oracle, on keys that defeat equal bins: a few heavily tied values, ties of
whole (key, row-id) entries, one far outlier, and bins around the sizes one
warp (32, 128) and one CTA (4096) rank."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 2_200_003


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
    np.testing.assert_array_equal(gk, wk)


@pytest.mark.parametrize("kt", [np.int64, np.int32])
@pytest.mark.parametrize("values", [2, 3, 40])
@pytest.mark.parametrize("k", [8193, 100_000, 2_000_000])
def test_tied_values(ctx, kt, values, k):
    vals = datagen.splitmix64(3, values).view(np.int64)
    keys = (vals if kt is np.int64 else (vals >> 33).astype(np.int32))[(datagen.splitmix64(4, N) % np.uint64(values)).astype(np.int64)]
    _check(ctx, keys, k, olap.DESC)
    _check(ctx, keys, k, olap.ASC)


@pytest.mark.parametrize("k", [50_000, 400_000])
def test_identical_entries(ctx, k):
    """Explicit row-ids with few values: thousands of equal (key, row-id)."""
    keys = (datagen.splitmix64(5, N) % np.uint64(3)).astype(np.int64)
    rowids = (datagen.splitmix64(6, N) % np.uint64(7)).astype(np.uint32)
    _check(ctx, keys, k, olap.DESC, rowids)


@pytest.mark.parametrize("m", [31, 32, 33, 127, 128, 129, 4096, 4097])
def test_bin_sizes(ctx, m):
    """Groups of m keys close together, far from the next group, and an
    outlier that stretches the interval."""
    n = 20_000
    g = np.arange(n, dtype=np.int64) // m
    keys = g * (1 << 40) + (np.arange(n, dtype=np.int64) % m)
    keys[7] = 1 << 62
    keys = keys[np.random.default_rng(m).permutation(n)]
    for k in (8200, 15_000, n):
        _check(ctx, keys, k, olap.DESC)
