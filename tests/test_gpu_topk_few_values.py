"""GPU parity of the sampled Top-K on columns of few distinct values, where the
rows up to the sampled threshold would not fit the candidate buffer and the
streaming pass only counts them, against the CPU oracle: on both sides of the
sizes where the paths change, one and two columns, implicit and explicit
row-ids, a K-th row among the ties, below them and past what the sample says,
and samples that misjudge the column altogether."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SAMPLE = 8192


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


def _values(n, distinct, typ, seed):
    vals = datagen.splitmix64(seed, distinct)
    vals = {"i64": vals.view(np.int64), "f32": (vals.view(np.int64) / 1e12).astype(np.float32),
            "u32": (vals >> np.uint64(32)).astype(np.uint32)}[typ]
    return vals[(datagen.splitmix64(seed + 1, n) % np.uint64(distinct)).astype(np.int64)]


@pytest.mark.parametrize("typ", ["i64", "f32", "u32"])
@pytest.mark.parametrize("n", [(3 << 17) + 1, 600_011, 1 << 21, (1 << 21) + 1, 3_000_017])
def test_few_values(ctx, n, typ):
    for distinct in (1, 2, 12, 100):
        keys = _values(n, distinct, typ, n + distinct)
        for k in (1, 300, n // 256):
            _check(ctx, keys, k, olap.DESC)
            if distinct <= 12:
                assert ctx.topk_info()["path"] == 2
        # row-ids in no order, repeated, and up to the highest value
        for rid in (np.random.default_rng(n).permutation(n).astype(np.uint32),
                    (datagen.splitmix64(n, n) % np.uint64(5)).astype(np.uint32),
                    np.uint32(0xFFFFFFFF) - np.arange(n, dtype=np.uint32)):
            _check(ctx, keys, n // 300, olap.ASC, rid)


@pytest.mark.parametrize("n", [600_011, 3_000_017])
def test_row_ids_in_host_memory(ctx, n):
    keys = _values(n, 3, "i64", 5)
    rid = np.random.default_rng(n).permutation(n).astype(np.uint32)
    hk, hr = torch.from_numpy(keys).pin_memory(), torch.from_numpy(rid.view(np.int32)).pin_memory()
    gk, gr = ctx.topk(hk, 500, olap.DESC, rowids=hr)
    wk, wr = oracle.topk(keys, 500, olap.DESC, rid)
    np.testing.assert_array_equal(np.asarray(gr).view(np.uint32), wr)
    np.testing.assert_array_equal(np.asarray(gk), wk)


@pytest.mark.parametrize("n", [600_011, 3_000_017])
@pytest.mark.parametrize("better", [0, 5, 300, 301, 6000])
def test_rows_better_than_the_ties(ctx, n, better):
    """The threshold is the value most rows hold; `better` rows lie below it."""
    keys = np.full(n, 1000, dtype=np.int64)
    at = np.random.default_rng(better).permutation(n)[:better]
    keys[at] = np.arange(better) - 5_000_000
    keys[np.random.default_rng(7).permutation(n)[: n // 3]] = 2000
    for k in (1, 300, 2000):
        _check(ctx, keys, k, olap.ASC)


@pytest.mark.parametrize("n", [600_011, 3_000_017])
def test_misjudged_samples(ctx, n):
    """All sampled rows hold one value, and hardly any other row does."""
    j = np.arange(SAMPLE, dtype=np.int64)
    at = (j * n) // SAMPLE + (n // SAMPLE) // 2
    keys = datagen.splitmix64(3, n).view(np.int64) >> 2
    for v in (-(1 << 62), 0):                  # better than the others; in their middle
        keys[at] = v
        for k in (1, 2000, n // 256):
            _check(ctx, keys, k, olap.ASC)
            _check(ctx, keys, k, olap.DESC)


@pytest.mark.parametrize("n", [600_011, (1 << 21) + 1])
def test_pair(ctx, n):
    for d0, d1 in ((1, 1), (1, 2), (3, 5), (2, 1 << 30)):
        c0 = (datagen.splitmix64(1, n) % np.uint64(d0)).astype(np.int32)
        c1 = (datagen.splitmix64(2, n) % np.uint64(d1)).astype(np.int32)
        for k in (1, 1500):
            g = ctx.topk_pair(torch.from_numpy(c0).cuda(), olap.DESC, torch.from_numpy(c1).cuda(), olap.ASC, k)
            for a, b in zip(g, oracle.topk_pair(c0, olap.DESC, c1, olap.ASC, k)):
                np.testing.assert_array_equal(a, b)
