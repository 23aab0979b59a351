"""GPU parity of the Top-K streaming pass (32-byte loads, one comparison per
key in the key's own bit domain, remainder split evenly over the CTAs, a first
refine pass binned over the sampled interval) against the CPU oracle, where
those can go wrong: every alignment of the first key, rounds of the grid that
end just below or above a whole one, thresholds of either sign and order, ties
at the threshold, keys far below the sampled interval."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N0 = (1 << 21) + 1                                   # smallest sampled size
ROUND = 304 * 1024                                   # 32-byte vectors per round of the default grid


@pytest.fixture(scope="module")
def ctx():
    c = olap.Context(0)
    yield c
    c.close()


def _u(a):
    return a.view(np.uint64 if a.dtype.itemsize == 8 else np.uint32)


def _check(ctx, keys, k, order, offset=0, rowids=None):
    base = torch.from_numpy(np.concatenate([keys[:offset], keys])).cuda()
    dk = base[offset:]
    dr = None if rowids is None else torch.from_numpy(rowids.view(np.int32)).cuda()
    gk, gr = ctx.topk(dk, k, order, rowids=dr)
    wk, wr = oracle.topk(keys, k, order, rowids)
    np.testing.assert_array_equal(gr, wr)
    np.testing.assert_array_equal(_u(gk), _u(wk))


@pytest.mark.parametrize("kt", ["i64", "f32"])
@pytest.mark.parametrize("offset", range(8))
def test_alignment(ctx, kt, offset):
    _check(ctx, datagen.topk_keys(N0 + offset, "uniform", kt, seed=offset), 300, olap.DESC, offset)


@pytest.mark.parametrize("kt,vec", [("i64", 4), ("f32", 8)])
@pytest.mark.parametrize("extra", [-1, 0, 1, 304 * 32 - 1, 304 * 32 + 1])
def test_rounds(ctx, kt, vec, extra):
    n = (2 * ROUND + extra) * vec
    _check(ctx, datagen.topk_keys(n, "uniform", kt, seed=5), 1000, olap.ASC)


@pytest.mark.parametrize("kt", ["i64", "u64", "f64", "i32", "u32", "f32"])
@pytest.mark.parametrize("order", [olap.ASC, olap.DESC])
@pytest.mark.parametrize("sign", [-1, 1])
def test_thresholds(ctx, kt, order, sign):
    """All keys on one side of zero, clustered, with some far outside the
    interval the sample sees and many ties."""
    dt = {"i64": np.int64, "u64": np.uint64, "f64": np.float64, "i32": np.int32, "u32": np.uint32,
          "f32": np.float32}[kt]
    rng = np.random.default_rng(3)
    v = rng.integers(1000, 3000, N0).astype(np.float64)
    v[rng.integers(0, N0, 50)] = 5
    v[rng.integers(0, N0, 50)] = 100_000
    keys = (v * (sign if kt[0] != "u" else 1)).astype(dt)
    for k in (1, 40, 2000):
        _check(ctx, keys, k, order)


@pytest.mark.parametrize("off1", [0, 4, 1])           # co-aligned to 32 and to 16 bytes, and not at all
@pytest.mark.parametrize("orders", [(olap.DESC, olap.ASC), (olap.ASC, olap.DESC)])
def test_pair_alignment_and_ties(ctx, off1, orders):
    n = N0 + 5
    c0 = (datagen.splitmix64(1, n) % np.uint64(3)).astype(np.int32)
    c1 = (datagen.splitmix64(2, n) % np.uint64(50)).astype(np.int32)
    d0 = torch.from_numpy(c0).cuda()
    d1 = torch.from_numpy(np.concatenate([c1[:off1], c1])).cuda()[off1:]
    for k in (10, 3000):
        g = ctx.topk_pair(d0, orders[0], d1, orders[1], k)
        w = oracle.topk_pair(c0, orders[0], c1, orders[1], k)
        for a, b in zip(g, w):
            np.testing.assert_array_equal(a, b)
