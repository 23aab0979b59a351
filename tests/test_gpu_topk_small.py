"""GPU parity of small Top-K queries against the CPU oracle: the kernel that
works in every CTA's own shared memory (n up to 12,288), the direct path above
it and the streaming pass inside the select kernel (n up to 2^21), at the sizes
where one takes over from the next, with ties, clusters and equal entries."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NS = [1, 2, 31, 33, 1023, 1025, 4095, 4097, 12_287, 12_288, 12_289, 393_215, 393_216, 393_217, (1 << 21) - 1, 1 << 21]


def _keys(n, dist, kt, seed):
    if dist in ("uniform", "ascending", "dup1024"):
        return datagen.topk_keys(n, dist, kt, seed=seed)
    rng = np.random.default_rng(seed)
    dt = {"i64": np.int64, "f32": np.float32, "f64": np.float64, "u32": np.uint32}[kt]
    if dist == "equal":
        return np.full(n, 3, dtype=dt)
    v = rng.integers(10_000, 10_003, n).astype(np.float64)         # three values, and outliers at both ends
    v[rng.integers(0, n, 2)] = 1
    v[rng.integers(0, n, 2)] = 1e9
    return v.astype(dt)


@pytest.fixture(scope="module")
def ctx():
    c = olap.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("kt", ["i64", "f32", "f64", "u32"])
@pytest.mark.parametrize("dist", ["uniform", "ascending", "dup1024", "equal", "cluster"])
def test_sizes(ctx, kt, dist):
    for j, n in enumerate(NS):
        keys = _keys(n, dist, kt, n)
        off = j % 5
        dk = torch.from_numpy(np.concatenate([keys[:1].repeat(off), keys])).cuda()[off:]
        for k in sorted({1, 10, 65, 1000, min(n, 4096), n}) if n < 20_000 else (1, 100, 1500):
            order = olap.DESC if (j + k) % 2 else olap.ASC
            gk, gr = ctx.topk(dk, k, order)
            wk, wr = oracle.topk(keys, k, order)
            np.testing.assert_array_equal(gr, wr)
            np.testing.assert_array_equal(gk.view(np.uint8), wk.view(np.uint8))


@pytest.mark.parametrize("n", [100, 5000, 12_288])
@pytest.mark.parametrize("ids", [1, 3])
def test_identical_entries(ctx, n, ids):
    """Equal keys with explicit row-ids of one or three values."""
    keys = np.full(n, 9, dtype=np.int64)
    rid = (datagen.splitmix64(2, n) % np.uint64(ids)).astype(np.uint32)
    dr = torch.from_numpy(rid.view(np.int32)).cuda()
    for k in (1, 64, n // 2, n):
        gk, gr = ctx.topk(torch.from_numpy(keys).cuda(), k, olap.DESC, rowids=dr)
        np.testing.assert_array_equal(gr, oracle.topk(keys, k, olap.DESC, rid)[1])


@pytest.mark.parametrize("n", [7, 3000, 12_288, 400_001])
def test_pairs_and_noalloc(ctx, n):
    c0 = (datagen.splitmix64(1, n) % np.uint64(4)).astype(np.int32)
    c1 = datagen.splitmix64(2, n).astype(np.int32)
    for k in (1, 50, min(n, 900)):
        g = ctx.topk_pair(torch.from_numpy(c0).cuda(), olap.DESC, torch.from_numpy(c1).cuda(), olap.ASC, k)
        for a, b in zip(g, oracle.topk_pair(c0, olap.DESC, c1, olap.ASC, k)):
            np.testing.assert_array_equal(a, b)
        ok = torch.empty(min(n, k), dtype=torch.int32, device="cuda")
        orow = torch.empty_like(ok)
        st = torch.full((1,), -1, dtype=torch.int32, device="cuda")
        olap.topk_noalloc(torch.from_numpy(c1).cuda(), k, olap.ASC, ok, orow, dev_status=st)
        torch.cuda.synchronize()
        assert int(st.item()) == olap.OK
        np.testing.assert_array_equal(orow.cpu().numpy().view(np.uint32), oracle.topk(c1, k, olap.ASC)[1])
