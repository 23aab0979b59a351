"""GPU parity of the batched Top-K's selection by bins against the CPU oracle:
item sizes around one CTA's sort (4096), the sample (16 K), the parts (2^16)
and the split threshold (2^17), with keys that fill the bins evenly, crowd one
of them (ties, an outlier) or fall below the sampled interval."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (31, 40), (4095, 10), (4096, 4096), (4097, 4096), (5000, 1), (16_000, 1000), (16_001, 1000),
          (65_535, 4095), (131_071, 100), (131_072, 100), (131_073, 4096), (400_003, 1000)]


def _keys(n, dist, kt, seed):
    if dist in ("uniform", "ascending", "dup1024"):
        return datagen.topk_keys(n, dist, kt, seed=seed)
    rng = np.random.default_rng(seed)
    dt = {"i64": np.int64, "f32": np.float32, "f64": np.float64, "u32": np.uint32}[kt]
    if dist == "equal":
        return np.full(n, 3, dtype=dt)
    if dist == "two":
        return rng.integers(1, 3, n).astype(dt)
    v = rng.integers(10_000, 20_000, n).astype(np.float64)         # clustered, with outliers at both ends
    v[rng.integers(0, n, 3)] = 1
    v[rng.integers(0, n, 3)] = 1e9
    return v.astype(dt)


@pytest.mark.parametrize("kt", ["i64", "f32", "f64", "u32"])
@pytest.mark.parametrize("dist", ["uniform", "ascending", "dup1024", "equal", "two", "cluster"])
def test_items(kt, dist):
    items, held = [], []
    for j, (n, k) in enumerate(SHAPES):
        keys = _keys(n, dist, kt, 50 + j)
        order = olap.DESC if j % 2 else olap.ASC
        rid = np.arange(n, dtype=np.uint32)[::-1].copy() if j % 3 == 0 else None
        off = j % 5                                              # keys at every alignment
        dk = torch.from_numpy(np.concatenate([keys[:1].repeat(off), keys])).cuda()[off:]
        dr = None if rid is None else torch.from_numpy(rid.view(np.int32)).cuda()
        c = min(n, k)
        ok = torch.empty(c, dtype=dk.dtype, device="cuda")
        orow = torch.empty(c, dtype=torch.int32, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
        items.append(olap.topk_item(dk, k, order, ok, orow, cnt, d_rowids=dr))
        held.append((keys, rid, k, order, dk, dr, ok, orow, cnt))
    with olap.Context(0) as ctx:
        bt = ctx.batch(items)
        bt.run()
        ctx.sync()
        assert bt.errors() == 0
        for keys, rid, k, order, _dk, _dr, ok, orow, cnt in held:
            wk, wr = oracle.topk(keys, k, order, rid)
            assert int(cnt.item()) == wr.shape[0]
            np.testing.assert_array_equal(orow.cpu().numpy().view(np.uint32), wr)
            np.testing.assert_array_equal(ok.cpu().numpy().view(np.uint8), wk.view(np.uint8))
        bt.free()
