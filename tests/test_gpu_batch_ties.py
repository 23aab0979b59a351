"""GPU parity of batched Top-K items of few distinct keys against the CPU
oracle: inputs and candidate lists whose bins hold too many entries to rank, so
that the kept bins are sorted (K from one to all of the input, kept bins of up
to 4096 entries and more), with row-ids in and out of order and repeated."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kt", ["i64", "f32"])
@pytest.mark.parametrize("rowids", ["index", "shuffled", "repeated"])
def test_few_values(kt, rowids):
    items, held = [], []
    for n in (2, 300, 511, 512, 1000, 2049, 4095, 4096, 4097, 20_000, 70_000, 200_000):
        for distinct in (2, 3, 12, 40, 100):
            vals = datagen.splitmix64(distinct, distinct).view(np.int64) >> 3
            keys = vals[(datagen.splitmix64(n + distinct, n) % np.uint64(distinct)).astype(np.int64)]
            keys = keys if kt == "i64" else (keys / 1e12).astype(np.float32)
            rid = {"index": None, "shuffled": np.random.default_rng(n).permutation(n).astype(np.uint32),
                   "repeated": (datagen.splitmix64(n, n) % np.uint64(7)).astype(np.uint32)}[rowids]
            for k in sorted({1, min(n, 600), min(n, 4096)}):
                dk = torch.from_numpy(keys).cuda()
                dr = None if rid is None else torch.from_numpy(rid.view(np.int32)).cuda()
                ok = torch.empty(k, dtype=dk.dtype, device="cuda")
                orow = torch.empty(k, dtype=torch.int32, device="cuda")
                cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
                order = olap.DESC if (n + k) % 2 else olap.ASC
                items.append(olap.topk_item(dk, k, order, ok, orow, cnt, d_rowids=dr))
                held.append((keys, rid, k, order, dk, dr, ok, orow, cnt))
    with olap.Context(0) as ctx:
        bt = ctx.batch(items)
        for _ in range(2):
            bt.run()
            ctx.sync()
            assert bt.errors() == 0
            for keys, rid, k, order, _dk, _dr, ok, orow, cnt in held:
                wk, wr = oracle.topk(keys, k, order, rid)
                assert int(cnt.item()) == k
                np.testing.assert_array_equal(orow.cpu().numpy().view(np.uint32), wr)
                np.testing.assert_array_equal(ok.cpu().numpy().view(np.uint8), wk.view(np.uint8))
                orow.zero_()
        bt.free()
