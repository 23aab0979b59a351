"""GPU parity of blocking calls whose kernels write results, status and pair
counts into host memory themselves, against the CPU oracle: pageable and
page-locked outputs on both sides of the row limit (4096), unaligned buffers
(which take the copy), bytes next to the outputs, and counts over repeated
probes, overflows and empty ones on one context."""
import ctypes

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


@pytest.mark.parametrize("n", [5000, 100_000, 600_000, 3_000_000])
@pytest.mark.parametrize("where", ["pageable", "pinned"])
def test_results(ctx, n, where):
    keys = datagen.topk_keys(n, "dup1024", "f32", seed=n)
    dk = torch.from_numpy(keys).cuda()
    for k in (1, 4095, 4096, 4097):
        ok, orow = torch.zeros(k + 2, dtype=torch.float32), torch.zeros(k + 2, dtype=torch.int32)
        if where == "pinned":
            ok, orow = ok.pin_memory(), orow.pin_memory()
        else:
            ok, orow = ok.numpy(), orow.numpy()
        ctx.topk(dk, k, olap.ASC, out_keys=ok[1:k + 1], out_rowids=orow[1:k + 1])
        wk, wr = oracle.topk(keys, k, olap.ASC)
        ok, orow = np.asarray(ok), np.asarray(orow)
        np.testing.assert_array_equal(orow[1:k + 1].view(np.uint32), wr)
        np.testing.assert_array_equal(ok[1:k + 1].view(np.uint32), wk.view(np.uint32))
        assert ok[0] == ok[-1] == 0 and orow[0] == orow[-1] == 0


@pytest.mark.parametrize("shift", [1, 2, 4])
def test_unaligned_outputs(ctx, shift):
    """Outputs at any byte address, through the C call."""
    keys = datagen.topk_keys(200_000, "uniform", "i64", seed=3)
    dk = torch.from_numpy(keys).cuda()
    raw_k, raw_r = np.zeros(100 * 8 + 16, dtype=np.uint8), np.zeros(100 * 4 + 16, dtype=np.uint8)
    got = ctypes.c_uint64()
    st = ctx.lib.olap_topk(ctx.h, dk.data_ptr(), olap.KEY_I64, None, olap.MEM_DEVICE, keys.shape[0], 100, olap.DESC,
                           raw_k.ctypes.data + shift, raw_r.ctypes.data + shift, olap.MEM_HOST, ctypes.byref(got))
    assert st == olap.OK and got.value == 100
    wk, wr = oracle.topk(keys, 100, olap.DESC)
    np.testing.assert_array_equal(raw_k[shift:shift + 800].view(np.uint8), wk.view(np.uint8))
    np.testing.assert_array_equal(raw_r[shift:shift + 400].view(np.uint8), wr.view(np.uint8))


def test_pair_results(ctx):
    c0 = (datagen.splitmix64(1, 500_000) % np.uint64(9)).astype(np.int32)
    c1 = datagen.splitmix64(2, 500_000).astype(np.int32)
    for k in (10, 4096, 4097):
        g = ctx.topk_pair(torch.from_numpy(c0).cuda(), olap.ASC, torch.from_numpy(c1).cuda(), olap.DESC, k)
        for a, b in zip(g, oracle.topk_pair(c0, olap.ASC, c1, olap.DESC, k)):
            np.testing.assert_array_equal(a, b)


def test_counts(ctx):
    """The context's count and row counter return to zero after every probe."""
    b = datagen.join_build(50_000, "mult14", seed=4)
    p = datagen.join_probe(70_001, b, 0.6, "uniform", seed=4)
    need = p.expected_pairs(b)
    t = ctx.join_build(torch.from_numpy(b.keys).cuda())
    dk = torch.from_numpy(p.keys).cuda()
    out = torch.empty((need, 2), dtype=torch.int32, device="cuda")
    cnt = torch.full((1,), 77, dtype=torch.int64, device="cuda")
    for _ in range(3):
        assert ctx.join_probe(t, dk, out=out).shape[0] == need
        with pytest.raises(olap.OlapError, match=f"need {need} pairs"):
            ctx.join_probe(t, dk, out=out, capacity=need - 1)
        assert ctx.join_probe(t, dk[:0], out=out).shape[0] == 0
        ctx.join_probe_async(t, dk, out, need, cnt)
        ctx.sync()
        assert int(cnt.item()) == need
        assert ctx.join_probe(t, p.keys[:1000]).shape[0] == oracle.join(b.keys, p.keys[:1000]).shape[0]
    t.free()
