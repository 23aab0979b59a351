"""GPU parity of Top-K calls whose outputs lie over their inputs (results in the
place of the keys or row-ids they come from), against the CPU oracle, on both
sides of the one-launch limit (12,288 keys): blocking, enqueue-only and
allocation-free calls, one and two columns.  Such a call takes the path that
writes behind a grid barrier; one whose buffers only touch keeps the single
launch."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LOCAL_N = 12_288
TYPES = {"i64": torch.int64, "f32": torch.float32}


@pytest.fixture(scope="module")
def ctx():
    c = olap.Context(0)
    yield c
    c.close()


def _inputs(n, typ):
    keys = datagen.topk_keys(n, "dup1024", typ, seed=n)
    rid = np.random.default_rng(n).permutation(n).astype(np.uint32) * np.uint32(3)
    return keys, rid


def _same(got_k, got_r, want):
    np.testing.assert_array_equal(got_r.cpu().numpy().view(np.uint32), want[1])
    np.testing.assert_array_equal(got_k.cpu().numpy().view(np.uint8), want[0].view(np.uint8))


@pytest.mark.parametrize("typ", sorted(TYPES))
@pytest.mark.parametrize("n", [17, 3001, LOCAL_N, LOCAL_N + 1, 400_001])
def test_one_column(ctx, n, typ):
    keys, rid = _inputs(n, typ)
    for k in sorted({9, min(n, 1000) - 1, min(n, 1365)}):
        want = oracle.topk(keys, k, olap.DESC, rid)
        for shift in (0, n - k, (n - k) // 2):                # results at the start, the end and inside of the columns
            for call in ("block", "async", "noalloc"):
                dk = torch.from_numpy(keys).cuda()
                dr = torch.from_numpy(rid.view(np.int32)).cuda()
                ok, orow = dk[shift:shift + k], dr[shift:shift + k]
                before = ctx.launches()
                if call == "block":
                    ctx.topk(dk, k, olap.DESC, rowids=dr, out_keys=ok, out_rowids=orow)
                elif call == "async":
                    ctx.topk_async(dk, k, olap.DESC, ok, orow, d_rowids=dr)
                    ctx.sync()
                else:
                    olap.topk_noalloc(dk, k, olap.DESC, ok, orow, d_rowids=dr)
                    torch.cuda.synchronize()
                _same(ok, orow, want)
                if call != "noalloc":
                    assert ctx.launches() - before == 2


@pytest.mark.parametrize("n", [300, LOCAL_N, LOCAL_N + 1])
def test_each_buffer_alone(ctx, n):
    """One output over one input: keys over row-ids, row-ids over keys."""
    keys, rid = _inputs(n, "f32")
    k = 200
    want = oracle.topk(keys, k, olap.ASC, rid)
    for over in ("keys", "rowids", "keys over rowids", "rowids over keys"):
        dk, dr = torch.from_numpy(keys).cuda(), torch.from_numpy(rid.view(np.int32)).cuda()
        ok, orow = torch.empty(k, dtype=torch.float32, device="cuda"), torch.empty(k, dtype=torch.int32, device="cuda")
        if over == "keys":
            ok = dk[50:50 + k]
        elif over == "rowids":
            orow = dr[n - k:]
        elif over == "keys over rowids":
            ok = dr[:k].view(torch.float32)
        else:
            orow = dk[:k].view(torch.int32)
        before = ctx.launches()
        ctx.topk(dk, k, olap.ASC, rowids=dr, out_keys=ok, out_rowids=orow)
        _same(ok, orow, want)
        assert ctx.launches() - before == 2


@pytest.mark.parametrize("n", [300, LOCAL_N, LOCAL_N + 1])
def test_pair(ctx, n):
    c0 = (datagen.splitmix64(1, n) % np.uint64(5)).astype(np.int32)
    c1 = datagen.splitmix64(2, n).astype(np.int32)
    k = 250
    d0, d1 = torch.from_numpy(c0).cuda(), torch.from_numpy(c1).cuda()
    orow = torch.empty(k, dtype=torch.int32, device="cuda")
    before = ctx.launches()
    ctx.topk_pair(d0, olap.ASC, d1, olap.DESC, k, out_keys0=d0[:k], out_keys1=d1[n - k:], out_rowids=orow)
    assert ctx.launches() - before == 2
    for a, b in zip((d0[:k], d1[n - k:], orow), oracle.topk_pair(c0, olap.ASC, c1, olap.DESC, k)):
        np.testing.assert_array_equal(a.cpu().numpy().view(np.uint32), b.view(np.uint32))


def test_touching_buffers_keep_one_launch(ctx):
    n, k = 4000, 128
    keys, rid = _inputs(n, "i64")
    buf = torch.empty(n + 2 * k, dtype=torch.int64, device="cuda")
    dk = buf[k:k + n]
    dk.copy_(torch.from_numpy(keys))
    orow = buf[k + n:].view(torch.int32)[:k]
    before = ctx.launches()
    ctx.topk(dk, k, olap.DESC, out_keys=buf[:k], out_rowids=orow)
    assert ctx.launches() - before == 1
    _same(buf[:k], orow, oracle.topk(keys, k, olap.DESC))
