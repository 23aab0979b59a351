"""GPU parity of Top-K over columns in host memory that the streaming pass reads
and copies itself, against the CPU oracle: page-locked and pageable columns,
offsets from a 32-byte boundary, ragged ends, row ids, key columns that are not
aligned to their type (refused), and columns where the sample misleads, so that the
selection reads the copy."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N0 = 1 << 21


@pytest.fixture(scope="module")
def ctx():
    c = olap.Context(0)
    yield c
    c.close()


def column(keys, where, shift):
    buf = torch.empty(keys.shape[0] + shift, dtype=torch.from_numpy(keys[:1]).dtype, pin_memory=where == "pinned")
    buf[shift:] = torch.from_numpy(keys)
    return buf[shift:] if where == "pinned" else buf.numpy()[shift:]


def check(ctx, keys, col, k, order, rowids=None):
    gk, gr = ctx.topk(col, k, order, rowids=rowids)
    wk, wr = oracle.topk(keys, k, order, rowids=None if rowids is None else np.asarray(rowids).view(np.uint32))
    np.testing.assert_array_equal(np.asarray(gr).view(np.uint32), wr)
    np.testing.assert_array_equal(np.ascontiguousarray(gk).view(np.uint8), wk.view(np.uint8))


@pytest.mark.parametrize("where", ["pageable", "pinned"])
@pytest.mark.parametrize("kind", ["f32", "i64", "f64"])
@pytest.mark.parametrize("n,shift", [(N0 + 1, 0), (N0 + 32, 1), (2_500_003, 2), (3_000_017, 3), (1 << 22, 5)])
def test_offsets(ctx, where, kind, n, shift):
    keys = datagen.topk_keys(n, "uniform", kind, seed=n + shift)
    col = column(keys, where, shift)
    check(ctx, keys, col, 100, olap.ASC)
    check(ctx, keys, col, n // 256, olap.DESC)


@pytest.mark.parametrize("where", ["pageable", "pinned"])
@pytest.mark.parametrize("kind", ["f32", "i64"])
@pytest.mark.parametrize("dist", ["equal", "blocks"])
def test_selection_from_the_copy(ctx, where, kind, dist):
    n = 3_000_001
    keys = np.zeros(n, dtype=np.float32 if kind == "f32" else np.int64)
    if dist == "blocks":                       # low keys between the sampled rows only
        keys[:] = datagen.splitmix64(5, n) % np.uint64(1 << 20)
        keys += 10
        step = n / 8192
        at = (np.arange(n) % step).astype(np.int64)
        keys[(at > 10) & (at < 100)] -= 9
        keys[0], keys[-1] = 0, 0
    for shift in (0, 3):
        col = column(keys, where, shift)
        check(ctx, keys, col, 1000, olap.ASC)
        check(ctx, keys, col, 10, olap.DESC)


@pytest.mark.parametrize("where", ["pageable", "pinned"])
def test_rowids(ctx, where):
    n = 2_200_007
    keys = datagen.topk_keys(n, "dup1024", "f64", seed=9)
    rid = np.random.default_rng(4).permutation(n).astype(np.uint32)
    r = column(rid.view(np.int32), where, 1)
    check(ctx, keys, column(keys, where, 1), 500, olap.ASC, r if where == "pinned" else r.view(np.uint32))


@pytest.mark.parametrize("shift", [1, 4])
def test_column_off_its_alignment(ctx, shift):
    """Refused, as on the other paths."""
    n, k = N0 + 9, 64
    keys = datagen.topk_keys(n, "uniform", "i64", seed=2)
    raw = np.zeros(n * 8 + 8, dtype=np.uint8)
    raw[shift:shift + n * 8] = keys.view(np.uint8)
    ok, orow, got = np.zeros(k, dtype=np.int64), np.zeros(k, dtype=np.uint32), ctypes.c_uint64()
    st = ctx.lib.olap_topk(ctx.h, raw.ctypes.data + shift, olap.KEY_I64, None, olap.MEM_HOST, n, k, olap.ASC,
                           ok.ctypes.data, orow.ctypes.data, olap.MEM_HOST, ctypes.byref(got))
    assert st == olap.E_INVALID and got.value == 0
