"""A context's memory budget caps its device scratch and tables together: a
large build's partition scratch is checked beside the table that is being
built, is gone after the build, and without room for it the rows go to their
blocks one by one (fewer launches), with the oracle's pairs either way."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (1 << 22) + 5
TABLE = (1 << 23) * 32 + 256 + (1 << 19) * 32    # buckets, control block and filter of N rows
SCRATCH = N * 12
MIB = 1 << 20
GRANULE = 2 * MIB                                # in which the device hands out memory


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@pytest.fixture(scope="module")
def sides():
    b = datagen.join_build(N, "unique", seed=6)
    p = datagen.join_probe(100_003, b, 0.5, "uniform", seed=6)
    return torch.from_numpy(b.keys).cuda(), torch.from_numpy(p.keys).cuda(), oracle.join(b.keys, p.keys)


def _check(ctx, table, sides):
    out = torch.empty((sides[2].shape[0], 2), dtype=torch.int32, device="cuda")
    got = ctx.join_probe(table, sides[1], out=out).cpu().numpy().view(np.uint32).astype(np.uint64)
    np.testing.assert_array_equal(np.sort((got[:, 0] << np.uint64(32)) | got[:, 1]), sides[2])


@pytest.mark.parametrize("spare,launches", [(2 * MIB, 2), (SCRATCH - MIB, 2), (SCRATCH + 2 * MIB, 4)])
def test_build_scratch(sides, spare, launches):
    olap.device_trim(0)
    with olap.Context(0, mem_budget_bytes=TABLE + spare) as ctx:
        torch.cuda.empty_cache()
        free, before = _free(), ctx.launches()
        t = ctx.join_build(sides[0])
        assert ctx.launches() - before == launches
        assert free - _free() == -(-TABLE // GRANULE) * GRANULE      # the table alone stays
        _check(ctx, t, sides)
        t.free()
        t = ctx.join_build(sides[0])                     # and the budget is whole again
        assert ctx.launches() - before >= 2 * launches
        with pytest.raises(olap.OlapError) as ei:
            ctx.join_build(sides[0])
        assert ei.value.status == olap.E_NOMEM
        t.free()


def test_scratch_is_kept_and_returned_without_a_budget(sides):
    with olap.Context(0) as ctx:
        olap.device_trim(0)
        for _ in range(2):
            before = ctx.launches()
            t = ctx.join_build(sides[0])
            assert ctx.launches() - before == 4
            _check(ctx, t, sides)
            t.free()
        assert TABLE + SCRATCH <= olap.device_trim(0) < TABLE + SCRATCH + 4 * MIB


def test_probe_and_row_scratch_count():
    """What a partitioned probe and a full-row Top-K hold on to is part of the
    cap that later calls are checked against."""
    keys = torch.randint(-(1 << 62), 1 << 62, (1 << 20,), device="cuda")
    table = (1 << 20) * 64                               # bytes of its table, at most
    out = torch.empty((1 << 20, 2), dtype=torch.int32, device="cuda")
    rows = torch.randint(0, 255, (1 << 20, 16), dtype=torch.uint8, device="cuda")
    for use in ("probe", "rows"):
        with olap.Context(0, mem_budget_bytes=2 * table + 8 * MIB, join_partitions=16) as ctx:
            t = ctx.join_build(keys)
            ctx.join_build(keys).free()                  # room for a second one
            if use == "probe":
                ctx.join_probe(t, keys, out=out)         # 12 MiB of partitioned rows
            else:
                ctx.topk_rows(rows, 16, 0, olap.KEY_I64, 100)    # 8 MiB of keys, and the selection's scratch
            with pytest.raises(olap.OlapError) as ei:
                ctx.join_build(keys)
            assert ei.value.status == olap.E_NOMEM
            t.free()
            ctx.join_build(keys).free()                  # one still fits
