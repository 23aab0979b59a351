"""GPU parity of the block-wise join build (rows appended to blocks of 1024
buckets, each block built in one CTA's shared memory, chains wrapping within
it) against the CPU oracle: tables of one bucket up to several blocks and
tiles, partitioned builds, full blocks (high load factors), copies that crowd
a block so that the general build takes over, and the Bloom filter of each."""
import numpy as np
import pytest

import oracle
from paper_2601_19911_gb300 import datagen, olap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _packed(pairs):
    p = np.asarray(pairs, dtype=np.uint32).reshape(-1, 2).astype(np.uint64)
    return np.sort((p[:, 0] << np.uint64(32)) | p[:, 1])


def _check(ctx, bk, pk, load=0.0, br=None):
    want = oracle.join(bk, pk, br)
    t = ctx.join_build(torch.from_numpy(bk).cuda(), None if br is None else torch.from_numpy(br.view(np.int32)).cuda(),
                       load)
    out = torch.empty((max(1, want.shape[0]), 2), dtype=torch.int32, device="cuda")
    got = ctx.join_probe(t, torch.from_numpy(pk).cuda(), out=out).cpu().numpy().view(np.uint32)
    np.testing.assert_array_equal(_packed(got), want)
    t.free()


def _sides(n, seed, copies=1, key=None):
    distinct = datagen.splitmix64(seed, max(1, n // copies)).view(np.int64)
    bk = np.repeat(distinct, copies)[:n] if n else np.zeros(0, dtype=np.int64)
    if key is not None:
        bk[: n // 2] = key
    rng = np.random.default_rng(seed)
    bk = bk[rng.permutation(bk.shape[0])]
    pool = np.concatenate([bk, datagen.splitmix64(seed + 1, 2000).view(np.int64), np.array([-1], dtype=np.int64)])
    return np.ascontiguousarray(bk), np.ascontiguousarray(pool[rng.integers(0, pool.shape[0], 3000)])


@pytest.mark.parametrize("pre", [olap.PREFILTER_OFF, olap.PREFILTER_ON])
@pytest.mark.parametrize("load", [0.05, 0.5, 0.9])
def test_sizes(pre, load):
    with olap.Context(0, join_prefilter=pre) as ctx:
        for n in (0, 1, 2, 3, 7, 511, 512, 513, 921, 922, 1024, 1844, 4095, 4097, 30_011):
            bk, pk = _sides(n, 20 + n)
            br = (datagen.splitmix64(n, n) >> np.uint64(33)).astype(np.uint32) if n else None
            _check(ctx, bk, pk, load, br)


@pytest.mark.parametrize("pre", [olap.PREFILTER_OFF, olap.PREFILTER_ON])
@pytest.mark.parametrize("copies", [2, 5, 300])
def test_copies_within_blocks(pre, copies):
    with olap.Context(0, join_prefilter=pre) as ctx:
        _check(ctx, *_sides(20_000, 7, copies), 0.7)


@pytest.mark.parametrize("key", [5, -1])
@pytest.mark.parametrize("n", [4090, 4094, 60_000])
def test_crowded_blocks(key, n):
    """Half the rows carry one key: its block overflows (or, for the empty
    marker, none does, and the rows go to the side list)."""
    with olap.Context(0, join_prefilter=olap.PREFILTER_ON) as ctx:
        bk, pk = _sides(n, 11, key=key)
        _check(ctx, bk, pk[:40], 0.9)


@pytest.mark.parametrize("load,mult", [(0.0, "unique"), (0.9, "mult14")])
def test_partitioned_build(load, mult):
    """More blocks than a tile counts: ordered by the partition passes first."""
    b = datagen.join_build((1 << 23) + 11, mult, seed=5)
    p = datagen.join_probe(300_007, b, 0.6, "uniform", seed=5)
    with olap.Context(0) as ctx:
        _check(ctx, b.keys, p.keys, load)


def test_build_without_scratch_for_partitions():
    """A budget that holds the table but not the partition scratch: the rows go
    to their blocks one by one."""
    b = datagen.join_build((1 << 22) + 5, "unique", seed=6)
    p = datagen.join_probe(100_003, b, 0.5, "uniform", seed=6)
    table = (1 << 23) * 32 + (1 << 19) * 32
    with olap.Context(0, mem_budget_bytes=table + (30 << 20)) as ctx:
        _check(ctx, b.keys, p.keys)
