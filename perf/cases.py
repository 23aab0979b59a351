"""What a user of the library runs, as measurable cases.

Each case is one call (or one unit of work) through the public entry points of
``paper_2601_19911_gb300.olap``, over the sizes, key types, orders and kinds of
memory the configurations, tests and benchmark of this repository use:

* ``topk``: ORDER BY key LIMIT k over one column, by the blocking call with
  results in host memory (``mode`` "host"), the blocking call with results on
  the device ("block"), the enqueue-only call ("async") or the call that
  allocates nothing ("noalloc").
* ``pair``: ORDER BY c0, c1 LIMIT k over two 4-byte columns.
* ``probe``: a probe of a resident hash table, its pairs materialised as a
  column (the matching build row of every probe row, -1 without one).
* ``join``: a whole hash join: build, probe, materialise, free.
* ``batch``: one run of a captured batch of Top-K queries and probes.

The order of a join's pairs is unspecified, so a case returns what a query
does with them: the scattered column for a build with unique keys, the sorted
pairs for one with duplicates.
"""
import math

import numpy as np
import torch

from paper_2601_19911_gb300 import olap

DEV = "cuda"
KEYS = {"i64": torch.int64, "f64": torch.float64, "u64": torch.uint64, "i32": torch.int32, "f32": torch.float32,
        "u32": torch.uint32}
ORDERS = {"asc": olap.ASC, "desc": olap.DESC}
MAX_N = 1 << 28
MAX_PROBE = 1 << 25
MAX_BUILD = 1 << 24


def listed():
    return [
        # a small dashboard query over a filtered table: 10 k doubles, ten rows wanted, answer in host memory
        dict(name="topk_f64_10k", op="topk", type="f64", n=10_007, k=10, order="asc", dist="normal", rowids=False,
             where="device", mode="host"),
        # the single-query configuration: 2^20 int64 keys with row-ids, K = 100, answer in host memory
        dict(name="topk_i64_1m", op="topk", type="i64", n=1 << 20, k=100, order="desc", dist="uniform", rowids=True,
             where="device", mode="host"),
        # key-only offload end to end (the paper's N = 3 M doubles): keys cross the link, K rows come back
        dict(name="topk_f64_3m_pinned", op="topk", type="f64", n=3_000_000, k=100, order="desc", dist="normal",
             rowids=False, where="pinned", mode="host"),
        # an ordinary ragged column already on the device, part of a queued plan
        dict(name="topk_f32_20m", op="topk", type="f32", n=20_000_003, k=1000, order="desc", dist="normal",
             rowids=False, where="device", mode="async"),
        # the headline configuration: 2^28 int64 keys with row-ids, K = 1000
        dict(name="topk_i64_2p28", op="topk", type="i64", n=1 << 28, k=1000, order="desc", dist="uniform", rowids=True,
             where="device", mode="async"),
        # a large K over a column with many ties (an export of the first 100,000 rows)
        dict(name="topk_i32_100m_k1e5", op="topk", type="i32", n=100_000_001, k=100_000, order="asc", dist="dup1024",
             rowids=False, where="device", mode="async"),
        # a two-column ORDER BY: a low-cardinality column first
        dict(name="pair_2p26", op="pair", n=1 << 26, k=1000, order0="desc", order1="asc", rowids=False),
        # a small probe of a dimension table that stays in cache
        dict(name="probe_100k", op="probe", build=1 << 20, n=100_003, hit=0.5, dist="uniform", rowids=False),
        # the join configuration: 2^24 unique build keys, uniform probe keys, most of them hits
        dict(name="probe_30m_hit90", op="probe", build=1 << 24, n=30_000_001, hit=0.9, dist="uniform", rowids=False),
        # a selective join over a skewed fact column with row-ids of its own
        dict(name="probe_2p25_zipf_hit10", op="probe", build=1 << 24, n=1 << 25, hit=0.1, dist="zipf", rowids=True),
        # a whole join: the table is built for this query and dropped after it
        dict(name="join_4m_8m", op="join", build=4_000_037, n=8_000_009, hit=0.9, mult="unique"),
        # many small queries in one launch
        dict(name="batch_512_128", op="batch", topk=512, probe=128, build=1 << 20, sizes=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(["topk", "pair", "probe", "join", "batch"], [9, 2, 4, 2, 2])[0]
    if op == "topk":
        where = rng.choices(["device", "pinned", "pageable"], [7, 1, 1])[0]
        mode = rng.choice(["host", "block", "async", "noalloc"]) if where == "device" else "host"
        n = _log(rng, 1e3, MAX_N if where == "device" and mode != "noalloc" else 1 << 24)
        typ = rng.choice(sorted(KEYS))
        dist = rng.choice(["uniform", "dup1024", "ascending"] if typ[0] != "f" else ["normal", "dup1024", "ascending"])
        k = _log(rng, 1, min(n, 4096 if mode == "noalloc" else 100_000))
        return dict(op=op, type=typ, n=n, k=k, order=rng.choice(["asc", "desc"]), dist=dist,
                    rowids=rng.random() < 0.5, where=where, mode=mode)
    if op == "pair":
        n = _log(rng, 1e3, 1 << 27)
        return dict(op=op, n=n, k=_log(rng, 1, min(n, 10_000)), order0=rng.choice(["asc", "desc"]),
                    order1=rng.choice(["asc", "desc"]), rowids=rng.random() < 0.5)
    if op == "probe":
        return dict(op=op, build=_log(rng, 1e3, MAX_BUILD), n=_log(rng, 1e3, MAX_PROBE),
                    hit=rng.choice([0.1, 0.5, 0.9]), dist=rng.choice(["uniform", "zipf"]), rowids=rng.random() < 0.5)
    if op == "join":
        mult = rng.choice(["unique", "unique", "mult14"])
        cap = 1 << 23 if mult == "unique" else 1 << 20
        return dict(op=op, build=_log(rng, 1e3, cap), n=_log(rng, 1e3, cap), hit=rng.choice([0.1, 0.5, 0.9]), mult=mult)
    return dict(op=op, topk=_log(rng, 16, 512), probe=_log(rng, 4, 128), build=_log(rng, 1e4, 1 << 20),
                sizes=rng.randrange(1 << 20))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

_ctx = None


def _context():
    """The program's one context, made on first use."""
    global _ctx
    if _ctx is None:
        _ctx = olap.Context(0)
    return _ctx


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, n, typ):
    if typ in ("f32", "f64"):
        return torch.randn(n, dtype=KEYS[typ], device=DEV, generator=g) * 1000
    if typ in ("i64", "u64"):
        return torch.randint(-(1 << 63), (1 << 63) - 1, (n,), dtype=torch.int64, device=DEV, generator=g)
    return torch.randint(-(1 << 31), (1 << 31) - 1, (n,), dtype=torch.int32, device=DEV, generator=g)


def _column(g, n, typ, dist):
    """A key column; unsigned types as their signed bit patterns."""
    if dist in ("uniform", "normal"):
        return _uniform(g, n, typ)
    if dist == "dup1024":
        vals = _uniform(g, 1024, typ)
        return vals[torch.randint(0, 1024, (n,), device=DEV, generator=g)]
    # ascending, from a drawn start
    start = int(torch.randint(0, 1 << 20, (1,), device=DEV, generator=g).item())
    i = torch.arange(start, start + n, dtype=torch.int64, device=DEV)
    if typ in ("f32", "f64"):
        return (i - n // 2).to(KEYS[typ])
    return i * ((1 << 62) // (n + (1 << 20))) if typ in ("i64", "u64") else (i + n).to(torch.int32)


def _typed(t, typ):
    return t.view(KEYS[typ]) if typ in ("u64", "u32") else t


def _rowids(n):
    return torch.arange(n, dtype=torch.int32, device=DEV)


def _topk_inputs(case, seed):
    return _column(_gen(seed), case["n"], case["type"], case["dist"])


def _pair_inputs(case, seed):
    g = _gen(seed)
    return _column(g, case["n"], "i32", "dup1024"), _column(g, case["n"], "i32", "uniform")


def _build_keys(g, n, mult="unique"):
    """Unique: random 64-bit keys.  mult14: each distinct key one to four
    times, shuffled, about n rows."""
    if mult == "unique":
        return _uniform(g, n, "i64")
    distinct = _uniform(g, max(1, n * 2 // 5), "i64")
    rows = distinct.repeat_interleave(torch.randint(1, 5, distinct.shape, device=DEV, generator=g))
    return rows[torch.randperm(rows.numel(), device=DEV, generator=g)]


def _probe_keys(g, build, n, hit, dist="uniform"):
    d = build.numel()
    if dist == "zipf":
        w = torch.arange(1, d + 1, dtype=torch.float64, device=DEV).pow(-1.1).cumsum(0)
        u = torch.rand(n, dtype=torch.float64, device=DEV, generator=g) * w[-1]
        pick = torch.searchsorted(w, u).clamp_(max=d - 1)
    else:
        pick = torch.randint(0, d, (n,), device=DEV, generator=g)
    keys = build[pick]
    miss = torch.rand(n, device=DEV, generator=g) >= hit
    return torch.where(miss, _uniform(g, n, "i64"), keys)


def _probe_inputs(case, seed):
    g = _gen(seed)
    build = _build_keys(g, case["build"], case.get("mult", "unique"))
    return build, _probe_keys(g, build, case["n"], case["hit"], case.get("dist", "uniform"))


def _batch_sizes(case):
    """Top-K sizes (N log-uniform 1e3..4e6, K 1..1000) and probe sizes
    (log-uniform 1e3..1e6) of a batch."""
    r = np.random.RandomState(case["sizes"])
    ns = np.floor(1e3 * np.power(4e3, r.random_sample(case["topk"]))).astype(np.int64)
    ks = np.minimum(r.randint(1, 1001, case["topk"]), ns)
    ps = np.floor(1e3 * np.power(1e3, r.random_sample(case["probe"]))).astype(np.int64)
    return [int(x) for x in ns], [int(x) for x in ks], [int(x) for x in ps]


def _batch_inputs(case, seed):
    g = _gen(seed)
    ns, _, ps = _batch_sizes(case)
    build = _build_keys(g, case["build"])
    return _uniform(g, sum(ns), "i64"), build, _probe_keys(g, build, sum(ps), 0.5)


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def prepare(case, seed):
    ctx, s = _context(), {"op": case["op"], "case": case}
    s["ctx"] = ctx
    if case["op"] == "topk":
        keys = _typed(_topk_inputs(case, seed), case["type"])
        rowids = _rowids(case["n"]) if case["rowids"] else None
        if case["where"] == "pinned":
            keys = keys.cpu().pin_memory()
            rowids = rowids.cpu().pin_memory() if rowids is not None else None
        elif case["where"] == "pageable":
            keys = keys.cpu().numpy()
            rowids = rowids.cpu().numpy() if rowids is not None else None
        s.update(keys=keys, rowids=rowids, order=ORDERS[case["order"]])
        if case["mode"] != "host":
            s["out_keys"] = torch.empty(case["k"], dtype=KEYS[case["type"]], device=DEV)
            s["out_rowids"] = torch.empty(case["k"], dtype=torch.int32, device=DEV)
    elif case["op"] == "pair":
        s["c0"], s["c1"] = _pair_inputs(case, seed)
        s["rowids"] = _rowids(case["n"]) if case["rowids"] else None
        s["out"] = [torch.empty(case["k"], dtype=torch.int32, device=DEV) for _ in range(3)]
    elif case["op"] == "probe":
        build, s["keys"] = _probe_inputs(case, seed)
        s["rowids"] = _rowids(case["n"]) if case["rowids"] else None
        s["table"] = ctx.join_build(build)
        s["pairs"] = torch.empty((case["n"], 2), dtype=torch.int32, device=DEV)
        s["match"] = torch.empty(case["n"], dtype=torch.int32, device=DEV)
    elif case["op"] == "join":
        s["build"], s["keys"] = _probe_inputs(case, seed)
        most = case["n"] if case["mult"] == "unique" else 4 * case["n"]
        s["pairs"] = torch.empty((most, 2), dtype=torch.int32, device=DEV)
        s["match"] = torch.empty(case["n"], dtype=torch.int32, device=DEV)
    else:
        ns, ks, ps = _batch_sizes(case)
        keys, build, probe = _batch_inputs(case, seed)
        total = sum(ps)
        s.update(keys=keys, probe=probe, rowids=_rowids(total), table=ctx.join_build(build))
        s["out_keys"] = torch.empty(sum(ks), dtype=torch.int64, device=DEV)
        s["out_rowids"] = torch.empty(sum(ks), dtype=torch.int32, device=DEV)
        s["counts"] = torch.zeros(len(ns) + len(ps), dtype=torch.int64, device=DEV)
        # every item appends to its own range; entries past its count name the spare row `total`
        s["pairs"] = torch.full((total, 2), total, dtype=torch.int32, device=DEV)
        s["match"] = torch.empty(total + 1, dtype=torch.int32, device=DEV)
        items, a, o = [], 0, 0
        for i, (n, k) in enumerate(zip(ns, ks)):
            items.append(olap.topk_item(keys[a:a + n], k, olap.DESC, s["out_keys"][o:o + k],
                                        s["out_rowids"][o:o + k], s["counts"][i:i + 1]))
            a, o = a + n, o + k
        a = 0
        for i, n in enumerate(ps):
            items.append(olap.probe_item(s["table"], probe[a:a + n], s["pairs"][a:a + n], n,
                                         s["counts"][len(ns) + i:len(ns) + i + 1], d_rowids=s["rowids"][a:a + n]))
            a += n
        s["batch"] = ctx.batch(items)
    return s


def _after(ctx):
    """Order torch's stream after the context's, to use what the context wrote."""
    torch.cuda.current_stream().wait_stream(torch.cuda.ExternalStream(ctx.stream))


def _materialise(s, pairs):
    """The build row of every probe row (unique build keys): -1 without one."""
    m = s["match"].fill_(-1)
    return m.scatter_(0, pairs[:, 0].long(), pairs[:, 1])


def run(s):
    ctx, op = s["ctx"], s["op"]
    if op == "topk":
        k, mode = s["case"]["k"], s["case"]["mode"]
        if mode == "host":
            return ctx.topk(s["keys"], k, s["order"], rowids=s["rowids"])
        if mode == "block":
            return ctx.topk(s["keys"], k, s["order"], rowids=s["rowids"], out_keys=s["out_keys"],
                            out_rowids=s["out_rowids"])
        if mode == "noalloc":
            olap.topk_noalloc(s["keys"], k, s["order"], s["out_keys"], s["out_rowids"], d_rowids=s["rowids"])
        else:
            ctx.topk_async(s["keys"], k, s["order"], s["out_keys"], s["out_rowids"], d_rowids=s["rowids"])
        return s["out_keys"], s["out_rowids"]
    if op == "pair":
        o, c = s["out"], s["case"]
        return ctx.topk_pair(s["c0"], ORDERS[c["order0"]], s["c1"], ORDERS[c["order1"]], c["k"], rowids=s["rowids"],
                             out_keys0=o[0], out_keys1=o[1], out_rowids=o[2])
    if op == "probe":
        return _materialise(s, ctx.join_probe(s["table"], s["keys"], rowids=s["rowids"], out=s["pairs"]))
    if op == "join":
        table = ctx.join_build(s["build"])
        pairs = ctx.join_probe(table, s["keys"], out=s["pairs"])
        table.free()
        if s["case"]["mult"] == "unique":
            return _materialise(s, pairs)
        return torch.sort(pairs.view(torch.int64).view(-1)).values
    s["batch"].run()
    _after(ctx)
    return s["out_keys"], s["out_rowids"], s["counts"], _materialise(s, s["pairs"])[:-1]


def work(case):
    """Each input read once, each output written once."""
    if case["op"] == "topk":
        w, k = (8 if case["type"].endswith("64") else 4), case["k"]
        return {"bytes": case["n"] * w + k * (w + 4) + (4 * k if case["rowids"] else 0), "flops": 0}
    if case["op"] == "pair":
        return {"bytes": case["n"] * 8 + case["k"] * (16 if case["rowids"] else 12), "flops": 0}
    if case["op"] == "probe":
        # a table slot is 16 bytes per build row, of which a probe reads at most one per row
        return {"bytes": case["n"] * (16 if case["rowids"] else 12) + 16 * min(case["build"], case["n"]), "flops": 0}
    if case["op"] == "join":
        out = case["n"] * (4 if case["mult"] == "unique" else 20 * case["hit"])
        return {"bytes": 8 * (case["build"] + case["n"]) + out, "flops": 0}
    ns, ks, ps = _batch_sizes(case)
    return {"bytes": 8 * sum(ns) + 12 * sum(ks) + 16 * sum(ps) + 16 * min(case["build"], sum(ps)), "flops": 0}


# ---------------------------------------------------------------------------
# The same results from torch alone
# ---------------------------------------------------------------------------

def _sortable(keys, typ):
    """Keys as a type torch sorts, in the key type's order."""
    if typ == "u64":
        return keys ^ -(1 << 63)
    if typ == "u32":
        return keys.long() & 0xFFFFFFFF
    return keys


def _top(keys, k, typ, desc):
    """Keys and row-ids of the first k rows, ties by row-id."""
    idx = torch.sort(_sortable(keys, typ), descending=desc, stable=True).indices[:k]
    sel = keys[idx]
    return (sel.double() if sel.is_floating_point() else _typed(sel, typ)), idx.to(torch.int32)


def _match(build, probe):
    b, at = torch.sort(build)
    pos = torch.searchsorted(b, probe).clamp_(max=b.numel() - 1)
    return torch.where(b[pos] == probe, at[pos].int(), -1)


def exact(case, seed):
    if case["op"] == "topk":
        keys = _topk_inputs(case, seed)
        k, r = _top(keys, case["k"], case["type"], case["order"] == "desc")
        return (k.cpu().numpy(), r.cpu().numpy().view(np.uint32)) if case["mode"] == "host" else (k, r)
    if case["op"] == "pair":
        c0, c1 = _pair_inputs(case, seed)
        i1 = torch.sort(c1, descending=case["order1"] == "desc", stable=True).indices
        idx = i1[torch.sort(c0[i1], descending=case["order0"] == "desc", stable=True).indices[:case["k"]]]
        return c0[idx], c1[idx], idx.to(torch.int32)
    if case["op"] in ("probe", "join"):
        build, probe = _probe_inputs(case, seed)
        if case.get("mult", "unique") == "unique":
            return _match(build, probe)
        b, at = torch.sort(build)
        lo, hi = torch.searchsorted(b, probe), torch.searchsorted(b, probe, right=True)
        cnt = hi - lo
        first = (cnt.cumsum(0) - cnt).repeat_interleave(cnt)
        pos = lo.repeat_interleave(cnt) + torch.arange(first.numel(), device=DEV) - first
        rows = torch.arange(probe.numel(), device=DEV).repeat_interleave(cnt)
        return torch.sort((at[pos] << 32) | rows).values
    ns, ks, ps = _batch_sizes(case)
    keys, build, probe = _batch_inputs(case, seed)
    tops = [_top(part, k, "i64", True) for part, k in zip(keys.split(ns), ks)]
    m = _match(build, probe)
    hits = torch.stack([(part >= 0).sum() for part in m.split(ps)])
    counts = torch.cat([torch.tensor(ks, dtype=torch.int64, device=DEV), hits])
    return torch.cat([t[0] for t in tops]), torch.cat([t[1] for t in tops]), counts, m
