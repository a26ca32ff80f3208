"""Performance cases of the fused columnar query library.

Each case is one unit of work that a program using the library repeats: a
prepared query launched and its records read, an ad hoc query that builds its
join tables first, a batch, a join chain replayed from its graph, a table
load.  ``listed()`` names the standing ones, ``draw(rng)`` gives more of the
same ranges.  Every result is whole numbers, so outputs compare exactly.

Inputs are generated from the seed on the GPU and handed to the library as
host arrays, as a loader would; the shapes follow the workloads of
``synth/tables.py`` (uniform foreign keys into dimensions of 2,000 / 30,000 /
200,000 rows, a seven-year date dimension, Zipf dictionary keys, word text).

    family  what it stands for
    scan    filter and aggregate over one table: dashboards, the smallest calls
    star    four-way star join with a group-by, the flagship analytic query
    prefix  LIKE 'p%' over raw strings grouped by a dictionary key
            (plen = 0: every row passes, a pure group-by over a Zipf key)
    text    LIKE over word text: '%w%', 'w%' and general patterns, raw or FSST
    chain   LINEITEM -> ORDERS -> CUSTOMER: two table builds, then the probe
    batch   many queries of mixed shapes and sizes in one launch
    load    host columns (every integer codec, raw strings) into device pages

    call      how the program runs it
    prepared  dpf_launch of a prepared batch, then dpf_read_result
    graph     the same from its captured CUDA graph
    adhoc     prepare, launch, read and release (and build tables) every time
    async     adhoc with the tables built by enqueue-only builds
    noalloc   dpf_execute_noalloc into the caller's device buffers
"""

import datetime
import math

import numpy as np
import torch

import paper_2605_10511_gb300 as dpf

DEV = "cuda" if torch.cuda.is_available() else "cpu"
YEARS = 7


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the first workload of the benchmark: a million rows, where launch and read-back count
        {"name": "scan_1m", "family": "scan", "rows": 1 << 20, "page_rows": 0, "a_lt": 25, "b_hi": 3, "call": "prepared"},
        # a small interactive query on a chain of joins whose tables are built for it
        {"name": "chain_adhoc_60k", "family": "chain", "rows": 60_000, "page_rows": 0, "sparse": False, "call": "adhoc"},
        # the headline: 67 M fact rows sorted by date, replayed from a graph
        {"name": "star_64m", "family": "star", "rows": 1 << 26, "page_rows": 0, "clustered": True, "bigint": False,
         "year": False, "host": False, "call": "graph"},
        # an unsorted fact with a 64-bit measure and ragged length, results left on the device
        {"name": "star_bigint_5m", "family": "star", "rows": 5_000_011, "page_rows": 0, "clustered": False, "bigint": True,
         "year": False, "host": False, "call": "noalloc"},
        # a fact table too large for device memory: its pages are read over the host link
        {"name": "star_host_16m", "family": "star", "rows": 1 << 24, "page_rows": 0, "clustered": True, "bigint": False,
         "year": False, "host": True, "call": "prepared"},
        # one-letter prefix over raw strings, 1,024 Zipf groups
        {"name": "prefix_32m", "family": "prefix", "rows": 1 << 25, "page_rows": 0, "plen": 1, "groups": 1024, "call": "graph"},
        # a pure group-by on a skewed key: every row is aggregated
        {"name": "groupby_10m", "family": "prefix", "rows": 10_000_019, "page_rows": 8192, "plen": 0, "groups": 1024,
         "call": "prepared"},
        # substring search over FSST-compressed text
        {"name": "contains_fsst_8m", "family": "text", "rows": 1 << 23, "page_rows": 0, "codec": "fsst", "op": "contains",
         "plen": 3, "rank": 20, "call": "prepared"},
        # a general LIKE pattern over raw text
        {"name": "like_str_3m", "family": "text", "rows": 3_000_017, "page_rows": 0, "codec": "str", "op": "like",
         "plen": 3, "rank": 20, "call": "prepared"},
        # the three-table pipeline as one graph: both builds and the probe scan
        {"name": "chain_16m", "family": "chain", "rows": 1 << 24, "page_rows": 0, "sparse": False, "call": "graph"},
        # a batch of uneven queries in one launch
        {"name": "batch_24", "family": "batch", "queries": 24, "log2_hi": 22.0, "page_rows": 0, "call": "prepared"},
        # a mixed table brought in from host memory
        {"name": "load_1m", "family": "load", "rows": 1 << 20, "page_rows": 0},
    ]


def _log(rng, lo, hi):
    """A whole number spread evenly over the logarithm, odd values included."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["scan", "star", "star", "prefix", "prefix", "text", "text", "chain", "chain", "batch", "load"])
    page_rows = rng.choice([0, 0, 4096, 8192])
    if family == "scan":
        return {"family": family, "rows": _log(rng, 4_096, 1 << 23), "page_rows": page_rows, "a_lt": rng.randint(2, 50),
                "b_hi": rng.randint(1, 20), "call": rng.choice(["prepared", "graph", "adhoc", "noalloc"])}
    if family == "star":
        return {"family": family, "rows": _log(rng, 1 << 14, 1 << 25), "page_rows": page_rows,
                "clustered": rng.random() < 0.6, "bigint": rng.random() < 0.3, "year": rng.random() < 0.25,
                "host": rng.random() < 0.15, "call": rng.choice(["prepared", "graph", "noalloc"])}
    if family == "prefix":
        return {"family": family, "rows": _log(rng, 1 << 13, 1 << 24), "page_rows": page_rows, "plen": rng.choice([0, 1, 1, 2]),
                "groups": _log(rng, 3, 8192), "call": rng.choice(["prepared", "graph"])}
    if family == "text":
        codec = rng.choice(["str", "fsst"])
        return {"family": family, "rows": _log(rng, 1 << 12, 1 << 22), "page_rows": page_rows, "codec": codec,
                "op": rng.choice(["contains", "prefix"] + (["like"] if codec == "str" else [])),
                "plen": rng.randint(2, 12), "rank": _log(rng, 1, 400), "call": rng.choice(["prepared", "graph"])}
    if family == "chain":
        return {"family": family, "rows": _log(rng, 1 << 14, 1 << 24), "page_rows": page_rows, "sparse": rng.random() < 0.3,
                "call": rng.choice(["graph", "adhoc", "async"])}
    if family == "batch":
        return {"family": family, "queries": rng.randint(3, 24), "log2_hi": round(rng.uniform(16, 21.5), 2),
                "page_rows": page_rows, "call": rng.choice(["prepared", "graph"])}
    return {"family": family, "rows": _log(rng, 1 << 6, 1 << 13) * 128 + rng.randint(96, 127), "page_rows": page_rows}


# ----------------------------------------------------------------- generation
class _Gen:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(DEV)
        self.g.manual_seed(int(seed) * 7919 + 12345)

    def ints(self, lo, hi, n):
        """n whole numbers in [lo, hi)."""
        return torch.randint(int(lo), int(hi), (int(n),), generator=self.g, device=DEV, dtype=torch.int64).to(torch.int32)

    def perm(self, n):
        return torch.randperm(int(n), generator=self.g, device=DEV).to(torch.int32)

    def unit(self, n):
        return torch.rand((int(n),), generator=self.g, device=DEV, dtype=torch.float64)

    def one(self, lo, hi):
        return int(self.ints(lo, hi, 1)[0])


def _dates():
    first = datetime.date(1992, 1, 1)
    days = [first + datetime.timedelta(days=i) for i in range(2556)]
    return torch.tensor([d.year * 10000 + d.month * 100 + d.day for d in days], dtype=torch.int32, device=DEV)


def _zipf(g, rows, n, s=1.1):
    w = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) ** (-s)
    cdf = torch.cumsum(w, 0) / w.sum()
    return torch.clamp(torch.searchsorted(cdf, g.unit(rows), right=True), max=n - 1)


def _values(g, count, lo, hi):
    """count distinct ascending values of [lo, hi)."""
    return torch.sort(g.perm(hi - lo)[:count])[0] + lo


def _col(codec, t):
    return {"codec": codec, "t": t}


def _page(case):
    return case["page_rows"] or 65536


def _scan(g, rows, a_lt, b_lo, b_hi):
    cols = {"a": _col("for", g.ints(1, 51, rows)), "b": _col("for", g.ints(1, 51, rows)),
            "c": _col("for", g.ints(1, 11, rows)), "d": _col("for", g.ints(900, 105001, rows))}
    query = {"preds": [{"col": "a", "op": "lt", "args": [a_lt]}, {"col": "b", "op": "between", "args": [b_lo, b_hi]}],
             "joins": [], "group": [], "aggs": [{"op": "sum_mul", "cols": ["c", "d"]}]}
    return {"fact": cols}, query


def _star(g, rows, clustered, bigint, year):
    n1, n2, n3 = 2_000, 30_000, 200_000
    a1, a2, a3 = _values(g, 10, 0, 1000), _values(g, 25, 0, 1000), _values(g, 25, 0, 1000)
    b3 = _values(g, 5, 0, 100)
    dk = _dates()
    dp = dk[g.perm(dk.numel()).long()]
    tables = {
        "dim1": {"k": _col("for", g.perm(n1) + 1), "A1": _col("dict", a1[g.ints(0, 10, n1).long()])},
        "dim2": {"k": _col("for", g.perm(n2) + 1), "A2": _col("dict", a2[g.ints(0, 25, n2).long()])},
        "dim3": {"k": _col("for", g.perm(n3) + 1), "A3": _col("dict", a3[g.ints(0, 25, n3).long()]),
                 "B3": _col("dict", b3[g.ints(0, 5, n3).long()])},
        "date": {"k": _col("for", dp), "year": _col("dict", dp // 10000)},
    }
    di = g.ints(0, dk.numel(), rows)
    if clustered:
        di = torch.sort(di)[0]
    m1 = g.ints(1, 10_000_000, rows)
    fact = {"fk1": _col("for", g.ints(1, n1 + 1, rows)), "fk2": _col("for", g.ints(1, n2 + 1, rows)),
            "fk3": _col("for", g.ints(1, n3 + 1, rows)), "fkd": _col("delta" if clustered else "for", dk[di.long()])}
    fact["m1"] = _col("for64", (m1.long() << 20) + g.ints(1, 100_000, rows)) if bigint else _col("for", m1)
    tables["fact"] = fact
    i3 = g.one(0, 24)
    pick = [int(a1[g.one(0, 10)]), int(a2[g.one(0, 25)]), int(a3[i3]), int(a3[i3 + 1]), 1992 + g.one(0, YEARS)]
    query = {"preds": [], "joins": [
        {"fk": "fk1", "dim": "dim1", "key": "k", "preds": [{"col": "A1", "op": "eq", "args": pick[:1]}], "payload": []},
        {"fk": "fk2", "dim": "dim2", "key": "k", "preds": [{"col": "A2", "op": "eq", "args": pick[1:2]}], "payload": []},
        {"fk": "fk3", "dim": "dim3", "key": "k", "preds": [{"col": "A3", "op": "in", "args": pick[2:4]}], "payload": ["B3"]},
        {"fk": "fkd", "dim": "date", "key": "k",
         "preds": [{"col": "year", "op": "eq", "args": pick[4:]}] if year else [], "payload": ["year"]}],
        "group": [{"join": 2, "field": 0}, {"join": 3, "field": 0}], "aggs": [{"op": "sum", "cols": ["m1"]}]}
    return tables, query


def _offsets(lengths):
    off = torch.zeros(lengths.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lengths.long(), 0, out=off[1:])
    return off


def _prefix(g, rows, plen, groups):
    off = _offsets(g.ints(10, 45, rows))
    letters = torch.tensor(list(b"abcdefghijklmnopqrstuvwxyz "), dtype=torch.uint8, device=DEV)
    data = letters[torch.randint(0, 27, (int(off[-1]),), generator=g.g, device=DEV, dtype=torch.uint8).int()]
    keys = _values(g, groups, -32768, 32768)
    cols = {"s": {"codec": "str", "bytes": data, "offsets": off}, "key": _col("dict", keys[_zipf(g, rows, groups)]),
            "m": _col("for", g.ints(1, 1_000_001, rows))}
    want = bytes(int(letters[g.one(0, 27)]) for _ in range(plen))
    query = {"preds": [{"col": "s", "op": "prefix", "args": [want]}], "joins": [], "group": [{"col": "key"}],
             "aggs": [{"op": "count"}, {"op": "sum", "cols": ["m"]}]}
    return {"fact": cols}, query


def _words(g, rows):
    """Word text cut into strings of 10..44 bytes, and the vocabulary."""
    n_words = 512
    wl = g.ints(3, 10, n_words).long()
    W = (g.ints(97, 123, n_words * 10)).reshape(n_words, 10).to(torch.uint8)
    at = torch.arange(10, device=DEV)[None, :]
    W = torch.where(at < wl[:, None], W, torch.full_like(W, 32))
    off = _offsets(g.ints(10, 45, rows))
    total = int(off[-1])
    need = total // 5 + 64                # a word and its space take at least 4 bytes, 6 to 7 on average
    parts, have = [], 0
    while have < total:
        pick = _zipf(g, need, n_words)
        part = W[pick][at < (wl + 1)[pick][:, None]]
        parts.append(part)
        have += part.numel()
    words = [bytes(W[i, :int(k)].tolist()) for i, k in enumerate(wl.tolist())]
    return torch.cat(parts)[:total].contiguous(), off, words


def _pattern(words, op, plen, rank):
    """A pattern from the vocabulary: common words at low ranks."""
    a, b, c = (words[(rank + i) % len(words)] for i in range(3))
    if op == "like":                      # '%ab_%cd%': runs, a single-byte wildcard, two parts
        return b"%" + a[:plen] + b"_%" + b[:2] + b"%"
    return (a + b" " + b + b" " + c)[:plen]


def _text(g, rows, codec, op, plen, rank):
    data, off, words = _words(g, rows)
    keys = _values(g, 64, -32768, 32768)
    cols = {"s": {"codec": codec, "bytes": data, "offsets": off}, "key": _col("dict", keys[_zipf(g, rows, 64)]),
            "m": _col("for", g.ints(1, 1_000_001, rows))}
    query = {"preds": [{"col": "s", "op": op, "args": [_pattern(words, op, plen, rank)]}], "joins": [],
             "group": [{"col": "key"}], "aggs": [{"op": "count"}, {"op": "sum", "cols": ["m"]}]}
    return {"fact": cols}, query


def _chain(g, rows, sparse):
    n_ord = max(rows // 4, 1)
    n_cust = max(n_ord // 10, 1)
    dk = _dates()
    seg = _values(g, 5, 0, 100)
    customer = {"c_custkey": _col("for", g.perm(n_cust) + 1), "c_segment": _col("dict", seg[g.ints(0, 5, n_cust).long()]),
                "c_nation": _col("dict", g.ints(0, 25, n_cust))}
    if sparse:                            # order keys over the whole positive range, 4 ascending steps' worth of gaps
        gap = (2**31 - 2) // n_ord
        okeys = torch.arange(n_ord, dtype=torch.int64, device=DEV) * gap + 1 + g.ints(0, gap, n_ord).long()
        okeys = okeys.to(torch.int32)
    else:
        okeys = torch.sort(g.perm(4 * n_ord)[:n_ord])[0] + 1
    oi = g.ints(0, dk.numel() - 151, n_ord).long()
    perm = g.perm(n_ord).long()           # ORDERS is not stored in key order
    orders = {"o_orderkey": _col("for", okeys[perm]), "o_custkey": _col("for", g.ints(1, n_cust + 1, n_ord)),
              "o_orderdate": _col("for", dk[oi[perm]]), "o_priority": _col("dict", g.ints(1, 6, n_ord))}
    li = torch.sort(g.ints(0, n_ord, rows))[0].long()
    fact = {"l_orderkey": _col("delta", okeys[li]), "l_shipdate": _col("for", dk[oi[li] + g.ints(1, 122, rows).long()]),
            "l_price": _col("for", g.ints(90_000, 10_500_001, rows)), "l_discount": _col("for", g.ints(0, 11, rows))}
    cut = int(dk[int(dk.numel() * 0.45)])
    query = {"preds": [{"col": "l_shipdate", "op": "gt", "args": [cut]}],
             "joins": [{"fk": "l_orderkey", "dim": "orders", "key": "o_orderkey",
                        "preds": [{"col": "o_orderdate", "op": "lt", "args": [cut]}],
                        "payload": [{"join": 0, "field": 0}, "o_priority"],
                        "joins": [{"fk": "o_custkey", "dim": "customer", "key": "c_custkey",
                                   "preds": [{"col": "c_segment", "op": "eq", "args": [int(seg[g.one(0, 5)])]}],
                                   "payload": ["c_nation"]}]}],
             "group": [{"join": 0, "field": 0}, {"join": 0, "field": 1}],
             "aggs": [{"op": "count"}, {"op": "sum", "cols": ["l_price"]}, {"op": "sum_mul", "cols": ["l_price", "l_discount"]}]}
    return {"customer": customer, "orders": orders, "fact": fact}, query


def _batch_shapes(case):
    """Shape and rows of each query: uneven, the last one largest."""
    n = case["queries"]
    return [(("scan", "star", "prefix")[i % 3], int(2.0 ** (12.0 + (case["log2_hi"] - 12.0) * ((i * 7 + 3) % n + 1) / n)) + i)
            for i in range(n)]


def _load(g, rows):
    # widths and string bytes are the same in every block of 128 rows, so
    # that pages have the same sizes whatever the seed
    keys = _values(g, 1000, -32768, 32768)
    blocks = torch.rand((rows // 128, 128), generator=g.g, device=DEV).argsort(1).reshape(-1)
    off = _offsets(10 + torch.cat([blocks, torch.arange(rows % 128, device=DEV)]) % 48)
    return {"fact": {"id": _col("delta", torch.cumsum(g.ints(0, 8, rows), 0).to(torch.int32)),
                     "price": _col("for", g.ints(90_000, 10_500_001, rows)), "key": _col("dict", keys[g.ints(0, 1000, rows).long()]),
                     "big": _col("for64", (g.ints(1, 10_000_000, rows).long() << 20) + g.ints(1, 100_000, rows)),
                     "s": {"codec": "str", "bytes": g.ints(97, 123, int(off[-1])).to(torch.uint8), "offsets": off}}}, None


def _tables(case, seed):
    """[(tables, query)] of a case: one, or one per query of a batch."""
    g = _Gen(seed)
    f = case["family"]
    if f == "scan":
        return [_scan(g, case["rows"], case["a_lt"], 1, case["b_hi"])]
    if f == "star":
        return [_star(g, case["rows"], case["clustered"], case["bigint"], case["year"])]
    if f == "prefix":
        return [_prefix(g, case["rows"], case["plen"], case["groups"])]
    if f == "text":
        return [_text(g, case["rows"], case["codec"], case["op"], case["plen"], case["rank"])]
    if f == "chain":
        return [_chain(g, case["rows"], case["sparse"])]
    if f == "load":
        return [_load(g, case["rows"])]
    make = {"scan": lambda n: _scan(g, n, g.one(2, 50), g.one(1, 10), g.one(10, 20)),
            "star": lambda n: _star(g, n, g.one(0, 2) == 1, False, False),
            "prefix": lambda n: _prefix(g, n, g.one(1, 3), 1024)}
    return [make[s](n) for s, n in _batch_shapes(case)]


def _host(col):
    """A column as the library takes it: host arrays."""
    if "bytes" in col:
        return {"codec": col["codec"], "bytes": col["bytes"].cpu().numpy(), "offsets": col["offsets"].cpu().numpy().view(np.uint64)}
    return {"codec": col["codec"], "values": col["t"].cpu().numpy()}


def _workload(case, i, tables, query):
    return {"name": f"w{i}", "fact": "fact", "query": query,
            "tables": {t: {"rows": int(next(iter(c.values()))["t"].numel()) if "t" in next(iter(c.values()))
                           else int(next(iter(c.values()))["offsets"].numel()) - 1,
                           "page_rows": _page(case), "cols": {k: _host(v) for k, v in c.items()}} for t, c in tables.items()}}


# ------------------------------------------------------------------- the path
def prepare(case, seed):
    ws = [_workload(case, i, t, q) for i, (t, q) in enumerate(_tables(case, seed))]
    if case["family"] == "load":
        return {"call": "load", "ctx": dpf.Context(0), "cols": ws[0]["tables"]["fact"]["cols"], "page_rows": case["page_rows"]}
    call = case["call"]
    eng = dpf.Engine(device=0)
    for w in ws:
        eng.load_workload(w, fact_placement="host" if case.get("host") else None)
        for t in w["tables"].values():     # a program that has loaded its columns drops the host copies
            t["cols"] = {k: None for k in t["cols"]}
    s = {"eng": eng, "ws": ws, "call": call, "n": len(ws), "room": _room(case)}
    if call in ("adhoc", "async"):
        return s
    if case["family"] == "chain":
        s["prep"] = eng.prepare_chain(ws[0])
        s["chain"] = True
    else:
        s["plans"] = [eng.plan(w) for w in ws]
        if call == "noalloc":
            s["out"] = torch.zeros((s["room"][0], 6), dtype=torch.int64, device=DEV)
            s["count"] = torch.zeros(1, dtype=torch.int32, device=DEV)
            return s
        s["prep"] = eng.ctx.prepare(s["plans"])
    s["stream"] = torch.cuda.Stream()
    if call == "graph":
        eng.ctx.capture_graph(s["prep"], s["stream"])
    return s


def _room(case):
    """Most records of each of the case's queries: its group domain."""
    one = {"scan": 1, "star": 5 * YEARS, "prefix": case.get("groups", 1024), "text": 64, "chain": 25 * 5}
    return [one[s] for s, _ in _batch_shapes(case)] if case["family"] == "batch" else [one[case["family"]]]


def _records(room, got):
    """The queries' records one after the other, each in its own room."""
    if len(room) > 1 or len(got[0]) < room[0]:
        r = np.zeros(sum(room), dpf.RECORD_DTYPE)
        at = 0
        for n, g in zip(room, got):
            r[at:at + len(g)] = g
            at += n
    else:
        r = got[0]
    return {"key": r["key"], "count": r["count"], "val": r["val"]}


def run(state):
    call = state["call"]
    if call == "load":
        ctx = state["ctx"]
        ids = [ctx.load_column(c, table=1, page_rows=state["page_rows"]) for c in state["cols"].values()]
        pages = [ctx.column_bytes(i) for i in ids]
        for i in ids:
            ctx.drop_column(i)
        return pages
    eng = state["eng"]
    ctx = eng.ctx
    if call == "noalloc":
        ctx.execute_noalloc(state["plans"][0], state["out"].data_ptr(), state["out"].shape[0], state["count"].data_ptr())
        return {"count": state["count"], "records": state["out"]}
    if call in ("adhoc", "async"):
        w = state["ws"][0]
        h = eng.plan(w, asynchronous=call == "async")
        rec = ctx.fetch(ctx.execute([h])[0])
        if call == "async":
            eng.wait_joins(w)
        for ht in eng.chain_tables(w):     # this query's tables are its own
            ctx.drop_hash(ht)
        eng.hts.clear()
        return _records(state["room"], [rec])
    if call == "graph":
        ctx.launch_graph(state["prep"], state["stream"])
    else:
        ctx.launch(state["prep"], state["stream"])
    out = [ctx.read_result(state["prep"], i) for i in range(state["n"])]
    if state.get("chain"):
        eng.wait_joins(state["ws"][0], deferred=True)
    return _records(state["room"], out)


def _bits(case):
    """Encoded bytes of the columns that a case's queries read (per row: the
    packed widths, and 8 or 16 bytes of header per 128 values)."""
    def per(*widths):
        return sum(w / 8 + h / 128 for w, h in widths)
    scan = per((6, 8), (6, 8), (4, 8), (17, 8))
    dims = 2_000 * 2 + 30_000 * 3 + 200_000 * 4
    f = case["family"]
    rows = case.get("rows", 0)
    strings = 27.0 + per((6, 12), (20, 8))
    if f == "scan":
        return rows * scan
    if f == "star":
        return rows * per((11, 8), (15, 8), (18, 8), (1, 16) if case["clustered"] else (17, 8), (44, 16) if case["bigint"] else (24, 8))
    key = per((max(1, math.ceil(math.log2(case.get("groups", 64)))), 8))
    if f == "prefix":
        return rows * (key + (strings if case["plen"] else per((20, 8))))
    if f == "text":
        return rows * (key + (strings if case["codec"] == "str" else strings - 12.0))
    if f == "chain":
        return rows * (per((3, 16), (12, 8), (24, 8), (4, 8)) + per((24, 8), (20, 8), (17, 8), (3, 8)) / 4 + per((20, 8), (3, 8), (5, 8)) / 40)
    if f == "batch":
        one = {"scan": scan, "star": per((11, 8), (15, 8), (18, 8), (9, 12), (24, 8)), "prefix": strings + per((10, 8))}
        return sum(n * one[s] for s, n in _batch_shapes(case)) + dims * sum(s == "star" for s, _ in _batch_shapes(case))
    # load: the host values in, the pages out (and read back)
    return rows * (4 + 4 + 4 + 8 + 33 + 8 + 2 * (33 + per((3, 16), (24, 8), (10, 8), (44, 16), (6, 12))))


def work(case):
    """One pass reads the encoded columns once; records are negligible beside
    them.  No floating-point work."""
    return {"bytes": float(_bits(case)), "flops": 0}


def tolerance(case):
    return "exact"                         # int64 sums and page bytes


# ---------------------------------------------------------------- the answers
def _group(keys, aggs):
    """Records of rows with dictionary keys (list of int tensors) and
    aggregate values (list of int64 tensors): ascending by key."""
    if not keys:
        r = np.zeros(1, dpf.RECORD_DTYPE)
        r["count"] = aggs[0].numel()
        r["val"][0, :len(aggs)] = [int(a.sum()) for a in aggs]
        return r
    both = torch.stack([k.long() for k in keys] + [torch.zeros_like(keys[0]).long()] * (2 - len(keys)), 1)
    u, inv, cnt = torch.unique(both, dim=0, return_inverse=True, return_counts=True)
    r = np.zeros(u.shape[0], dpf.RECORD_DTYPE)
    r["key"], r["count"] = u.to(torch.int32).cpu().numpy(), cnt.cpu().numpy()
    for i, a in enumerate(aggs):
        r["val"][:, i] = torch.zeros(u.shape[0], dtype=torch.int64, device=u.device).index_add_(0, inv, a).cpu().numpy()
    return r


def _cmp(v, op, args):
    if op == "lt":
        return v < args[0]
    if op == "gt":
        return v > args[0]
    if op == "eq":
        return v == args[0]
    if op == "between":
        return (v >= args[0]) & (v <= args[1])
    return torch.isin(v, torch.tensor(args, device=v.device, dtype=v.dtype))


def _matches(col, op, pat):
    """Which strings match: each part of the pattern found greedily."""
    data, off = col["bytes"], col["offsets"]
    start, end = off[:-1].clone(), off[1:]
    total = data.numel()
    ok = torch.ones(start.numel(), dtype=torch.bool, device=data.device)
    if op == "prefix":
        for i, b in enumerate(pat):
            at = start + i
            ok &= (at < end) & (data[torch.clamp(at, max=total - 1)] == b)
        return ok
    for part in [p for p in pat.split(b"%") if p] if op == "like" else [pat]:
        hit = torch.ones(max(total - len(part) + 1, 0), dtype=torch.bool, device=data.device)
        for i, b in enumerate(part):
            if op != "like" or b != ord("_"):
                hit &= data[i:i + hit.numel()] == b
        at = torch.full((total + 1,), 2 * total, dtype=torch.int64, device=data.device)
        at[:hit.numel()] = torch.where(hit, torch.arange(hit.numel(), device=data.device), at[:hit.numel()])
        nxt = torch.flip(torch.cummin(torch.flip(at, [0]), 0)[0], [0])
        start = nxt[torch.clamp(start, max=total)] + len(part)
        ok &= start <= end
    return ok


def _lookup(tables, j, fk):
    """(match, payload values) of foreign keys fk in join j's dimension rows."""
    d = tables[j["dim"]]
    keep = torch.ones(d[j["key"]]["t"].numel(), dtype=torch.bool, device=fk.device)
    for p in j["preds"]:
        keep &= _cmp(d[p["col"]]["t"], p["op"], p["args"])
    subs = []
    for s in j.get("joins", []):
        m, pay = _lookup(tables, s, d[s["fk"]]["t"])
        keep &= m
        subs.append(pay)
    pay = [subs[c["join"]][c["field"]] if isinstance(c, dict) else d[c]["t"] for c in j["payload"]]
    keys, order = torch.sort(d[j["key"]]["t"])
    at = torch.clamp(torch.searchsorted(keys, fk), max=keys.numel() - 1)
    row = order[at]
    return (keys[at] == fk) & keep[row], [p[row] for p in pay]


def _answer(tables, q):
    fact = tables["fact"]
    n = next(iter(c["t"].numel() for c in fact.values() if "t" in c))
    ok = torch.ones(n, dtype=torch.bool, device=DEV)
    for p in q["preds"]:
        c = fact[p["col"]]
        ok &= _matches(c, p["op"], p["args"][0]) if "bytes" in c else _cmp(c["t"], p["op"], p["args"])
    pays = []
    for j in q["joins"]:
        m, pay = _lookup(tables, j, fact[j["fk"]]["t"])
        ok &= m
        pays.append(pay)
    rows = torch.nonzero(ok)[:, 0]
    keys = [(fact[k["col"]]["t"] if "col" in k else pays[k["join"]][k["field"]])[rows] for k in q["group"]]
    aggs = []
    for a in q["aggs"]:
        v = [fact[c]["t"][rows].long() for c in a.get("cols", [])]
        aggs.append(torch.ones(rows.numel(), dtype=torch.int64, device=DEV) if a["op"] == "count"
                    else v[0] * v[1] if a["op"] == "sum_mul" else v[0])
    return _group(keys, aggs)


def exact(case, seed):
    if case["family"] == "load":
        return None                        # page bytes: a format, not numbers computed
    got = [_answer(t, q) for t, q in _tables(case, seed)]
    room = _room(case)
    if case["call"] == "noalloc":
        out = np.zeros((room[0], 6), np.int64)
        out[:len(got[0])] = np.ascontiguousarray(got[0]).view(np.int64).reshape(-1, 6)
        return {"count": np.array([len(got[0])], np.int32), "records": out}
    return _records(room, got)
