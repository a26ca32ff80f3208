"""GPU parity of the cooperative string search (CONTAINS, general LIKE) at the
edges of its pieces: 16-byte chunks that start inside a mini block, strings
longer than a search window (4,096 bytes), matches that end at a row's end or
would cross into the next row, empty strings, patterns of 1, 4, 5 and 32
bytes, literal bytes behind FSST escapes (0xff among them), rows that all are
LIKE candidates (the queue of 32 fills and drains), ragged page tails."""

import numpy as np
import pytest

import oracle
import paper_2605_10511_gb300 as dpf

pytestmark = pytest.mark.gpu


def _strings(kind, rows, rng):
    if kind == "runs":        # one letter, many matches, matches at row ends
        return [b"a" * int(n) for n in rng.integers(0, 40, rows)]
    if kind == "escapes":     # bytes of every value: most are escaped on FSST pages
        return [rng.integers(0, 256, int(n), dtype=np.uint8).tobytes() + b"\xff" * int(n % 5)
                for n in rng.integers(0, 30, rows)]
    if kind == "long":        # beyond one search window
        return [bytes(rng.integers(97, 101, int(n), dtype=np.uint8)) for n in rng.integers(0, 9000, rows)]
    return [b"xyab"[:int(n % 5)] + b"cd" * int(n % 3) + b"ab" * int(n % 2) for n in rng.integers(0, 60, rows)]


def _workload(kind, rows, page_rows, codec, seed):
    rng = np.random.default_rng(seed)
    s = _strings(kind, rows, rng)
    off = np.zeros(rows + 1, np.uint64)
    off[1:] = np.cumsum([len(x) for x in s])
    data = np.frombuffer(b"".join(s) or b"\0", np.uint8)
    cols = {"s": {"codec": codec, "bytes": data, "offsets": off},
            "m": {"codec": "for", "values": rng.integers(1, 1000, rows).astype(np.int32)}}
    return {"name": f"search_{kind}_{codec}_{rows}_{page_rows}", "fact": "f",
            "tables": {"f": {"rows": rows, "page_rows": page_rows, "cols": cols}},
            "query": {"preds": [], "joins": [], "group": [], "aggs": [{"op": "count"}, {"op": "sum", "cols": ["m"]}]}}, s


@pytest.mark.parametrize("keys", [20_000, 75_000, 81_000])
@pytest.mark.parametrize("codec,op,pat", [("str", "contains", b"abcd"), ("fsst", "contains", b"cdab"), ("str", "like", b"%ab%c_%")])
def test_search_beside_shared_memory_tables(codec, op, pat, keys):
    """Join tables placed in shared memory until it is full (81,000 keys of two
    bytes are within the accumulators' and lists' budget and not within what the
    search's scratch leaves: that table is probed in device memory)."""
    w, s = _workload("short", 6007, 4096, codec, keys)
    rng = np.random.default_rng(keys)
    dim = {"k": {"codec": "for", "values": rng.permutation(keys).astype(np.int32) + 1},
           "p": {"codec": "dict", "values": (np.arange(keys) % 1024).astype(np.int32)}}
    w["tables"]["d"] = {"rows": keys, "page_rows": 4096, "cols": dim}
    w["tables"]["f"]["cols"]["fk"] = {"codec": "for", "values": rng.integers(1, keys + 1, len(s)).astype(np.int32)}
    w["name"] += f"_smem_{op}"
    w["query"] = {"preds": [{"col": "s", "op": op, "args": [pat]}], "group": [{"join": 0, "field": 0}],
                  "joins": [{"fk": "fk", "dim": "d", "key": "k", "preds": [], "payload": ["p"]}],
                  "aggs": [{"op": "count"}, {"op": "sum", "cols": ["m"]}, {"op": "sum_mul", "cols": ["m", "m"]}]}
    want = oracle.run_query(w, from_encoded=False)
    e = dpf.Engine(device=0)
    try:
        for threads in (128, 256):
            got = e.run(w, tuning=dpf.Tuning(0, threads, dpf.HT_PLACE["smem"], 0, 0, 0))
            assert got.shape == want.shape and all(np.array_equal(got[f], want[f]) for f in ("key", "count", "val"))
    finally:
        e.close()


@pytest.mark.parametrize("codec,op,pat", [("str", "contains", b"abcda"), ("fsst", "contains", b"cd"), ("str", "like", b"%cd_b%"),
                                          ("fsst", "contains", b"\xff")])
@pytest.mark.parametrize("kind,rows,page_rows", [("escapes", 2500, 128), ("long", 389, 256), ("short", 70_003, 65536)])
def test_search_over_host_resident_pages(kind, rows, page_rows, codec, op, pat):
    w, _ = _workload(kind, rows, page_rows, codec, rows + 2)
    w["query"]["preds"] = [{"col": "s", "op": op, "args": [pat]}]
    want = oracle.run_query(w, from_encoded=False)
    e = dpf.Engine(device=0)
    try:
        e.load_workload(w, fact_placement="host")
        got = e.run(w)
        assert np.array_equal(got["count"], want["count"]) and np.array_equal(got["val"], want["val"])
    finally:
        e.close()


def _lengths(bits, rows, rng):
    """Lengths whose fields take `bits` bits, most of them at the largest."""
    top = 2**bits - 1
    n = np.where(rng.random(rows) < 0.9, top, rng.integers(0, top, rows))
    n[::128] = 0
    n[1::128] = top
    return n


@pytest.mark.parametrize("bits", [10, 11, 12])
@pytest.mark.parametrize("codec", ["str", "fsst"])
def test_starts_of_strings_with_wide_length_fields(bits, codec):
    """Mini blocks whose length fields have 11 bits (summed two to a register)
    and 12 (one), at their largest in every row."""
    rng = np.random.default_rng(bits)
    rows = 700
    n = _lengths(bits, rows, rng)
    s = [bytes(rng.integers(97, 123, int(k), dtype=np.uint8)) for k in n]
    s = [x[:-4] + b"%03dz" % (i % 1000) if len(x) > 8 else x for i, x in enumerate(s)]
    off = np.zeros(rows + 1, np.uint64)
    off[1:] = np.cumsum([len(x) for x in s])
    w = {"name": f"wide_{bits}_{codec}", "fact": "f",
         "tables": {"f": {"rows": rows, "page_rows": 256, "cols": {
             "s": {"codec": codec, "bytes": np.frombuffer(b"".join(s), np.uint8), "offsets": off},
             "m": {"codec": "for", "values": np.arange(rows, dtype=np.int32)}}}},
         "query": {"preds": [], "joins": [], "group": [], "aggs": [{"op": "sum", "cols": ["m"]}]}}
    e = dpf.Engine(device=0)
    try:
        for pat in [b"%03dz" % i for i in (0, 5, 126, 127, 128, 255, 511, 699)] + [b"00z"]:
            got = e.run(dict(w, query=dict(w["query"], preds=[{"col": "s", "op": "contains", "args": [pat]}])))
            hit = [i for i, x in enumerate(s) if pat in x]
            assert int(got["count"][0]) == len(hit) and int(got["val"][0, 0]) == sum(hit), pat
    finally:
        e.close()


@pytest.mark.parametrize("codec", ["str", "fsst"])
@pytest.mark.parametrize("kind,rows,page_rows", [("runs", 3001, 1024), ("escapes", 2500, 128), ("long", 389, 256),
                                                 ("short", 5003, 4096), ("short", 1, 128)])
def test_contains_at_the_edges(kind, rows, page_rows, codec):
    w, s = _workload(kind, rows, page_rows, codec, rows)
    pats = [b"a", b"ab", b"abcd", b"cdab", b"abcda", b"\xff", b"\xff\xff\xff", b"a" * 32]
    pats += [x[i:i + n] for x in s[:40] for i, n in ((0, 4), (3, 9), (max(0, len(x) - 5), 5)) if len(x) > i][:12]
    e = dpf.Engine(device=0)
    try:
        for pat in pats:
            q = dict(w, query=dict(w["query"], preds=[{"col": "s", "op": "contains", "args": [pat]}]))
            got, want = e.run(q), oracle.run_query(q, from_encoded=False)
            hits = sum(pat in x for x in s)
            assert (int(got["count"].sum()) if len(got) else 0) == hits, (kind, codec, pat)
            assert np.array_equal(got["val"], want["val"]), (kind, codec, pat)
    finally:
        e.close()


@pytest.mark.parametrize("kind,rows,page_rows", [("runs", 3001, 1024), ("long", 200, 128), ("short", 5003, 4096)])
def test_like_at_the_edges(kind, rows, page_rows):
    w, _ = _workload(kind, rows, page_rows, "str", rows + 1)
    e = dpf.Engine(device=0)
    try:
        for pat in (b"%a_a%", b"_%_", b"%ab%cd%", b"a%a", b"%_", b"%cd_b%", b"x%b", b"%aaaa_aaaa%aa"):
            q = dict(w, query=dict(w["query"], preds=[{"col": "s", "op": "like", "args": [pat]}]))
            got, want = e.run(q), oracle.run_query(q, from_encoded=False)
            assert np.array_equal(got["count"], want["count"]) and np.array_equal(got["val"], want["val"]), (kind, pat)
    finally:
        e.close()
