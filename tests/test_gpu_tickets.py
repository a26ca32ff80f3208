"""Every row is counted once whatever the ticket layout: tables around one
mini block, one mini block per resident warp, one whole ticket per warp, the
size from which the 1,024-thread build runs, and batches of very uneven
queries; sums whose low 32 bits carry many times, in both directions."""

import numpy as np
import pytest

import paper_2605_10511_gb300 as dpf

pytestmark = pytest.mark.gpu

WARPS = 152 * 3 * 8


def _table(rows, page_rows, seed):
    rng = np.random.default_rng(seed)
    v = rng.integers(-2**31, 2**31, rows, dtype=np.int64).astype(np.int32)
    g = (np.arange(rows) % 7).astype(np.int32)
    return {"name": f"tickets_{rows}_{page_rows}_{seed}", "fact": "f",
            "tables": {"f": {"rows": rows, "page_rows": page_rows, "cols": {
                "v": {"codec": "for", "values": v}, "g": {"codec": "dict", "values": g}}}},
            "query": {"preds": [], "joins": [], "group": [{"col": "g"}],
                      "aggs": [{"op": "count"}, {"op": "sum", "cols": ["v"]}, {"op": "sum_mul", "cols": ["v", "v"]}]}}, v, g


def _check(rec, v, g, what):
    w = v.astype(np.int64)
    for r in rec:
        m = g == r["key"][0]
        assert r["count"] == r["val"][0] == int(m.sum()), what
        assert r["val"][1] == int(w[m].sum()), what
        with np.errstate(over="ignore"):
            assert r["val"][2] == int((w[m] * w[m]).sum()), what  # wraps modulo 2^64 in both
    assert len(rec) == len(np.unique(g)), what


@pytest.mark.parametrize("page_rows", [1024, 65536])
@pytest.mark.parametrize("rows", [1, 127, 128, 129, WARPS * 128 - 1, WARPS * 128 + 1, 2**23 - 1, 2**23 + 1,
                                  WARPS * 4096, WARPS * 4096 + 1])
def test_rows_around_the_ticket_sizes(rows, page_rows):
    w, v, g = _table(rows, page_rows, rows % 1000)
    e = dpf.Engine(device=0)
    try:
        for t in (None, dpf.Tuning(512, 0, 0, 0, 0, 0), dpf.Tuning(4096, 256, 0, 4, 0, 0)):
            _check(e.run(w, tuning=t), v, g, (rows, page_rows, t and t.chunk_rows))
    finally:
        e.close()


def _clustered(rows, page_rows, seed):
    """A table sorted by day, a year of which is asked for: pages at both ends
    are skipped, and (days scattered over a second column) some in between."""
    rng = np.random.default_rng(seed)
    day = np.sort(rng.integers(0, 2000, rows)).astype(np.int32)
    g = rng.integers(0, 7, rows).astype(np.int32)
    v = rng.integers(-2**31, 2**31, rows, dtype=np.int64).astype(np.int32)
    d0 = int(rng.integers(0, 1700))
    w = {"name": f"year_{rows}_{page_rows}_{seed}", "fact": "f",
         "tables": {"f": {"rows": rows, "page_rows": page_rows, "cols": {
             "day": {"codec": "for", "values": day}, "v": {"codec": "for", "values": v}, "g": {"codec": "dict", "values": g}}}},
         "query": {"preds": [{"col": "day", "op": "between", "args": [d0, d0 + 285]}], "joins": [], "group": [{"col": "g"}],
                   "aggs": [{"op": "count"}, {"op": "sum", "cols": ["v"]}, {"op": "sum_mul", "cols": ["v", "v"]}]}}
    keep = (day >= d0) & (day <= d0 + 285)
    return w, v[keep], g[keep]


@pytest.mark.parametrize("tuning", [None, (1024, 256, 0, 0, 0, 0), (4096, 1024, 0, 1, 0, 0), (65536, 128, 0, 0, 0, 0)])
def test_batch_of_queries_that_skip_pages(tuning):
    """Tables of which a seventh is read, one of which nothing is, one read
    whole, and one whose pages are read here and there; every ticket size."""
    e = dpf.Engine(device=0)
    try:
        tabs = [_clustered(n, p, n % 89) for n, p in ((1_000_003, 1024), (300_000, 4096), (2_500_001, 65536), (999, 128),
                                                      (700_000, 8192))]
        w, v, g = _table(400_001, 4096, 3)
        tabs.append((w, v, g))
        w, v, g = _clustered(500_009, 4096, 5)
        w = dict(w, name="none", query=dict(w["query"], preds=[{"col": "day", "op": "gt", "args": [5000]}]))
        tabs.append((w, v[:0], g[:0]))
        rng = np.random.default_rng(8)
        page = rng.permutation(np.arange(250) % 10).astype(np.int32)          # one page in ten matches
        a = np.repeat(page, 1024)
        v, g = rng.integers(-99, 99, a.size).astype(np.int32), (np.arange(a.size) % 7).astype(np.int32)
        w = {"name": "scattered", "fact": "f", "tables": {"f": {"rows": a.size, "page_rows": 1024, "cols": {
            "a": {"codec": "for", "values": a}, "v": {"codec": "for", "values": v}, "g": {"codec": "dict", "values": g}}}},
            "query": {"preds": [{"col": "a", "op": "eq", "args": [3]}], "joins": [], "group": [{"col": "g"}],
                      "aggs": [{"op": "count"}, {"op": "sum", "cols": ["v"]}, {"op": "sum_mul", "cols": ["v", "v"]}]}}
        tabs.append((w, v[a == 3], g[a == 3]))
        for w, _, _ in tabs:
            e.load_workload(w)
        t = dpf.Tuning(*tuning) if tuning else None
        for sel in (range(len(tabs)), [0], [6], [7], [6, 6], [2, 7, 5]):
            prep = e.ctx.prepare([e.plan(tabs[i][0]) for i in sel], t)
            for _ in range(3):
                e.ctx.launch(prep)
                for k, i in enumerate(sel):
                    _check(e.ctx.read_result(prep, k), tabs[i][1], tabs[i][2], (tabs[i][0]["name"], list(sel)))
            e.ctx.release(prep)
    finally:
        e.close()


def test_batch_of_large_queries_in_order():
    """At least 2^24 rows a query on average: every ticket is in the pool."""
    e = dpf.Engine(device=0)
    try:
        tabs = [_table(n, 65536, n % 97) for n in (2**25 + 12_345, 3_000_001, 2**24 - 1)]
        for w, _, _ in tabs:
            e.load_workload(w)
        prep = e.ctx.prepare([e.plan(w) for w, _, _ in tabs])
        for _ in range(2):
            e.ctx.launch(prep)
            for i, (w, v, g) in enumerate(tabs):
                _check(e.ctx.read_result(prep, i), v, g, w["name"])
        e.ctx.release(prep)
    finally:
        e.close()


def test_what_a_batch_was_prepared_with_prepares_it_again():
    """The tuning that a batch reports, open fields filled in, is one that the
    library takes and that prepares the same launch."""
    e = dpf.Engine(device=0)
    try:
        w, v, g = _table(600_001, 8192, 4)
        e.load_workload(w)
        for n in (1, 3):
            prep = e.ctx.prepare([e.plan(w)] * n)
            t = e.ctx.prep_tuning(prep)
            again = e.ctx.prepare([e.plan(w)] * n, dpf.Tuning(*t.values()))
            assert e.ctx.prep_tuning(again) == t
            e.ctx.launch(again)
            _check(e.ctx.read_result(again, n - 1), v, g, n)
            for p in (prep, again):
                e.ctx.release(p)
    finally:
        e.close()


def test_uneven_batch():
    e = dpf.Engine(device=0)
    try:
        tabs = [_table(n, 4096, n % 97) for n in (1, 130, 5000, 1_000_003, 77, 300_000, 4_000_000, 128)]
        for w, _, _ in tabs:
            e.load_workload(w)
        prep = e.ctx.prepare([e.plan(w) for w, _, _ in tabs])
        for _ in range(2):
            e.ctx.launch(prep)
            for i, (w, v, g) in enumerate(tabs):
                _check(e.ctx.read_result(prep, i), v, g, w["name"])
        e.ctx.release(prep)
    finally:
        e.close()
