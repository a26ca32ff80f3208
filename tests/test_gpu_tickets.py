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
