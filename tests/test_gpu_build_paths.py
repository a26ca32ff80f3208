"""An exactly sized build gives the same table by either path: one pass over
the key column's load-time bounds (no memory budget, a span of at most 2^20
keys) and count + insert (a context with a budget): entries, capacity and the
records of a query that probes it; tables that keep no row, one row, a narrow
key range, spans at the edge, and duplicate keys refused."""

import numpy as np
import pytest

import oracle
import paper_2605_10511_gb300 as dpf

pytestmark = pytest.mark.gpu


def _workload(span, keep, seed):
    rng = np.random.default_rng(seed)
    n = 3000
    keys = np.sort(rng.choice(span, n, replace=False)).astype(np.int32) - 77
    keys[0], keys[-1] = -77, span - 78
    a = np.arange(n, dtype=np.int32)
    fk = keys[rng.integers(0, n, 20_001)] + (rng.integers(0, 5, 20_001) == 0).astype(np.int32)
    cols = {"k": {"codec": "for", "values": keys[rng.permutation(n)]}, "a": {"codec": "for", "values": a},
            "p": {"codec": "dict", "values": (a % 7).astype(np.int32)}}
    lo, hi = keep
    return {"name": f"paths_{span}_{lo}_{hi}", "fact": "f",
            "tables": {"d": {"rows": n, "page_rows": 1024, "cols": cols},
                       "f": {"rows": fk.size, "page_rows": 1024, "cols": {"fk": {"codec": "for", "values": fk.astype(np.int32)}}}},
            "query": {"preds": [], "group": [{"join": 0, "field": 0}], "aggs": [{"op": "count"}],
                      "joins": [{"fk": "fk", "dim": "d", "key": "k", "payload": ["p"],
                                 "preds": [{"col": "a", "op": "between", "args": [lo, hi]}]}]}}


@pytest.mark.parametrize("keep", [(0, 2999), (5, 5), (10, 9), (100, 400)])
@pytest.mark.parametrize("span", [3000, 2**20, 2**20 + 1])
def test_both_paths_give_the_same_table(span, keep):
    w = _workload(span, keep, span % 101)
    want = oracle.run_query(w, from_encoded=False)
    info = []
    for budget in (0, 1 << 30):
        e = dpf.Engine(device=0, hbm_budget=budget)
        try:
            got = e.run(w)
            assert got.shape == want.shape and all(np.array_equal(got[f], want[f]) for f in ("key", "count", "val"))
            info.append(e.ctx.hash_info(e.chain_tables(w)[0]))
        finally:
            e.close()
    assert info[0] == info[1]


@pytest.mark.parametrize("n", [3000, 20_000])  # encoded on the host, and on the device
@pytest.mark.parametrize("asynchronous", [False, True])
def test_delta_keys_that_wrap(n, asynchronous):
    """Keys that run past the largest int32 to the smallest (DELTA adds modulo
    2^32), inside the last mini block: no header names a negative one, and the
    column's bounds are the whole of int32 all the same."""
    at = np.arange(n, dtype=np.int64)
    keys = (2**31 - 3 - 7 * (n - 25) + 7 * at).astype(np.uint32).astype(np.int32)
    assert keys.min() < 0 < keys.max() and -2**31 not in keys
    fk = keys[np.random.default_rng(n).integers(0, n, 9001)]
    w = {"name": f"wrap_{n}_{asynchronous}", "fact": "f",
         "tables": {"d": {"rows": n, "page_rows": 1024, "cols": {"k": {"codec": "delta", "values": keys},
                                                                 "p": {"codec": "dict", "values": (at % 7).astype(np.int32)}}},
                    "f": {"rows": fk.size, "page_rows": 1024, "cols": {"fk": {"codec": "for", "values": fk}}}},
         "query": {"preds": [], "group": [{"join": 0, "field": 0}], "aggs": [{"op": "count"}],
                   "joins": [{"fk": "fk", "dim": "d", "key": "k", "payload": ["p"], "preds": []}]}}
    want = oracle.run_query(w, from_encoded=False)
    e = dpf.Engine(device=0)
    try:
        got = e.run(w, asynchronous=asynchronous)
        assert got.shape == want.shape and all(np.array_equal(got[f], want[f]) for f in ("key", "count", "val"))
    finally:
        e.close()


def test_for_pages_whose_fields_wrap():
    """A mini block of another writer, its base near the largest int32: base +
    field wraps, and every key is found."""
    n = 128
    enc = dpf.encode_column({"codec": "for", "values": 2 * np.arange(n, dtype=np.int32)}, 128)
    enc["blob"][16:20].view(np.int32)[0] = 2**31 - 99
    keys = (2 * np.arange(n, dtype=np.int64) + 2**31 - 99).astype(np.uint32).astype(np.int32)
    assert keys.min() < 0 < keys.max() and -2**31 not in keys
    with dpf.Context(0) as ctx:
        k = ctx.load_encoded(enc, table=1)
        assert ctx.hash_info(ctx.build_hash(k))["entries"] == n


def test_duplicate_keys_are_refused_by_both():
    keys = np.array([1, 5, 9, 5], np.int32)
    for budget in (0, 1 << 30):
        with dpf.Context(0, hbm_budget=budget) as ctx:
            base = ctx.memory_used()
            k = ctx.load_column({"codec": "for", "values": keys}, table=1)
            held = ctx.memory_used()
            with pytest.raises(dpf.DpfError) as e:
                ctx.build_hash(k)
            assert e.value.status == -4  # DPF_EDUPKEY
            assert ctx.memory_used() == held > base
