"""Columns that a load encodes on the device have the pages that the host
encoder writes, byte for byte: every such codec, widths from 0 to full,
negative and wrapping values, ragged page tails, string offsets that start
above 0, empty strings; and what the encoder refuses is still refused."""

import numpy as np
import pytest

import paper_2605_10511_gb300 as dpf

pytestmark = pytest.mark.gpu


def _columns(n, rng):
    spans = [(5, 5), (-3, 4), (900, 105001), (-2**31, 2**31 - 1), (2**31 - 2, 2**31 - 1)]
    for lo, hi in spans:
        v = rng.integers(lo, hi, n, endpoint=True).astype(np.int32)
        yield {"codec": "for", "values": v}
        yield {"codec": "delta", "values": v if lo == -3 else np.sort(v)}
    vals = rng.integers(-30000, 30000, int(rng.integers(1, 3000))).astype(np.int32)
    yield {"codec": "dict", "values": vals[rng.integers(0, vals.size, n)]}
    yield {"codec": "dict", "values": (vals[rng.integers(0, vals.size, n)] * 70000).astype(np.int32)}  # a wide range
    for lo, hi in [(7, 7), (-5, 5), (-2**40, 2**40), (-2**63, 2**63 - 1)]:
        yield {"codec": "for64", "values": rng.integers(lo, hi, n, dtype=np.int64, endpoint=True)}
    for top in (1, 2, 45, 300):
        off = np.zeros(n + 1, np.uint64)
        off[1:] = np.cumsum(rng.integers(0, top, n).astype(np.uint64))
        off += np.uint64(top % 7)
        yield {"codec": "str", "bytes": rng.integers(0, 256, int(off[-1]) + 3, dtype=np.uint8), "offsets": off}


@pytest.mark.parametrize("n", [1023, 1024, 1025, 16383, 16384, 16385, 100_003])
@pytest.mark.parametrize("page_rows", [128, 4096, 65536])
def test_pages_equal_the_host_encoders(n, page_rows):
    rng = np.random.default_rng(n + page_rows)
    with dpf.Context(0) as ctx:
        base = ctx.memory_used()
        for col in _columns(n, rng):
            enc = dpf.encode_column(col, page_rows)
            cid = ctx.load_column(col, table=1, page_rows=page_rows)
            assert np.array_equal(ctx.column_bytes(cid), enc["blob"]), (col["codec"], n, page_rows)
            host = ctx.load_encoded(enc, table=1)
            assert ctx.column_info(cid) == ctx.column_info(host), col["codec"]
            ctx.drop_column(host)
            ctx.drop_column(cid)
        assert ctx.memory_used() == base


def test_a_load_gives_its_raw_values_back():
    """Half a GB of values that encode to 8 MB: what a load leaves allocated is the
    pages and at most 256 MiB of blocks for the next one."""
    import torch
    n = 1 << 27
    with dpf.Context(0) as ctx:
        ctx.load_column({"codec": "for", "values": np.arange(20_000, dtype=np.int32)}, table=1)
        free = torch.cuda.mem_get_info(0)[0]
        for _ in range(2):
            cid = ctx.load_column({"codec": "for", "values": np.zeros(n, np.int32)}, table=2)
            assert ctx.column_info(cid)["encoded_bytes"] < 16 << 20
            assert free - torch.cuda.mem_get_info(0)[0] <= 300 << 20
        for _ in range(2):   # small ones are kept
            ctx.load_column({"codec": "for64", "values": np.arange(1 << 20, dtype=np.int64)}, table=3)
        assert free - torch.cuda.mem_get_info(0)[0] <= 300 << 20


def _workload(enc_cols, page_rows, n, preds, group, name):
    return {"name": name, "fact": "f", "tables": {"f": {"rows": n, "page_rows": page_rows, "cols": enc_cols}},
            "query": {"preds": preds, "joins": [], "group": group, "aggs": [{"op": "count"}, {"op": "sum", "cols": ["m"]}]}}


@pytest.mark.parametrize("codec,page_rows", [("for", 1024), ("delta", 4096), ("dict", 1024)])
def test_zones_and_dictionaries_made_on_the_device(codec, page_rows):
    """Ranges that skip most pages, and a group-by over the dictionary, give the
    same records on the column encoded on the device and on the one loaded from
    the host encoder's pages, and those of the values themselves."""
    rng = np.random.default_rng(page_rows)
    n = 50_021
    top = {"for": 2**31 - 1, "delta": 2_000_000_000, "dict": 40_000}[codec]
    v = np.sort(rng.integers(-top, top, n)).astype(np.int32)
    if codec == "dict":
        v = (v // 97 * 97).astype(np.int32)
    if codec == "for":                          # unsorted inside a page, sorted over pages
        for p in range(0, n, page_rows):
            v[p:p + page_rows] = rng.permutation(v[p:p + page_rows])
    m = rng.integers(1, 1000, n).astype(np.int32)
    cols = {"v": {"codec": codec, "values": v}, "m": {"codec": "for", "values": m}}
    lo, hi = int(np.sort(v)[n // 3]), int(np.sort(v)[n // 3 + 700])
    ranges = [(lo, hi), (int(v.min()), int(v.min())), (int(v.max()), int(v.max())), (hi, lo - 1), (-2**31, lo), (int(v[n // 2]),) * 2]
    e = dpf.Engine(device=0)
    try:
        dev = _workload(cols, page_rows, n, [], [], f"dev_{codec}")
        e.load_workload(dev)
        host = _workload(cols, page_rows, n, [], [], f"host_{codec}")
        e.tables[(host["name"], "f")] = 991
        for k, c in cols.items():
            e.cols[(host["name"], "f", k)] = e.ctx.load_encoded(dpf.encode_column(c, page_rows), table=991)
        group = [{"col": "v"}] if codec == "dict" and np.unique(v).size <= 65536 else []
        for a, b in ranges:
            keep = (v >= a) & (v <= b)
            got = []
            for w in (dev, host):
                q = dict(w, query=dict(w["query"], preds=[{"col": "v", "op": "between", "args": [a, b]}], group=group))
                got.append(e.run(q))
            assert got[0].tobytes() == got[1].tobytes(), (codec, a, b)
            assert int(got[0]["count"].sum()) == int(keep.sum()) and int(got[0]["val"][:, 1].sum()) == int(m[keep].sum())
            if group:
                u, c = np.unique(v[keep], return_counts=True)
                assert np.array_equal(got[0]["key"][:, 0], u) and np.array_equal(got[0]["count"], c)
    finally:
        e.close()


def test_refusals_stay():
    off = np.arange(40001, dtype=np.uint64)
    off[100] = 0
    bad = [{"codec": "dict", "values": np.arange(70_000, dtype=np.int32)},
           {"codec": "str", "bytes": np.zeros(50_000, np.uint8), "offsets": off}]
    with dpf.Context(0) as ctx:
        base = ctx.memory_used()
        for col in bad:
            with pytest.raises(dpf.DpfError) as e:
                ctx.load_column(col, table=1)
            assert e.value.status == -1  # DPF_EINVAL
        assert ctx.memory_used() == base
