"""Ticket layouts (csrc/tickets.cpp) as a pure function: every ticket of every
query is drawn once, and the tickets' rows cover what a launch reads of each
table once, over odd sizes, named ticket sizes, tables of which only some pages
are read, and batches; and no CTA owns much more than an even share."""

import ctypes as C
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_10511_gb300", "csrc")
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))),
                    "include")
SOURCE = r"""
#include <cstring>
#include <vector>
#include "kernels.h"
using namespace dpf;
// in[i] = {nrows, page_rows, row0, rows}, share[i] = {live, cost}; begin: 2 n + 2
// out; counts[i] = tickets; then rows(): first and last row of one ticket.
static std::vector<DevQuery> qs;
extern "C" void layout(int n, const uint64_t (*in)[4], const double (*share)[2], uint64_t warps, uint32_t chunk,
                      uint64_t* begin, uint64_t* counts) {
  qs.assign(n, DevQuery());
  std::vector<ScanShare> s(n);
  for (int i = 0; i < n; ++i) {
    std::memset(&qs[i], 0, sizeof(DevQuery));
    qs[i].nrows = in[i][0];
    qs[i].page_rows = uint32_t(in[i][1]);
    s[i] = ScanShare{in[i][2], in[i][3], share[i][0], share[i][1]};
  }
  layout_tickets(qs.data(), s.data(), n, warps, chunk, begin);
  for (int i = 0; i < n; ++i) counts[i] = qs[i].nchunks;
}
extern "C" void rows(int i, uint64_t t0, uint64_t n, uint64_t* out) {
  for (uint64_t k = 0; k < n; ++k) ticket_rows(qs[i], t0 + k, out + 2 * k, out + 2 * k + 1);
}
extern "C" uint64_t owned_of(int i) { return qs[i].tail_first; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tickets")
    src, out = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    cmd = ["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{CUDA}", f"-I{CSRC}", src, os.path.join(CSRC, "tickets.cpp"),
           "-o", out]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    so = C.CDLL(out)
    so.owned_of.restype = C.c_uint64
    return so


def _layout(lib, queries, warps, chunk):
    """queries: (nrows, page_rows, row0, rows, live, cost) each.  Returns
    (begin, per query an array of ticket [first, last) rows)."""
    n = len(queries)
    a = np.array([q[:4] for q in queries], np.uint64)
    s = np.array([q[4:] for q in queries], np.float64)
    begin, counts = np.zeros(2 * n + 2, np.uint64), np.zeros(n, np.uint64)
    p = lambda x: x.ctypes.data_as(C.c_void_p)
    lib.layout(n, p(a), p(s), C.c_uint64(warps), C.c_uint32(chunk), p(begin), p(counts))
    out = []
    for i in range(n):
        r = np.zeros((int(counts[i]), 2), np.uint64)
        lib.rows(i, C.c_uint64(0), C.c_uint64(int(counts[i])), p(r))
        out.append(r.astype(np.int64))
    return begin.astype(np.int64), out


def _query(rng, nrows, page_rows):
    npages = -(-nrows // page_rows)
    first = rng.randrange(npages) if rng.random() < 0.5 else 0
    last = rng.randrange(first, npages)
    if rng.random() < 0.4:
        first, last = 0, npages - 1
    rows = min(nrows, (last + 1) * page_rows) - first * page_rows
    if rng.random() < 0.1:
        return nrows, page_rows, 0, 1, 0.0, rng.uniform(0.25, 10)   # no page is read
    return nrows, page_rows, first * page_rows, rows, rng.choice([1.0, 1.0, 0.9, 0.5, 0.01]), rng.uniform(0.25, 10)


def _check(lib, queries, warps, chunk):
    begin, tickets = _layout(lib, queries, warps, chunk)
    n = len(queries)
    assert begin[0] == begin[n + 1] == 0
    for i, (nrows, page_rows, row0, rows, _, _) in enumerate(queries):
        t = tickets[i]
        owned, pool = begin[i + 1] - begin[i], begin[n + 2 + i] - begin[n + 1 + i]
        assert owned >= 0 and pool >= 0 and owned + pool == len(t) >= 1
        # a draw maps an owned index to itself and a pool index behind the owned ones
        assert owned in (0, int(lib.owned_of(i)))
        size = t[:, 1] - t[:, 0]
        assert (size > 0).all() and size.max() <= max(chunk, 128)
        assert (t[:, 0] % 128 == 0).all() and t[0, 0] == row0
        assert (t[1:, 0] == t[:-1, 1]).all()                       # one after the other, none twice
        assert t[-1, 1] >= row0 + rows and t[-1, 0] < row0 + rows and t[-1, 1] <= nrows
        assert (((t[:, 1] % 128) == 0) | (t[:, 1] == nrows)).all()
    return begin, tickets


@pytest.mark.parametrize("n", [1, 2, 5, 40])
def test_every_row_is_in_one_ticket(lib, n):
    rng = random.Random(n)
    for case in range(120 if n < 40 else 12):
        warps = rng.choice([8, 3648, 4864])
        chunk = rng.choice([512, 1024, 4096, 4096, 65536])
        hi = 17 if warps == 8 else 25
        qs = [_query(rng, max(1, int(2 ** rng.uniform(0, hi)) + rng.randrange(3) - 1), rng.choice([128, 4096, 8192, 65536]))
              for _ in range(n)]
        _check(lib, qs, warps, chunk)


def test_sizes_around_the_edges(lib):
    for warps in (8, 3648):
        for nrows in (1, 127, 128, 129, warps * 128 - 1, warps * 128, warps * 128 + 1, warps * 4096 - 1, warps * 4096,
                      warps * 4096 + 1, warps * 5120, warps * 5121, warps * 4096 * 3 + 7):
            for page_rows in (128, 8192, 65536):
                _check(lib, [(nrows, page_rows, 0, nrows, 1.0, 1.0)], warps, 4096)


def test_large_queries_of_a_batch_are_drawn_in_order(lib):
    qs = [(1 << 25, 65536, 0, 1 << 25, 1.0, 1.0), ((1 << 24) + 77, 8192, 0, (1 << 24) + 77, 1.0, 3.0)]
    begin, _ = _check(lib, qs, 3648, 4096)
    assert begin[2] == 0                                            # nothing owned


@pytest.mark.parametrize("chunk", [1024, 2048, 4096, 65536])
@pytest.mark.parametrize("ctas,warps", [(456, 8), (152, 32)])
def test_no_cta_owns_more_than_its_share_of_the_rows_read(lib, ctas, warps, chunk):
    """Queries over a seventh of a sorted table each, whatever the ticket size
    that is named: every CTA's run of owned tickets reads an even share."""
    qs = [(8_000_000 + 1000 * i, 65536, (i % 7) * 17 * 65536, 18 * 65536, 1.0, 1.0) for i in range(32)]
    begin, tickets = _check(lib, qs, ctas * warps, chunk)
    owned = np.concatenate([t[:int(lib.owned_of(i))] for i, t in enumerate(tickets)])
    assert len(owned) == begin[32] > 0
    rows = np.zeros(ctas)
    for b in range(ctas):
        a, e = len(owned) * b // ctas, len(owned) * (b + 1) // ctas
        rows[b] = (owned[a:e, 1] - owned[a:e, 0]).sum()
    even = sum(q[3] for q in qs) / ctas
    assert len(owned) == sum(len(t) for t in tickets) and rows.max() <= even + chunk
