// How a launch's queries are cut into tickets (ranges of rows, each processed
// by one warp) and how the tickets are shared out.
#include <algorithm>
#include <cmath>

#include "kernels.h"

namespace dpf {

namespace {

uint64_t round_up(uint64_t x, uint64_t m) { return (x + m - 1) / m * m; }

double read_part(const ScanShare& S) { return std::max(S.live, 0.125); }

// One query: owned tickets of `big` rows, then pool tickets of `small` rows
// over at least its last `tail` rows (none: tail == 0).
void cut(DevQuery& Q, uint64_t rows, uint64_t big, uint64_t small, uint64_t tail) {
  Q.chunk_rows = uint32_t(big);
  Q.page_tickets = 0;
  if (tail == 0 || small >= big) {
    Q.tail_first = Q.nchunks = (rows + big - 1) / big;
    Q.tail_row = rows;
    Q.tail_rows = uint32_t(big);
    return;
  }
  Q.tail_first = (rows - std::min(rows, tail)) / big;
  Q.tail_row = Q.tail_first * big;
  Q.tail_rows = uint32_t(small);
  Q.nchunks = Q.tail_first + (rows - Q.tail_row + small - 1) / small;
}

// One ticket per warp, of about per_warp rows.  A ticket that crosses a page
// is two runs of tiles, one after the other, which costs about as long as 256
// more rows of a star join or scan (a scan of 1 M rows: 17 against 14 us; a star
// of 4.1 M rows in pages of 4,096: 35 against 30), fewer of a dearer query; so
// when a page's equal tickets are not much larger than that, none crosses a
// page.
void cut_once(DevQuery& Q, const ScanShare& S, uint64_t per_warp, uint64_t warps) {
  const uint64_t P = Q.page_rows, big = round_up(per_warp, kMB);
  cut(Q, S.rows, big, 0, 0);
  if (big >= P) return;
  for (uint64_t per = (P + big - 1) / big; per > 0; --per) {
    const uint64_t rows = round_up((P + per - 1) / per, kMB), n = (P + rows - 1) / rows;  // n <= per tickets a page
    if (double(rows) > double(big) + std::min(256.0, 320.0 / S.cost)) return;
    const uint64_t count = S.rows / P * n + (S.rows % P + rows - 1) / rows;
    if (count > std::max(warps, Q.nchunks)) continue;
    Q.chunk_rows = uint32_t(rows);
    Q.page_tickets = uint32_t(n);
    Q.tail_first = Q.nchunks = count;
    Q.tail_rows = uint32_t(rows);
    return;
  }
}

}  // namespace

// How long a warp takes for a ticket is set by chains of dependent loads more
// than by its rows, so a launch is fastest when every warp gets the same few
// tickets.  The rows are those from the first to the last page that the first
// step's range meets (ScanShare): of a table sorted by the column of a range,
// all that is read and nothing else, which is what makes equal shares equal.
//  - A query of at most chunk_rows rows per warp is cut into one ticket per
//    warp (whole mini blocks); there is no pool.  Rows of skipped pages between
//    those read do not count (ScanShare::live): a table of which a seventh is
//    read has seven tickets per warp, eight at most, as a ticket that skips
//    its page costs a load too.
//  - A larger one into equal tickets of at most chunk_rows, the same number
//    for every warp, and a pool of two 512-row tickets per warp, which even
//    out the warps' different speeds.  When whole tickets of chunk_rows leave
//    about as much (512 rows a warp, half a ticket at most), the tickets are
//    whole and the rest is the pool: of 4,096 rows, sixteen make a page, and a
//    ticket is one run of tiles and one survivor list (chain of 67 M rows 323 ->
//    307 us, star 194 -> 184).
//  - A batch is cut into tickets of about equal cost, the same number for every
//    warp, all owned, in runs: a CTA that changes its query flushes it, meets
//    and loads the next one's tables, which a pool drawn in query order makes
//    every CTA do (24 queries of up to 4 M rows: 148 us, with a fifth of the
//    rows in a pool 220).  What the estimates miss is taken over from CTAs that
//    have most left (draw_batch; without it 32 queries over a year of 8 M rows
//    1,380 us, with it 690).  A ticket costs at most what 4,096 rows of a star
//    join do, and has at most kBatchRows rows, as little as a meeting waits for:
//    of 1,024, 2,048 and 4,096 rows 64 queries of up to 24 M rows take 1,150,
//    1,060 and 1,080 us, the 24 queries 147, 148 and 195, the 32 676, 695 and
//    785, 12 star joins of 6 to 11 M rows 500, 410 and 397.
//  - A batch of large queries (kInOrderRows each on average) is drawn whole
//    from the pool, query by query, each query's last rows in small tickets:
//    the CTAs' meetings at its few switches cost little and no estimate of a
//    query's cost is needed (16 queries over 67 M rows: 3.6 ms, in owned runs
//    5.8).
void layout_tickets(DevQuery* Q, const ScanShare* S, int n, uint64_t warps, uint32_t chunk_rows, uint64_t* begin) {
  constexpr uint64_t kInOrderRows = uint64_t(1) << 24, kBatchRows = 2048;
  const uint64_t tile = kMbPerWarpTile * kMB, chunk = chunk_rows;
  uint64_t all = 0;
  for (int i = 0; i < n; ++i) {
    Q[i].row0 = S[i].row0;
    all += S[i].rows;
  }
  const bool in_order = n > 1 && all / uint64_t(n) >= kInOrderRows;
  if (in_order) {
    const uint64_t small = std::max<uint64_t>(tile, chunk / 8 / tile * tile);
    uint64_t want = 2 * warps * small;  // from the last query backwards
    for (int i = n - 1; i >= 0; --i) {
      const uint64_t rows = std::min(S[i].rows, want);
      want -= rows;
      cut(Q[i], S[i].rows, chunk, small, std::max(rows, std::min(S[i].rows, warps * small)));
    }
  } else if (n == 1) {
    const uint64_t read = std::max<uint64_t>(1, uint64_t(double(S->rows) * read_part(*S)));
    const uint64_t per_warp = (read + warps - 1) / warps, pool = 2 * tile;
    if (per_warp <= std::max(chunk, pool)) {
      cut_once(*Q, *S, std::min(per_warp, chunk), warps);
    } else {
      const uint64_t whole = per_warp / chunk * chunk, rest = per_warp - whole;
      if (rest >= tile && rest <= chunk / 2) {
        cut(*Q, S->rows, chunk, rest > pool ? pool : tile, uint64_t(double(S->rows) * double(rest) / double(per_warp)));
      } else {
        const uint64_t own = per_warp - pool, k = (own + chunk - 1) / chunk;
        cut(*Q, S->rows, round_up((own + k - 1) / k, tile), tile, warps * pool);
      }
    }
  } else {
    double total = 0;
    for (int i = 0; i < n; ++i) total += double(S[i].rows) * read_part(S[i]) * S[i].cost;
    const double per_warp = total / double(warps);
    const double k = std::max(1.0, std::ceil(per_warp / double(kDefaultChunkRows)));
    for (int i = 0; i < n; ++i) {
      const double c = std::max(0.25, S[i].cost);
      const uint64_t big = std::min(std::min(chunk, kBatchRows), round_up(uint64_t(per_warp / k / c) + 1, kMB));
      cut(Q[i], S[i].rows, big, 0, 0);
    }
  }
  uint64_t owned = 0, pool = 0;
  for (int i = 0; i < n; ++i) {
    begin[i] = owned;
    begin[n + 1 + i] = pool;
    if (!in_order) owned += Q[i].tail_first;
    pool += Q[i].nchunks - (in_order ? 0 : Q[i].tail_first);
  }
  begin[n] = owned;
  begin[2 * n + 1] = pool;
}

}  // namespace dpf
