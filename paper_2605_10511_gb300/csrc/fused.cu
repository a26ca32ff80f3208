// Launch and occupancy of the fused kernel (fused_kernel.cuh): picks one of
// its six builds for a batch and sizes its dynamic shared memory.
#include <algorithm>
#include <cmath>

#include "tile.cuh"

namespace dpf {

cudaError_t fused_lean_launch(const FusedLaunch& L, size_t smem, uint32_t tb, cudaStream_t s);
cudaError_t fused_text_launch(const FusedLaunch& L, size_t smem, uint32_t tb, cudaStream_t s);
cudaError_t fused_host_launch(const FusedLaunch& L, size_t smem, uint32_t tb, cudaStream_t s);
cudaError_t fused_stage_launch(const FusedLaunch& L, size_t smem, uint32_t tb, cudaStream_t s);
cudaError_t fused_wide_launch(const FusedLaunch& L, size_t smem, uint32_t tb, cudaStream_t s);
int fused_wide_occupancy(int threads, size_t smem);
int fused_text_occupancy(int threads, size_t smem, int min_blocks);
int fused_host_occupancy(int threads, size_t smem, int min_blocks);
int fused_stage_occupancy(int threads, size_t smem, int min_blocks);

namespace {

uint64_t round_up(uint64_t x, uint64_t m) { return (x + m - 1) / m * m; }

// Relative cost of one row of a query: the measured times per row of its first
// step (a shared-table probe or an integer
// filter 1, a raw prefix 2, a substring 4, no filter 3: every row is
// aggregated).
double row_cost(const DevQuery& Q) {
  if (Q.nsteps == 0 || Q.steps[0].kind == ST_KEY || Q.steps[0].kind == ST_ALL) return 3.0;
  switch (Q.steps[0].kind) {
    case ST_PREFIX: return 2.0;
    case ST_CONTAINS:
    case ST_LIKE: return 4.0;
    default: return 1.0;
  }
}

double read_part(const DevQuery& Q) { return std::max(double(Q.live), 0.125); }

// One query: owned tickets of `big` rows, then pool tickets of `small` rows
// over at least its last `tail` rows (none: tail == 0).
void cut(DevQuery& Q, uint64_t big, uint64_t small, uint64_t tail) {
  Q.chunk_rows = uint32_t(big);
  Q.page_tickets = 0;
  if (tail == 0 || small >= big) {
    Q.tail_first = Q.nchunks = (Q.nrows + big - 1) / big;
    Q.tail_row = Q.nrows;
    Q.tail_rows = uint32_t(big);
    return;
  }
  Q.tail_first = (Q.nrows - std::min(Q.nrows, tail)) / big;
  Q.tail_row = Q.tail_first * big;
  Q.tail_rows = uint32_t(small);
  Q.nchunks = Q.tail_first + (Q.nrows - Q.tail_row + small - 1) / small;
}

// One ticket per warp, of about per_warp rows.  A ticket that crosses a page
// is two runs of tiles, one after the other, which costs about as long as 256
// more cheap rows (a scan of 1 M rows: 17 against 14 us); so when a page's
// equal tickets are not much larger than that, none crosses a page.
void cut_once(DevQuery& Q, uint64_t per_warp, uint64_t warps) {
  const uint64_t P = Q.page_rows, big = round_up(per_warp, kMB);
  cut(Q, big, 0, 0);
  if (big >= P) return;
  for (uint64_t per = (P + big - 1) / big; per > 0; --per) {
    const uint64_t rows = round_up((P + per - 1) / per, kMB), n = (P + rows - 1) / rows;  // n <= per tickets a page
    if (double(rows) > double(big) + 256.0 / row_cost(Q)) return;
    const uint64_t count = Q.nrows / P * n + (Q.nrows % P + rows - 1) / rows;
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
// tickets:
//  - a query of at most chunk_rows rows per warp is cut into one ticket per
//    warp (whole mini blocks); there is no pool.  Rows of pages that the first
//    step's range misses do not count (Q.live): a table of which a seventh is
//    read has seven tickets per warp, eight at most, as a ticket that skips
//    its page costs a load too;
//  - a larger one into equal tickets of at most chunk_rows, the same number
//    for every warp, and a pool of two 512-row tickets per warp, which even
//    out the warps' different speeds;
//  - a batch likewise over all its queries, tickets of equal cost, a tenth of
//    a warp's work in each of two pool tickets; a query with skipped pages is
//    in the pool as a whole, since they would fall to few CTAs;
//  - a batch of large queries (kInOrderRows each on average) is drawn whole
//    from the pool, query by query, each query's last rows in small tickets:
//    the CTAs' meetings at its few switches cost little and no estimate of a
//    query's cost is needed (16 queries over 67 M rows: 3.6 ms, in owned runs
//    5.8).
// With a fixed ticket size (a tuning names it) the last rows, two tickets of
// an eighth per warp, make the pool, in a batch one per warp and query.
bool layout_tickets(DevQuery* Q, int n, uint64_t warps, uint32_t chunk_rows, bool fixed, uint64_t* begin) {
  constexpr uint64_t kInOrderRows = uint64_t(1) << 24;
  uint64_t all = 0;
  for (int i = 0; i < n; ++i) all += Q[i].nrows;
  const bool in_order = n > 1 && all / uint64_t(n) >= kInOrderRows;
  const uint64_t tile = kMbPerWarpTile * kMB, chunk = chunk_rows;
  if (fixed || in_order) {
    const uint64_t small = std::max<uint64_t>(tile, chunk / 8 / tile * tile);
    uint64_t want = 2 * warps * small;  // from the last query backwards
    for (int i = n - 1; i >= 0; --i) {
      const uint64_t rows = std::min(Q[i].nrows, want);
      want -= rows;
      cut(Q[i], chunk, small, std::max(rows, n > 1 ? std::min(Q[i].nrows, warps * small) : 0));
    }
  } else if (n == 1) {
    const uint64_t read = std::max<uint64_t>(1, uint64_t(double(Q->nrows) * read_part(*Q)));
    const uint64_t per_warp = (read + warps - 1) / warps, pool = 2 * tile;
    if (per_warp <= chunk) {
      cut_once(*Q, per_warp, warps);
    } else {
      const uint64_t own = per_warp - pool, k = (own + chunk - 1) / chunk;
      cut(*Q, round_up((own + k - 1) / k, tile), tile, warps * pool);
    }
  } else {
    double total = 0;
    for (int i = 0; i < n; ++i) total += double(Q[i].nrows) * read_part(Q[i]) * Q[i].cost;
    const double per_warp = total / double(warps);
    const double k = std::max(1.0, std::ceil(0.8 * per_warp / double(chunk)));
    for (int i = 0; i < n; ++i) {
      const double c = std::max(0.25, double(Q[i].cost));
      const uint64_t big = std::min(chunk, round_up(uint64_t(0.8 * per_warp / k / c) + 1, kMB));
      const uint64_t small = std::min(big, round_up(uint64_t(0.1 * per_warp / c) + 1, kMB));
      cut(Q[i], big, small, uint64_t(0.2 * double(Q[i].nrows)));
      if (Q[i].live < 0.75f) {
        Q[i].tail_first = Q[i].tail_row = 0;
        Q[i].tail_rows = uint32_t(big);
        Q[i].nchunks = (Q[i].nrows + big - 1) / big;
      }
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
  return n == 1;
}

size_t fused_dynamic_smem(uint32_t acc_slots, size_t smem_tables, int threads, uint32_t stage_bw, bool text) {
  return ((acc_slots * sizeof(unsigned long long) + 15) & ~size_t(15)) + ((smem_tables + 15) & ~size_t(15)) +
         size_t(threads / 32) *
             (kListCap * sizeof(uint32_t) + stage_warp_bytes(stage_bw) + (text ? kSearchWords * sizeof(uint32_t) : 0));
}

// The occupancy of the string-capable build bounds the grid of both builds
// (same launch bounds and shared memory; the lean build needs no more
// registers); a staged launch (stage_bw > 0) runs the staging build.
int fused_blocks_per_sm(int threads, uint32_t acc_slots, size_t smem_tables, bool host_data, int min_blocks,
                        uint32_t stage_bw, bool text) {
  const size_t smem = fused_dynamic_smem(acc_slots, smem_tables, threads, stage_bw, text);
  if (threads > 256) return fused_wide_occupancy(threads, smem);
  if (host_data) return fused_host_occupancy(threads, smem, min_blocks);
  return stage_bw ? fused_stage_occupancy(threads, smem, min_blocks) : fused_text_occupancy(threads, smem, min_blocks);
}

// Host-resident batches and batches with a CONTAINS or FSST step run the
// string-capable build; device-resident batches without one run the lean
// build, or the staging build when the batch is staged.
cudaError_t launch_fused(const FusedLaunch& L, cudaStream_t s) {
  const size_t smem = fused_dynamic_smem(L.acc_slots, L.smem_tables, L.threads, L.stage_bw, L.text);
  const uint32_t tb = uint32_t((L.smem_tables + 15) & ~size_t(15));
  if (L.threads > 256) return fused_wide_launch(L, smem, tb, s);  // prepare admits lean batches only
  if (L.host_data) return fused_host_launch(L, smem, tb, s);
  if (L.text) return fused_text_launch(L, smem, tb, s);
  if (L.stage_bw) return fused_stage_launch(L, smem, tb, s);
  return fused_lean_launch(L, smem, tb, s);
}

}  // namespace dpf
