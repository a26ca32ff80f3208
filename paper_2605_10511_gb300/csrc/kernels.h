// Host-callable launchers of the library's kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dpf_internal.h"

namespace dpf {

// Shared-memory accumulator capacity of one CTA (int64 slots).
constexpr uint32_t kSmemAccSlots = 4096;
constexpr uint32_t kMbPerWarpTile = 4;
// The fused kernel is compiled twice, for 3 and for 4 resident 256-thread CTAs
// per SM (register budgets of 80 and 64 per thread): occupancy, more than
// issue, bounds it.  The 4-CTA build spills a little and wins when four CTAs'
// shared memory fits; the launch configuration (ctas_per_sm) picks one.
constexpr int kFusedMinBlocksLo = 3;
constexpr int kFusedMinBlocksHi = 4;
// Most rows of one scheduling ticket (one warp's unit of work) unless tuned.
constexpr uint32_t kDefaultChunkRows = 4096;
// Rows from which one query takes the 1,024-thread build unless tuned.
constexpr uint64_t kWideRows = uint64_t(1) << 23;
// Shared memory of one warp's survivor list (1,024 entries).
constexpr uint32_t kListBytesPerWarp = 1024 * 4;
// Words of one warp's scratch of the cooperative string search (search_mb),
// in launches that have a string-matcher step.
constexpr uint32_t kSearchWords = 384;
// Estimated selectivity of the first step from which step 1's mini blocks
// are prefetched into L2 during the dense tiles (DevQuery::pf_step).
constexpr double kPrefetchMinSel = 0.03;
// Staging of the first step's mini blocks unless tuned (DPF_STAGE_ON / _OFF).
constexpr int32_t kDefaultStaging = 2;
// Grouped aggregates are added with one int64 atomic per row unless tuned
// (DPF_GROUP_AGG_*): warp aggregation measured slower on GB300 both with
// 1,024 Zipf groups (1.8x) and with 15 groups, one holding 97 % of the rows
// (1.3x); the autotuner tries it per plan signature.
constexpr int32_t kDefaultGroupAgg = 2;
// Join-table representation by the key range of the kept rows (R8): a
// direct table of one word per key up to 2^22 keys (16 MB), a rank
// directory (2 bits per key plus the kept payloads) up to 2^28 keys, open
// addressing beyond.
constexpr uint64_t kDirectMaxRange = uint64_t(1) << 22;
constexpr uint64_t kDirectAlways = uint64_t(1) << 20;  // direct however few rows are kept
constexpr uint64_t kRankMaxRange = uint64_t(1) << 28;
// Shared-memory bytes of the code-level matcher tables of a PREFIX / CONTAINS
// step with a pattern of plen bytes on an FSST column: for every matcher
// state below plen, the next state after one symbol code (256 entries) and
// after one literal byte (256 entries), and behind the former a flag per code.
inline uint32_t fsst_match_bytes(uint32_t plen) { return (plen + 1) * 512u; }

// What a launch reads of a query's table, and how long a row of it takes.
struct ScanShare {
  uint64_t row0, rows;  // from the first to the last page that the first step's range meets (at least one row)
  double live;          // fraction of those rows in such pages
  double cost;          // time of a row, 1 = a star join's
};

// Cuts the n queries of a launch into tickets of at most chunk_rows rows for
// `warps` resident warps: sets each query's chunk_rows, page_tickets, tail_first,
// tail_row, tail_rows, row0 and nchunks and fills begin (2 n + 2 entries,
// FusedLaunch::qbegin).
void layout_tickets(DevQuery* Q, const ScanShare* S, int n, uint64_t warps, uint32_t chunk_rows, uint64_t* begin);

// Fused persistent kernel over a batch of compiled queries (Sec. 3.2).
// qbegin[0..nq] = first owned ticket of each query (qbegin[nq] = owned),
// qbegin[nq + 1 .. 2 nq + 1] = its first pool ticket (the last one = pool).
struct FusedLaunch {
  const DevQuery* queries;
  const uint64_t* qbegin;
  int nq;
  uint64_t owned, pool;
  unsigned int* drawn;  // batches with owned tickets: a counter per CTA, zero between launches (else nullptr)
  Sched* sched;
  unsigned int* status_out;   // where the launch leaves its status word (mapped host memory); nullptr: in sched
  int grid, threads;
  uint32_t acc_slots;   // int64 shared accumulators per CTA (max over the batch)
  size_t smem_tables;   // bytes of the CTA's join-table region
  bool host_data;       // some column lives in mapped pinned host memory
  int min_blocks;       // kFusedMinBlocksLo or kFusedMinBlocksHi: which build runs
  bool text;            // some query has a CONTAINS step or a string step on an FSST
                        // column (the build with the general string matcher runs)
  uint32_t stage_bw;    // bits a value of the warps' staging ring slots hold; 0 = no ring
};
cudaError_t launch_fused(const FusedLaunch& L, cudaStream_t s);
// Occupancy of the fused kernel for (threads, dynamic smem); also sets the
// kernel's dynamic shared-memory limit.
int fused_blocks_per_sm(int threads, uint32_t acc_slots, size_t smem_tables, bool host_data, int min_blocks,
                        uint32_t stage_bw, bool text);
size_t fused_dynamic_smem(uint32_t acc_slots, size_t smem_tables, int threads, uint32_t stage_bw, bool text);

// Hash build (Kernel #1 of Sec. 3.1).  `q` describes the dimension scan:
// cols/steps as for the fused kernel, build_key/build_pay name columns.
struct BuildLaunch {
  const DevQuery* q;          // device copy
  uint2* table;               // open addressing: capacity slots (mask + 1)
  uint32_t mask;
  uint32_t* direct;           // direct table: krange entries (or nullptr)
  int32_t kmin;
  uint32_t krange;
  uint4* rank_dir;            // rank table: (krange + 63) / 64 directory words (or nullptr)
  uint32_t* rank_pay;         //   payloads of the present keys, in key order
  uint32_t* rank_sums;        //   scratch: one count per 1,024 directory words
  uint2* rank_stage;          //   scratch: {key offset, payload} of each inserted row, in insertion order
  unsigned long long* stage_n;  //   its count
  uint32_t rank_cap;          //   payload words (= staged pairs) the table holds
  struct BuildStat* stat;     // status word and rows kept by the pass
  bool measure;               // the pass also records the kept keys' range
  uint64_t nrows, page_rows;
  bool host_data;
};
// Device-side outcome of a build pass: its status bits, the rows it kept
// (inserted, or counted) and their key range, kept by
// atomicMax from zero bytes on: the largest rank(key), and the largest ~rank.
struct BuildStat {
  Sched sched;
  unsigned long long inserted;
  uint32_t hi, lo;
  __host__ __device__ static uint32_t rank(int32_t key) { return uint32_t(key) ^ 0x80000000u; }
  __host__ __device__ int32_t key_hi() const { return int32_t(hi ^ 0x80000000u); }
  __host__ __device__ int32_t key_lo() const { return int32_t(~lo ^ 0x80000000u); }
};
cudaError_t launch_build_count(const BuildLaunch& L, cudaStream_t s);
cudaError_t launch_build_insert(const BuildLaunch& L, cudaStream_t s);
cudaError_t launch_init_table(uint2* table, uint32_t slots, cudaStream_t s);
cudaError_t launch_init_direct(uint32_t* table, uint32_t n, cudaStream_t s);

// Device-side encode of a loaded column (encode_dev.cu): raw values in device
// memory to the page images that dpf_encode_column writes.
struct EncodeMb {          // a mini block: FOR64's base is {base, first} as one int64, low half first
  int32_t base, first;
  uint32_t bw, word_off;   // word_off: 4-byte (FOR64: 8-byte) words into the page's payload
};
struct EncodePage {
  uint64_t bytes;          // size of the page image
  long long lo, hi;        // value bounds from its headers (FOR / DICT / DELTA)
  uint32_t max_bw, extra, bad, pad_;  // extra: offset of the byte region; bad: lengths the format cannot hold
};
struct EncodeDev {
  uint32_t codec, page_rows;
  uint64_t nrows, npages, nmb;
  const int32_t* v32;      // FOR / DELTA values, DICT codes
  const long long* v64;    // FOR64
  const uint8_t* bytes;    // STR: bytes from the first string on, and
  const unsigned long long* offs;  // the caller's row offsets (the first may be non-zero)
  EncodeMb* mb;            // [nmb]
  unsigned long long* mb_bytes;  // STR: [nmb] string bytes, then the mini block's byte start in its page
  EncodePage* pages;       // [npages]
  uint8_t* blob;           // write: the pages, zeroed
  const uint64_t* page_off;
};
cudaError_t launch_encode_plan(const EncodeDev& E, cudaStream_t s);   // fills mb and pages
cudaError_t launch_encode_write(const EncodeDev& E, cudaStream_t s);  // fills blob
// Dictionary of int32 values: their range (ranks of BuildStat), the distinct
// ones in ascending order (at most cap are written; bitmap and rank: nwords
// words over [lo, lo + 32 nwords), bitmap zeroed) and, in place, their codes.
cudaError_t launch_dict_range(const int32_t* v, uint64_t n, uint32_t* hi, uint32_t* lo, cudaStream_t s);
cudaError_t launch_dict_values(const int32_t* v, uint64_t n, int32_t lo, uint32_t nwords, uint32_t* bitmap, uint32_t* rank,
                               int32_t* values, uint32_t cap, unsigned long long* count, cudaStream_t s);
cudaError_t launch_dict_codes(int32_t* v, uint64_t n, int32_t lo, const uint32_t* bitmap, const uint32_t* rank,
                              cudaStream_t s);
// Columns of at least this many rows are encoded on the device when they are
// to live there: at 8,192 rows the host encoder takes 50 to 57 us (FOR, DELTA,
// FOR64) where the device's launches take 60, at 65,536 rows it is behind at
// every codec; its sort of a dictionary's values takes 280 us at 2,000 rows
// against the device's 140.
constexpr uint64_t kDeviceEncodeRows = 16384;
constexpr uint64_t kDeviceDictRows = 1024;
// Widest value range of a dictionary made on the device (its bitmap is ranked
// by one CTA).
constexpr uint64_t kDeviceDictRange = uint64_t(1) << 20;

// Unfused per-operator chain (baseline).  Buffers for every intermediate:
// decoded columns, predicate flags, two ping-pong (row id, group id) lists
// and the device-side list lengths.
struct UnfusedChain {
  DevQuery q;                 // host copy of the compiled plan
  const DevQuery* dq;         // device copy (read by the assembly kernel)
  int32_t* vals[kMaxCols];    // decoded int columns
  int32_t* lens[kMaxCols];    // decoded string lengths
  uint64_t* offs[kMaxCols];   // absolute string byte offsets in the column blob
  uint8_t* flags;
  uint32_t* rid[2];
  uint32_t* gid[2];
  unsigned long long* counts; // [2 + kMaxSteps] list lengths
  Sched* sched;
};
constexpr int kUnfusedCounts = 2 + kMaxSteps;
cudaError_t launch_unfused(const UnfusedChain& U, cudaStream_t s, uint32_t* launches);

}  // namespace dpf
