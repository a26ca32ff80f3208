// The fused persistent kernel (Sec. 3.2, Sec. 4.1 "fused kernel composition"),
// as a header: fused_lean.cu, fused_text.cu, fused_host.cu and fused_stage.cu
// each compile two of its builds (device-resident pages without / with the
// general string matcher, host-resident pages, device-resident pages staged
// in shared memory; 3 and 4 resident CTAs per SM) and fused_wide.cu those for
// CTAs of 512 and 1,024 threads, so the builds compile in parallel.
//
// One launch executes every query of a batch.  Each warp repeatedly takes a
// ticket (a range of rows of one query's fact table: the outer loop of Sec. 3.2
// without host intervention), splits it into tiles of TB mini blocks and runs
// decode -> predicates -> probes -> aggregation on them with all row state in
// registers.  Per-CTA int64 accumulators live in
// shared memory while the CTA stays on one query; they are added to the
// query's global accumulators when the CTA moves to another query or exits.
// The CTA that flushes a query's last ticket turns its accumulators into
// records ordered by key tuple (the record format of Kernel #3, Sec. 3.1) and
// zeroes the scratch state, so the kernel can be replayed from a CUDA graph.
#pragma once

#include <climits>

#include "../../include/dpf.h"
#include "tile.cuh"

namespace dpf {
namespace {

// The CTA's dynamic shared memory: accumulators, join tables, the warps'
// survivor lists (and staging rings).
extern __shared__ __align__(16) uint8_t dyn[];
__device__ __forceinline__ uint32_t* shared_acc() { return reinterpret_cast<uint32_t*>(dyn); }

struct alignas(16) CtaState {
  DevQuery q;
  int wq[32];          // query of the ticket each warp holds (INT_MAX: none left)
  unsigned int drawn;  // tickets drawn from the CTA's own range (one query)
  unsigned int victim; // batches: the CTA whose run this one's warps draw from, at first its own
  unsigned int mine;   // tickets of the current query this CTA processed
  int last;
  unsigned int warp_sum[32];
};

// Block-wide exclusive scan of a 0/1 flag; returns the rank, *total the sum.
__device__ __forceinline__ uint32_t block_rank(bool flag, CtaState& cs, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned b = __ballot_sync(kFull, flag);
  if (lane == 0) cs.warp_sum[warp] = __popc(b);
  __syncthreads();
  uint32_t before = 0, all = 0;
  for (int w = 0; w < nw; ++w) {
    const uint32_t x = cs.warp_sum[w];
    if (w < warp) before += x;
    all += x;
  }
  __syncthreads();
  *total = all;
  return before + __popc(b & ((1u << lane) - 1u));
}

// Aggregate a of group g (count rows): a COUNT is the group's row count and
// has no accumulator of its own.
__device__ __forceinline__ long long agg_value(const DevQuery& Q, uint32_t g, int a, long long count) {
  if (a >= int(Q.naggs)) return 0;
  if (Q.agg_op[a] == DPF_AGG_COUNT) return count;
  return (long long)__ldcg(Q.acc + uint64_t(g) * (1 + Q.naggs) + 1 + a);
}

// Converts a query's global accumulators into records and clears them.
__device__ void assemble(const DevQuery& Q, CtaState& cs) {
  const uint32_t S1 = 1 + Q.naggs;
  dpf_record* out = reinterpret_cast<dpf_record*>(Q.out);
  if (Q.nkeys == 0) {
    if (threadIdx.x == 0) {
      dpf_record r;
      r.key[0] = r.key[1] = 0;
      r.count = (long long)__ldcg(Q.acc);
      for (int a = 0; a < 4; ++a) r.val[a] = agg_value(Q, 0, a, r.count);
      out[0] = r;
      *Q.out_n = 1;
    }
  } else {
    uint32_t base = 0;
    for (uint32_t g0 = 0; g0 < Q.domain; g0 += blockDim.x) {
      const uint32_t g = g0 + threadIdx.x;
      const unsigned long long cnt = g < Q.domain ? __ldcg(Q.acc + uint64_t(g) * S1) : 0ull;
      uint32_t total;
      const uint32_t rank = block_rank(cnt != 0, cs, &total);
      if (cnt != 0) {
        dpf_record r;
        for (int k = 0; k < 2; ++k) {
          if (k < int(Q.nkeys)) {
            const uint32_t code = (g / Q.key_div[k]) % Q.key_dom[k];
            r.key[k] = __ldg(Q.key_dict[k] + code);
          } else {
            r.key[k] = 0;
          }
        }
        r.count = (long long)cnt;
        for (int a = 0; a < 4; ++a) r.val[a] = agg_value(Q, g, a, r.count);
        out[base + rank] = r;
      }
      base += total;
    }
    if (threadIdx.x == 0) *Q.out_n = base;
  }
  __syncthreads();
  const uint64_t n = uint64_t(Q.domain) * S1;
  for (uint64_t i = threadIdx.x; i < n; i += blockDim.x) Q.acc[i] = 0ull;
  if (threadIdx.x == 0) *Q.done = 0u;
  __threadfence();
}

// Adds the CTA's accumulators for Q to global memory, counts the chunks it
// processed and, if they were the query's last, assembles the result.  Each
// CTA starts at its own group, so that the CTAs leaving a query together add
// to different addresses.
__device__ void finish_query(const DevQuery& Q, uint32_t mine, CtaState& cs) {
  const uint32_t* sacc = shared_acc();
  const uint32_t S1 = 1 + Q.naggs;
  if (Q.use_smem_acc) {
    const uint32_t n = Q.domain * S1, rot = uint32_t((uint64_t(blockIdx.x) * n) / gridDim.x);
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
      const uint32_t j = i + rot < n ? i + rot : i + rot - n, g = j / S1;  // global accumulators: [group][slot]
      const uint32_t at = (j - g * S1) * Q.domain + g;
      const unsigned long long x = sacc[at] | ((unsigned long long)sacc[n + at] << 32);
      if (x) atomicAdd(Q.acc + j, x);
    }
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned old = atomicAdd(Q.done, mine);
    cs.last = (uint64_t(old) + mine == Q.nchunks);
  }
  __syncthreads();
  if (cs.last) {
    __threadfence();
    assemble(Q, cs);
  }
  __syncthreads();
}

// One accumulator slot of the groups that a warp adds to, in registers (taken
// once before a list's rounds, like PointCol): the CTA's shared accumulators,
// or the query's global int64 ones when the domain does not fit.  A shared
// int64 accumulator is kept as two 32-bit halves, all low halves first
// (slot-major: slot * domain + group, so that neighbouring groups lie in
// different banks), then all high halves.  32-bit shared atomics are done by
// the memory pipe, also when lanes of one instruction hit the same address;
// a 64-bit one is a compare-and-swap loop that repeats for each of them.  An
// add needs the high half only when it carries (or the value itself has high
// bits), so most adds are one 32-bit atomic; the sum is exact modulo 2^64.
struct AccSlot {
  unsigned long long* g;       // global accumulators of the slot, a group every `slots`
  uint32_t at, to_hi, slots;   // shared: index of the slot's group 0; distance to the high halves
  bool shared, warp;           // warp: warp-aggregated updates
  __device__ __forceinline__ AccSlot(const DevQuery& Q, uint32_t slot)
      : g(Q.acc + slot), at(slot * Q.domain), to_hi(Q.domain * (1 + Q.naggs)), slots(1 + Q.naggs),
        shared(Q.use_smem_acc != 0), warp(Q.warp_agg != 0) {}
};
__device__ __forceinline__ void acc_add(const AccSlot& A, uint32_t gid, unsigned long long x) {
  if (!A.shared) {
    atomicAdd(A.g + uint64_t(gid) * A.slots, x);
    return;
  }
  uint32_t* p = shared_acc() + A.at + gid;
  const uint32_t lo = uint32_t(x);
  const uint32_t old = atomicAdd(p, lo);
  const uint32_t hi = uint32_t(x >> 32) + uint32_t(old + lo < lo);
  if (hi) atomicAdd(p + A.to_hi, hi);
}

// Warp-aggregated group-by update (hash aggregation of Kernel #3, Sec. 3.1),
// by the round's leading group: the lanes holding the group id of the
// round's first valid lane combine their values with warp reductions and
// that lane issues the group's single atomic; every other valid lane adds
// its own value.  A hot group (a Zipf head, or one key holding most rows)
// thus costs one atomic per round instead of one per row on the same
// address.  The sum is exact modulo 2^64: a value is split into 16-bit parts
// whose sums over 32 lanes stay below 2^21 (kWide: four unsigned parts of
// the 64-bit value; otherwise the value is an int32, whose low 16 bits and
// signed high 16 bits are summed).  Warp-uniform call.
template <bool kWide>
__device__ __forceinline__ void lead_group_add(const AccSlot& A, uint32_t gid, unsigned long long x, bool valid,
                                               int lane) {
  const uint32_t vm = __ballot_sync(kFull, valid);
  if (vm == 0) return;
  const int lead = __ffs(vm) - 1;
  const uint32_t g0 = __shfl_sync(kFull, gid, lead);
  const bool mine = valid && gid == g0;
  const uint32_t m = __ballot_sync(kFull, mine);
  if (mine) {
    unsigned long long t;
    if (kWide) {
      const uint32_t lo = uint32_t(x), hi = uint32_t(x >> 32);
      t = (unsigned long long)__reduce_add_sync(m, lo & 0xffffu) +
          ((unsigned long long)__reduce_add_sync(m, lo >> 16) << 16) +
          ((unsigned long long)__reduce_add_sync(m, hi & 0xffffu) << 32) +
          ((unsigned long long)__reduce_add_sync(m, hi >> 16) << 48);
    } else {
      const int32_t v = int32_t(uint32_t(x));
      const uint32_t s_lo = __reduce_add_sync(m, uint32_t(v) & 0xffffu);
      const int32_t s_hi = int32_t(__reduce_add_sync(m, uint32_t(v >> 16)));  // |sum| < 2^20
      t = (unsigned long long)((long long)s_lo + (long long)s_hi * 65536ll);
    }
    if (lane == lead) acc_add(A, g0, t);
  } else if (valid) {
    acc_add(A, gid, x);
  }
}

// A grouped update: warp-aggregated by the leading group or one atomic per row.
template <bool kWide>
__device__ __forceinline__ void group_add(const AccSlot& A, uint32_t gid, unsigned long long x, bool valid, int lane) {
  if (A.warp) lead_group_add<kWide>(A, gid, x, valid, lane);
  else if (valid) acc_add(A, gid, x);
}

// Adds a warp's per-lane sums (an ungrouped aggregate) to group 0.
__device__ __forceinline__ void single_add(const AccSlot& A, unsigned long long sum, int lane) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) sum += __shfl_down_sync(kFull, sum, d);
  if (lane == 0 && sum != 0) acc_add(A, 0, sum);
}

// Group id of a list entry, and whether the row takes part: a group id beyond
// the domain is a corrupt dictionary code, which drops the row.
__device__ __forceinline__ uint32_t entry_group(uint32_t e, uint32_t domain, bool& valid, unsigned int* status) {
  const uint32_t gid = e >> kRowBits;
  if (valid && gid >= domain) {
    atomicOr(status, S_CORRUPT);
    valid = false;
  }
  return gid;
}

// One aggregate over a warp's list, specialised on its operation (dpf_agg_op)
// and on how its operands are read: kPoint = FOR/DICT columns, one bit field
// per row; otherwise any codec through row_value (DELTA decodes densely).
// count: the pass counts the rows too (slot 0), which saves a pass of its own.
template <bool kHost, int kOp, bool kPoint>
__device__ __forceinline__ void agg_pass(const DevQuery& Q, const PageState& P, uint32_t seg_mb,
                                         const uint32_t* list, uint32_t n, int lane, uint32_t slot, int ca, int cb,
                                         bool single, bool count, unsigned int* status) {
  constexpr bool kTwo = kOp == DPF_AGG_SUM_MUL || kOp == DPF_AGG_SUM_SUB;
  const AccSlot A(Q, slot);
  const uint32_t domain = Q.domain;
  const PointCol Ca = point_col(Q, ca, P, seg_mb), Cb = kTwo ? point_col(Q, cb, P, seg_mb) : Ca;
  long long sum = 0;
  for (uint32_t i0 = 0; i0 < n; i0 += 32) {
    bool valid = i0 + lane < n;
    const uint32_t e = valid ? list[i0 + lane] : 0u;
    const uint32_t r = e & ((1u << kRowBits) - 1u);
    const uint32_t gid = entry_group(e, domain, valid, status);
    if (count && valid) atomicAdd(shared_acc() + gid, 1u);
    const int32_t va = int32_t(kPoint ? point_at<kHost>(Ca, r)
                                      : row_value<kHost>(Q, ca, P, seg_mb, r, valid, lane, status));
    int32_t vb = 0;
    if (kTwo)
      vb = int32_t(kPoint ? point_at<kHost>(Cb, r) : row_value<kHost>(Q, cb, P, seg_mb, r, valid, lane, status));
    long long x = va;
    if (kOp == DPF_AGG_SUM_MUL)
      x = (long long)((unsigned long long)(long long)va * (unsigned long long)(long long)vb);
    else if (kOp == DPF_AGG_SUM_SUB)
      x = (long long)va - (long long)vb;
    if (single) sum += valid ? x : 0;
    else group_add<kTwo>(A, gid, (unsigned long long)x, valid, lane);
  }
  if (single) single_add(A, (unsigned long long)sum, lane);
}

// An aggregate with a FOR64 operand: one survivor per lane, int64 operands,
// arithmetic modulo 2^64.  Inlined: an out-of-line call made the caller
// spill around it, while inlined it leaves the 32-bit passes' register
// allocation as it was.
template <bool kHost, int kOp>
__device__ __forceinline__ void agg_pass_wide(const DevQuery& Q, const PageState& P, uint32_t seg_mb,
                                           const uint32_t* list, uint32_t n, int lane, uint32_t slot, int ca, int cb,
                                           bool single, bool count, unsigned int* status) {
  const AccSlot A(Q, slot);
  const uint32_t domain = Q.domain;
  unsigned long long sum = 0;
  for (uint32_t i0 = 0; i0 < n; i0 += 32) {
    bool valid = i0 + lane < n;
    const uint32_t e = valid ? list[i0 + lane] : 0u;
    const uint32_t r = e & ((1u << kRowBits) - 1u);
    const uint32_t gid = entry_group(e, domain, valid, status);
    if (count && valid) atomicAdd(shared_acc() + gid, 1u);
    const unsigned long long a = (unsigned long long)value64<kHost>(Q, ca, P, seg_mb, r, valid, lane, status);
    unsigned long long b = 0;
    if (kOp == DPF_AGG_SUM_MUL || kOp == DPF_AGG_SUM_SUB)
      b = (unsigned long long)value64<kHost>(Q, cb, P, seg_mb, r, valid, lane, status);
    const unsigned long long x = kOp == DPF_AGG_SUM ? a : (kOp == DPF_AGG_SUM_MUL ? a * b : a - b);
    if (single) sum += valid ? x : 0ull;
    else group_add<true>(A, gid, x, valid, lane);
  }
  if (single) single_add(A, sum, lane);
}

template <bool kHost, int kOp>
__device__ __forceinline__ void agg_dispatch(const DevQuery& Q, const PageState& P, uint32_t seg_mb,
                                             const uint32_t* list, uint32_t n, int lane, uint32_t slot, int ca, int cb,
                                             bool single, bool count, unsigned int* status) {
  if (Q.cols[ca].codec == C_FOR64 || (kOp != DPF_AGG_SUM && Q.cols[cb].codec == C_FOR64)) {
    agg_pass_wide<kHost, kOp>(Q, P, seg_mb, list, n, lane, slot, ca, cb, single, count, status);
    return;
  }
  const bool point = Q.cols[ca].codec != C_DELTA && (kOp == DPF_AGG_SUM || Q.cols[cb].codec != C_DELTA);
  if (point) agg_pass<kHost, kOp, true>(Q, P, seg_mb, list, n, lane, slot, ca, cb, single, count, status);
  else agg_pass<kHost, kOp, false>(Q, P, seg_mb, list, n, lane, slot, ca, cb, single, count, status);
}

// Aggregation over a warp's survivor list (Kernel #3 hash aggregation;
// int64 as in Sec. 4.3): slot 0 counts rows, slot 1 + a holds aggregate a
// (unused when that is a COUNT).
// domain == 1: per-lane int64 sums reduced across the warp; otherwise
// int64 atomics (one per row, or warp-aggregated by the round's leading
// group: group_add) into the CTA's shared accumulators (or the query's
// global ones for large domains), indexed by the dense group id.
template <bool kHost>
__device__ __forceinline__ void list_aggregate(const DevQuery& Q, const PageState& P, uint32_t seg_mb,
                                               const uint32_t* list, uint32_t n, int lane,
                                               unsigned int* status) {
  const bool single = Q.domain == 1;
  bool count = false;  // the next aggregate's pass counts the rows too
  if (single) {
    if (lane == 0) acc_add(AccSlot(Q, 0), 0, (unsigned long long)n);
  } else {
    // a shared count needs no high half while the table has fewer than 2^32
    // rows: then the first aggregate's pass makes it
    bool other = false;
    for (uint32_t a = 0; a < Q.naggs; ++a) other = other || Q.agg_op[a] != DPF_AGG_COUNT;
    count = Q.use_smem_acc && (Q.nrows >> 32) == 0 && !Q.warp_agg;
    if (!count || !other) {
      const AccSlot A(Q, 0);
      const uint32_t domain = Q.domain;
      for (uint32_t i0 = 0; i0 < n; i0 += 32) {
        bool valid = i0 + lane < n;
        const uint32_t gid = entry_group(valid ? list[i0 + lane] : 0u, domain, valid, status);
        if (!count) group_add<false>(A, gid, 1ull, valid, lane);
        else if (valid) atomicAdd(shared_acc() + gid, 1u);
      }
      count = false;
    }
  }
  for (uint32_t a = 0; a < Q.naggs; ++a) {
    const int ca = Q.agg_a[a], cb = Q.agg_b[a];
    switch (Q.agg_op[a]) {
      case DPF_AGG_COUNT: continue;  // the row count (slot 0)
      case DPF_AGG_SUM:
        agg_dispatch<kHost, DPF_AGG_SUM>(Q, P, seg_mb, list, n, lane, 1 + a, ca, cb, single, count, status);
        break;
      case DPF_AGG_SUM_MUL:
        agg_dispatch<kHost, DPF_AGG_SUM_MUL>(Q, P, seg_mb, list, n, lane, 1 + a, ca, cb, single, count, status);
        break;
      default:
        agg_dispatch<kHost, DPF_AGG_SUM_SUB>(Q, P, seg_mb, list, n, lane, 1 + a, ca, cb, single, count, status);
        break;
    }
    count = false;
  }
}

// The dense part of one tile, for one warp: the first step over all its rows
// (kGid: the step adds group-id contributions), then its survivors appended
// to the warp's list after the first n entries; returns the list length.
template <bool kHost, bool kText, bool kGid, bool kStaged = false>
__device__ __forceinline__ uint32_t tile_first_step(const DevQuery& Q, const PageState& P, const TileHdr& H,
                                                    uint32_t i0, uint32_t nmb, uint32_t row_base, const uint8_t* stab,
                                                    uint32_t* list, uint32_t n, int lane, unsigned int* status,
                                                    StagedPay sp = StagedPay{nullptr, 0, 0},
                                                    uint32_t* search = nullptr) {
  TileState T;
  tile_init<kGid>(P, i0, nmb, lane, T);
  tile_dense_step<kHost, kText, kGid, kStaged>(Q, 0, P, H, T, stab, lane, status, sp, search);
  return tile_compact<kHost, kGid>(T, list, n, row_base, lane);
}

// The first step's column of Q in page P: its page address and packed words.
struct FirstCol {
  int c;
  uint32_t codec;
  const uint8_t* pg;
  const uint8_t* pay;
};
__device__ __forceinline__ FirstCol first_col(const DevQuery& Q, const PageState& P) {
  FirstCol f;
  f.c = Q.steps[0].col;
  f.codec = Q.cols[f.c].codec;
  f.pg = reinterpret_cast<const uint8_t*>(__shfl_sync(kFull, P.pg, f.c));
  f.pay = f.pg + payload_offset(f.codec, P.prow);
  return f;
}

// One ticket (layout_tickets): a range of rows of Q's fact table, processed by
// one warp, cut at page boundaries into tiles.  A page whose
// zone map misses the first step's value range is skipped whole; inside a
// page, mini blocks whose headers miss it are skipped by the first step.
// Each tile loads its headers as it starts (the other resident warps hide
// the latency).  The list collects the survivors of consecutive tiles (a
// segment of at most 2^kRowBits rows of one page) before the later steps and
// the aggregation run on them.
template <bool kHost, bool kText, bool kStage>
__device__ void process_ticket(const DevQuery& Q, uint64_t chunk, const uint8_t* stab,
                               uint32_t* list, int lane, unsigned int* status,
                               uint8_t* ring) {
  const uint64_t PR = Q.page_rows;
  uint64_t r0, r1;
  ticket_rows(Q, chunk, &r0, &r1);
  const bool gid0 = Q.nsteps != 0 && step_adds_gid(Q.steps[0]);
  for (uint64_t p = r0 / PR; p <= (r1 - 1) / PR; ++p) {
    const uint64_t pr0 = tmax<uint64_t>(r0, p * PR), pr1 = tmin<uint64_t>(r1, (p + 1) * PR);
    const uint32_t mb0 = uint32_t((pr0 - p * PR) / kMB);
    const uint32_t mb1 = uint32_t((pr1 - p * PR + kMB - 1) / kMB);
    const uint32_t ntiles = (mb1 - mb0 + TB - 1) / TB;
    if (Q.nsteps != 0) {  // zone map: skip a page the first step's range misses
      const DevStep& S0 = Q.steps[0];
      const int2 z = __ldg(Q.cols[S0.col].zone + p);
      if (S0.zlo > S0.zhi || z.y < S0.zlo || z.x > S0.zhi) continue;
    }
    PageState P;
    page_begin<kHost>(Q, p, lane, P);
    // staged first step (StageRing in tile.cuh): the headers of tiles 0 and 1
    // and the words of tile 0 are in flight before the first decode
    // a staged launch stages every query (the host makes it so)
    const uint32_t bwcap = kStage && !kHost ? Q.stage : 0u;
    if (kStage && bwcap == 0) {
      if (lane == 0) atomicOr(status, S_INTERNAL);
      return;
    }
    if (kStage) {
      const FirstCol f = first_col(Q, P);
      stage_headers(ring, 0, f.pg, f.codec, mb0, tmin<uint32_t>(TB, mb1 - mb0), lane);
      cp_async_commit();
      cp_async_wait_all();
      __syncwarp();
      stage_payload(ring, bwcap, 0, 0, f.pay, f.codec, mb0, tmin<uint32_t>(TB, mb1 - mb0), lane);
      if (ntiles > 1) stage_headers(ring, 1, f.pg, f.codec, mb0 + TB, tmin<uint32_t>(TB, mb1 - mb0 - TB), lane);
      cp_async_commit();
    }
    uint32_t n = 0, seg_mb = mb0;
    for (uint32_t j = 0; j < ntiles; ++j) {
      const uint32_t i0 = mb0 + j * TB;
      const uint32_t nmb = tmin<uint32_t>(TB, mb1 - i0);
      const uint32_t row_base = (i0 - seg_mb) * kMB;
      if constexpr (kStage) {
        cp_async_wait_all();  // this tile's words and the next tile's headers have landed
        __syncwarp();
        const FirstCol f = first_col(Q, P);
        if (j + 1 < ntiles)
          stage_payload(ring, bwcap, (j + 1) % 3, (j + 1) % 2, f.pay, f.codec, i0 + TB,
                        tmin<uint32_t>(TB, mb1 - i0 - TB), lane);
        if (j + 2 < ntiles) {
          const uint32_t n2 = tmin<uint32_t>(TB, mb1 - i0 - 2 * TB);
          stage_headers(ring, (j + 2) % 3, f.pg, f.codec, i0 + 2 * TB, n2, lane);
          prefetch_other_headers(Q, P, f.c, i0 + 2 * TB, n2, lane);
        }
        cp_async_commit();
        const TileHdr H = staged_headers(ring, j % 3, f.c, f.codec, i0, nmb, lane);
        const StagedPay sp{stage_words(ring, j % 2, bwcap), stage_pw(bwcap), bwcap};
        if (gid0) n = tile_first_step<kHost, kText, true, true>(Q, P, H, i0, nmb, row_base, stab, list, n, lane, status, sp);
        else n = tile_first_step<kHost, kText, false, true>(Q, P, H, i0, nmb, row_base, stab, list, n, lane, status, sp);
      } else {
        const TileHdr H = load_headers<kHost>(Q, P, i0, nmb, lane);
        if (!kHost && Q.pf_step) prefetch_words(Q, P, H, Q.steps[1].col, nmb, lane);
        // without a staging ring its place holds the string search's scratch
        uint32_t* search = kText ? reinterpret_cast<uint32_t*>(ring) : nullptr;
        const StagedPay none{nullptr, 0, 0};
        if (gid0) n = tile_first_step<kHost, kText, true>(Q, P, H, i0, nmb, row_base, stab, list, n, lane, status, none, search);
        else n = tile_first_step<kHost, kText, false>(Q, P, H, i0, nmb, row_base, stab, list, n, lane, status, none, search);
      }
      const uint32_t next = i0 + TB;
      if (j + 1 == ntiles || n + kTileRows > kListCap || next + TB - seg_mb > kSegMbs) {
        n = list_steps<kHost, kText>(Q, P, seg_mb, list, n, stab, lane, status, 1);
        if (n) list_aggregate<kHost>(Q, P, seg_mb, list, n, lane, status);
        n = 0;
        seg_mb = next;
      }
    }
  }
}

// Copies a query's shared-memory join tables into the CTA's table region:
// open-addressing slots as they are, direct tables as 1/2/4-byte group-id
// contributions (all ones = absent) or presence bytes; builds the code-level
// matcher tables of string steps on FSST columns.
__device__ void load_smem_tables(const DevQuery& Q, uint8_t* stab) {
  for (uint32_t s = 0; s < Q.nsteps; ++s) {
    const DevStep& S = Q.steps[s];
    if ((S.kind == ST_PREFIX || S.kind == ST_CONTAINS) && S.smem_width != 0 && Q.cols[S.col].codec == C_FSST) {
      build_fsst_matcher(S, Q.cols[S.col].sym, Q.cols[S.col].nsym, stab + S.smem_off);
      continue;
    }
    if (S.kind != ST_PROBE || S.smem_width == 0) continue;
    if (S.ht_kind == HT_OPEN) {
      const uint2* src = static_cast<const uint2*>(S.ht);
      uint2* dst = reinterpret_cast<uint2*>(stab + S.smem_off);
      for (uint32_t i = threadIdx.x; i <= S.ht_mask; i += blockDim.x) dst[i] = __ldg(src + i);
      continue;
    }
    const uint32_t* src = static_cast<const uint32_t*>(S.ht);
    if (S.present) {  // eight coalesced loads together
      for (uint32_t i0 = threadIdx.x; i0 <= S.krange; i0 += 8 * blockDim.x) {
        uint32_t e[8];
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
          const uint32_t i = i0 + k * blockDim.x;
          e[k] = i < S.krange ? __ldg(src + i) : kAbsent;
        }
#pragma unroll
        for (uint32_t k = 0; k < 8; ++k) {
          const uint32_t i = i0 + k * blockDim.x;
          if (i <= S.krange) stab[S.smem_off + i] = e[k] != kAbsent;
        }
      }
      continue;
    }
    for (uint32_t i = threadIdx.x; i < S.krange; i += blockDim.x) {
      const uint32_t e = __ldg(src + i);
      const uint32_t c = (e & 0xffffu) * S.mul0 + (e >> 16) * S.mul1;
      if (S.smem_width == 1) stab[S.smem_off + i] = e == kAbsent ? 0xffu : uint8_t(c);
      else if (S.smem_width == 2)
        reinterpret_cast<uint16_t*>(stab + S.smem_off)[i] = e == kAbsent ? 0xffffu : uint16_t(c);
      else reinterpret_cast<uint32_t*>(stab + S.smem_off)[i] = e == kAbsent ? kAbsent : c;
    }
  }
}

// Batches: the warp's next ticket, from its CTA's run, or from another CTA's
// when that is used up.  A run's cost is an estimate, so the CTAs that finish
// early take over from those that hold most: the lanes look at 32 CTAs spread
// over the grid, and the one with the most tickets left is drawn from, unless it
// has no more than its own warps are about to draw.  Returns the ticket, or ~0
// when nothing is worth it.  The CTA's warps follow one another
// (CtaState::victim), so that they stay on one query.  Out of line: inside the
// loop over tickets it cost launches of one small query up to 1.5 us.
__device__ __noinline__ unsigned long long draw_batch(unsigned int* drawn, uint64_t owned, CtaState& cs, int lane) {
  unsigned long long t = ~0ull;
  if (lane == 0) {
    const uint32_t v = *const_cast<volatile unsigned int*>(&cs.victim);
    const uint64_t i = owned * v / gridDim.x + atomicAdd(drawn + v, 1u);
    if (i < owned * (v + 1) / gridDim.x) t = i;
  }
  t = __shfl_sync(kFull, t, 0);
  if (t != ~0ull) return t;
  for (uint32_t k = 1; k <= 4; ++k) {
    const uint32_t v = uint32_t((uint64_t(blockIdx.x) + k + uint64_t(lane) * gridDim.x / 32) % gridDim.x);
    const uint64_t v0 = owned * v / gridDim.x, v1 = owned * (v + 1) / gridDim.x;
    const uint32_t size = uint32_t(v1 - v0), x = __ldcg(drawn + v), left = size - tmin(size, x);
    const uint32_t best = __reduce_max_sync(kFull, left);
    if (best <= (blockDim.x >> 5)) return ~0ull;
    const int w = __ffs(__ballot_sync(kFull, left == best)) - 1;
    if (lane == w) {
      const uint32_t i = atomicAdd(drawn + v, 1u);
      if (i < size) {
        t = v0 + i;
        cs.victim = v;
      }
    }
    t = __shfl_sync(kFull, t, w);
    if (t != ~0ull) return t;
  }
  return ~0ull;
}

// kText = false: the build without the general string matcher (CONTAINS,
// FSST), launched for batches that have no such step.  kStage: the build
// with the staging ring (device-resident batches without such steps,
// launched when the tuning asks for staging).  kThreads: the largest CTA
// the build launches with (512- and 1,024-thread CTAs, 2 and 1 per SM, keep
// the 64 registers of the 4 x 256-thread build).
template <bool kHost, int kMinBlocks, bool kText, bool kStage = false, int kThreads = 256>
__global__ void __launch_bounds__(kThreads, kMinBlocks) fused_kernel(const DevQuery* __restrict__ queries,
                                                       const uint64_t* __restrict__ qbegin, int nq,
                                                       uint64_t owned, uint64_t pool, unsigned int* drawn, Sched* sched,
                                                       unsigned int* status_out, uint32_t acc_slots,
                                                       uint32_t tables_bytes, uint32_t stage_bw) {
  __shared__ CtaState cs;
  uint32_t* sacc = shared_acc();
  uint8_t* stab = dyn + ((acc_slots * sizeof(unsigned long long) + 15) & ~size_t(15));
  uint32_t* lists = reinterpret_cast<uint32_t*>(stab + tables_bytes);
  // Warps draw tickets on their own (one ticket = a range of rows of one
  // query, processed by one warp), so no CTA barrier separates tickets.  Each
  // CTA owns an equal share of the launch's `owned` tickets.  Of one query's it
  // is every gridDim-th one (a clustered table's skipped pages fall to every
  // CTA alike), drawn with a shared-memory counter, so a small launch's warps
  // need no global atomic.  Of a batch's it is a run, so that the CTA stays on
  // one query, or few, drawn with the CTA's counter in `drawn`, so that others
  // can take over (draw_batch).  Then the warps draw from the `pool` of small
  // tickets that all CTAs share (sched->next).  The CTA meets only when its warps' tickets
  // leave the current query: it flushes that query's accumulators and moves to
  // the smallest query any warp holds.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t* list = lists + uint32_t(warp) * kListCap;
  uint8_t* ring = reinterpret_cast<uint8_t*>(lists + nw * kListCap) +
                  size_t(warp) * (kText ? kSearchWords * sizeof(uint32_t) : stage_warp_bytes(stage_bw));
  if (threadIdx.x == 0) {
    cs.drawn = 0;
    cs.victim = blockIdx.x;
  }
  __syncthreads();
  // Draws the warp's next ticket: its query (INT_MAX: none left), and in t its
  // index among the query's tickets (owned ones first).  qbegin[0..nq] = each
  // query's first owned ticket, qbegin[nq + 1 ..] = its first pool ticket.
  auto draw = [&](unsigned long long& t) -> int {
    if (drawn != nullptr) {
      t = draw_batch(drawn, owned, cs, lane);
      if (t == ~0ull) return INT_MAX;
    } else {
      unsigned int x = 0;
      if (lane == 0) x = atomicAdd(&cs.drawn, 1u);
      x = __shfl_sync(kFull, x, 0);
      t = uint64_t(x) * gridDim.x + blockIdx.x;
    }
    const uint64_t* begin = qbegin;
    const bool mine = t < owned;
    if (!mine) {
      if (pool == 0) return INT_MAX;
      if (lane == 0) t = atomicAdd(&sched->next, 1ull);
      t = __shfl_sync(kFull, t, 0);
      if (t >= pool) return INT_MAX;
      begin += nq + 1;
    }
    int lo = 0, hi = nq - 1;  // last query with begin <= t
    while (lo < hi) {
      const int mid = (lo + hi + 1) / 2;
      if (__ldg(begin + mid) <= t) lo = mid; else hi = mid - 1;
    }
    if (nq > 1) t -= __ldg(begin + lo);
    if (!mine) t += nq > 1 ? __ldg(qbegin + lo + 1) - __ldg(qbegin + lo) : owned;
    return lo;
  };
  unsigned long long held;
  int hq = draw(held);
  int cur = -1;
  for (;;) {
    if (lane == 0) cs.wq[warp] = hq;
    __syncthreads();
    int next = INT_MAX;
    for (int w = 0; w < nw; ++w) next = min(next, cs.wq[w]);
    if (cur >= 0) finish_query(cs.q, cs.mine, cs);
    if (next == INT_MAX) break;
    {  // bring the query's plan into shared memory
      const uint4* src = reinterpret_cast<const uint4*>(queries + next);
      uint4* dst = reinterpret_cast<uint4*>(&cs.q);
      for (uint32_t i = threadIdx.x; i < sizeof(DevQuery) / 16; i += blockDim.x) dst[i] = __ldg(src + i);
    }
    if (threadIdx.x == 0) cs.mine = 0;
    __syncthreads();
    const DevQuery& Q = cs.q;
    if (Q.use_smem_acc) {
      const uint32_t n = 2 * Q.domain * (1 + Q.naggs);
      for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) sacc[i] = 0u;
    }
    load_smem_tables(Q, stab);
    __syncthreads();
    cur = next;
    uint32_t done_here = 0;
    while (hq == cur) {
      process_ticket<kHost, kText, kStage>(Q, held, stab, list, lane, &sched->status,
                                           ring);
      ++done_here;
      hq = draw(held);
    }
    if (lane == 0 && done_here) atomicAdd(&cs.mine, done_here);
  }
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned old = atomicAdd(&sched->exited, 1u);
    if (old == gridDim.x - 1) {
      sched->next = 0ull;
      sched->exited = 0u;
      if (drawn != nullptr)
        for (uint32_t i = 0; i < gridDim.x; ++i) drawn[i] = 0u;
      // every other CTA has left: the launch's status word, and a clean one for the next
      if (status_out) *status_out = atomicExch(&sched->status, 0u);
      __threadfence();
    }
  }
}


template <bool kHost, int kMinBlocks, bool kText, bool kStage = false, int kThreads = 256>
int occupancy_of(int threads, size_t smem) {
  int n = 0;
  auto* k = fused_kernel<kHost, kMinBlocks, kText, kStage, kThreads>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem);
  return n;
}

template <bool kHost, int kMinBlocks, bool kText, bool kStage = false, int kThreads = 256>
cudaError_t launch_as(const FusedLaunch& L, size_t smem, uint32_t tb, cudaStream_t s) {
  auto* k = fused_kernel<kHost, kMinBlocks, kText, kStage, kThreads>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (e != cudaSuccess) return e;
  k<<<L.grid, L.threads, smem, s>>>(
      L.queries, L.qbegin, L.nq, L.owned, L.pool, L.drawn, L.sched, L.status_out, L.acc_slots, tb, L.stage_bw);
  return cudaGetLastError();
}

}  // namespace
}  // namespace dpf
