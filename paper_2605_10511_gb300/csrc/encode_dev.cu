// Device-side loader: the page images that dpf_encode_column writes, byte for
// byte, made on the GPU from raw values in device memory (Sec. 4.2 data
// loader; Sec. 3.4.1 mini blocks; Sec. 3.4.2 variable-length pages).  A load
// is then one copy of the raw values over the host link and three small
// passes, instead of two passes over them on the host cores and an upload:
//  1. plan:  a warp per mini block finds its base, width (and string bytes);
//  2. pages: a CTA per page lays its mini blocks out, and finds the page's
//            size and value bounds, which the host reads back to place pages;
//  3. write: a warp per mini block packs it (and string bytes are moved).
// Bound by the calls around them (copies, allocations, the host's waits for
// the dictionary and the page sizes); each pass takes 5 to 25 us.  A mixed
// table of 2^20 rows (FOR, DELTA, DICT, FOR64 and 35 MB of strings), loaded
// and read back: 34.9 ms with the host encoder, 2.95 ms this way.
#include <climits>

#include "dpf_device.cuh"
#include "kernels.h"

namespace dpf {
namespace {

constexpr int kWarps = 8;  // per CTA

__device__ __forceinline__ uint64_t min_u64(uint64_t a, uint64_t b) { return a < b ? a : b; }

// Rows [a, a + cnt) of global mini block g.
__device__ __forceinline__ uint32_t mb_rows(const EncodeDev& E, uint64_t g, uint64_t* a) {
  const uint32_t per = E.page_rows / kMB;
  const uint64_t p = g / per, r0 = p * E.page_rows;
  *a = r0 + (g % per) * kMB;
  const uint64_t end = min_u64(E.nrows, r0 + E.page_rows);
  return uint32_t(min_u64(kMB, end - *a));
}

// The value that row j of a mini block packs, before its base is taken off
// (FOR / DICT: the value; DELTA: the wrapped difference with the row before,
// 0 for the first; STR: the length).
__device__ __forceinline__ uint32_t field32(const EncodeDev& E, uint64_t a, uint32_t j) {
  if (E.codec == C_STR) return uint32_t(E.offs[a + j + 1] - E.offs[a + j]);
  const uint32_t x = uint32_t(E.v32[a + j]);
  if (E.codec != C_DELTA) return x;
  return j == 0 ? 0u : x - uint32_t(E.v32[a + j - 1]);
}

__global__ void __launch_bounds__(32 * kWarps) plan_kernel(EncodeDev E) {
  const int lane = threadIdx.x & 31;
  for (uint64_t g = uint64_t(blockIdx.x) * kWarps + (threadIdx.x >> 5); g < E.nmb; g += uint64_t(gridDim.x) * kWarps) {
    uint64_t a;
    const uint32_t cnt = mb_rows(E, g, &a);
    EncodeMb m{0, 0, 0, 0};
    if (E.codec == C_FOR64) {
      long long lo = LLONG_MAX, hi = LLONG_MIN;
      for (uint32_t j = lane; j < cnt; j += 32) {
        const long long x = E.v64[a + j];
        lo = min(lo, x);
        hi = max(hi, x);
      }
      for (int d = 16; d > 0; d >>= 1) {
        lo = min(lo, __shfl_xor_sync(kFull, lo, d));
        hi = max(hi, __shfl_xor_sync(kFull, hi, d));
      }
      const unsigned long long span = (unsigned long long)hi - (unsigned long long)lo;
      m.base = int32_t(uint32_t((unsigned long long)lo));
      m.first = int32_t(uint32_t((unsigned long long)lo >> 32));
      m.bw = span == 0 ? 0u : 64u - uint32_t(__clzll((long long)span));
    } else if (E.codec == C_STR) {
      uint32_t lo = 0xffffffffu, hi = 0;
      unsigned long long sum = 0;
      bool bad = false;
      for (uint32_t j = lane; j < cnt; j += 32) {
        const unsigned long long o0 = E.offs[a + j], o1 = E.offs[a + j + 1];
        bad = bad || o1 < o0 || o1 - o0 > 0x7fffffffull;
        lo = min(lo, uint32_t(o1 - o0));
        hi = max(hi, uint32_t(o1 - o0));
        sum += o1 - o0;
      }
      for (int d = 16; d > 0; d >>= 1) sum += __shfl_xor_sync(kFull, sum, d);
      lo = __reduce_min_sync(kFull, lo);
      hi = __reduce_max_sync(kFull, hi);
      bad = __any_sync(kFull, bad) || sum > 0xffffffffull;
      m.base = int32_t(lo);
      m.bw = hi == lo ? 0u : 32u - uint32_t(__clz(int(hi - lo)));
      if (lane == 0) E.mb_bytes[g] = bad ? ~0ull : sum;
    } else {
      int32_t lo = INT32_MAX, hi = INT32_MIN;
      for (uint32_t j = lane; j < cnt; j += 32) {
        const int32_t x = int32_t(field32(E, a, j));
        lo = min(lo, x);
        hi = max(hi, x);
      }
      lo = __reduce_min_sync(kFull, lo);
      hi = __reduce_max_sync(kFull, hi);
      const uint32_t span = uint32_t(hi) - uint32_t(lo);
      m.base = lo;
      m.first = E.codec == C_DELTA ? E.v32[a] : 0;
      m.bw = span == 0 ? 0u : 32u - uint32_t(__clz(int(span)));
    }
    if (lane == 0) E.mb[g] = m;
  }
}

// Inclusive scan of x over the CTA's 256 threads; *total = the sum.
__device__ __forceinline__ unsigned long long block_scan(unsigned long long x, unsigned long long* total) {
  __shared__ unsigned long long part[kWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long y = __shfl_up_sync(kFull, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) part[warp] = x;
  __syncthreads();
  unsigned long long before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    if (w < warp) before += part[w];
    all += part[w];
  }
  __syncthreads();
  *total = all;
  return before + x;
}

__global__ void __launch_bounds__(32 * kWarps) page_kernel(EncodeDev E) {
  const uint64_t p = blockIdx.x, g0 = p * (E.page_rows / kMB);
  const uint32_t rows = uint32_t(min_u64(E.page_rows, E.nrows - p * E.page_rows)), nmb = (rows + kMB - 1) / kMB;
  unsigned long long words = 0, bytes = 0;
  long long lo = LLONG_MAX, hi = LLONG_MIN;
  uint32_t max_bw = 0;
  bool bad = false;
  for (uint32_t m0 = 0; m0 < nmb; m0 += 32 * kWarps) {
    const uint32_t m = m0 + threadIdx.x;
    const bool in = m < nmb;
    EncodeMb e{0, 0, 0, 0};
    if (in) e = E.mb[g0 + m];
    const unsigned long long w = in ? (E.codec == C_FOR64 ? 2ull : 4ull) * e.bw : 0ull;
    unsigned long long total;
    const unsigned long long wi = block_scan(w, &total);
    if (in) E.mb[g0 + m].word_off = uint32_t(words + wi - w);
    words += total;
    if (E.codec == C_STR) {
      const unsigned long long b = in ? E.mb_bytes[g0 + m] : 0ull;
      bad = bad || b == ~0ull;
      const unsigned long long use = b == ~0ull ? 0ull : b;
      const unsigned long long bi = block_scan(use, &total);
      if (in) E.mb_bytes[g0 + m] = bytes + bi - use;
      bytes += total;
    } else if (in && E.codec != C_FOR64) {  // value bounds of the page, as the loader derives them from headers
      const long long span = e.bw >= 32 ? 0xffffffffll : (1ll << e.bw) - 1;
      if (E.codec == C_DELTA) {
        lo = min(lo, (long long)e.first + 127 * min(0ll, (long long)e.base));
        hi = max(hi, (long long)e.first + 127 * max(0ll, (long long)e.base + span));
      } else {
        lo = min(lo, (long long)e.base);
        hi = max(hi, (long long)e.base + span);
      }
      max_bw = max(max_bw, e.bw);
    }
  }
  __shared__ long long s_lo[kWarps], s_hi[kWarps];
  __shared__ uint32_t s_bw[kWarps], s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  for (int d = 16; d > 0; d >>= 1) {
    lo = min(lo, __shfl_xor_sync(kFull, lo, d));
    hi = max(hi, __shfl_xor_sync(kFull, hi, d));
  }
  max_bw = __reduce_max_sync(kFull, max_bw);
  if (bad) s_bad = 1;
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo;
    s_hi[threadIdx.x >> 5] = hi;
    s_bw[threadIdx.x >> 5] = max_bw;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < kWarps; ++w) {
    lo = min(lo, s_lo[w]);
    hi = max(hi, s_hi[w]);
    max_bw = max(max_bw, s_bw[w]);
  }
  EncodePage q;
  const uint64_t end = payload_offset(E.codec, rows) + words * (E.codec == C_FOR64 ? 8 : 4);
  q.extra = E.codec == C_STR ? uint32_t(align16(end)) : 0u;
  q.bytes = E.codec == C_STR ? align16(align16(end) + bytes) : align16(end);
  q.lo = lo;
  q.hi = hi;
  q.max_bw = max_bw;
  q.bad = s_bad || bytes > 0xffffffffull || align16(end) > 0xffffffffull;
  E.pages[p] = q;
}

__global__ void __launch_bounds__(32 * kWarps) write_kernel(EncodeDev E) {
  __shared__ unsigned long long buf[kWarps][kMB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long* q = buf[warp];
  const uint32_t per = E.page_rows / kMB;
  for (uint64_t g = uint64_t(blockIdx.x) * kWarps + warp; g < E.nmb; g += uint64_t(gridDim.x) * kWarps) {
    uint64_t a;
    const uint32_t cnt = mb_rows(E, g, &a), m = uint32_t(g % per);
    const uint64_t p = g / per;
    const uint32_t rows = uint32_t(min_u64(E.page_rows, E.nrows - p * E.page_rows)), nmb = (rows + kMB - 1) / kMB;
    const EncodeMb e = E.mb[g];
    uint8_t* pg = E.blob + E.page_off[p];
    const uint32_t poff = payload_offset(E.codec, rows);
    if (lane == 0) {
      if (m == 0)
        *reinterpret_cast<uint4*>(pg) = make_uint4(kMagic | (E.codec << 24), rows, poff, E.codec == C_STR ? E.pages[p].extra : 0u);
      uint8_t* h = pg + kPageHdr + uint64_t(m) * mb_hdr_bytes(E.codec);
      const uint32_t wob = (e.word_off << 8) | e.bw;
      if (E.codec == C_FOR64) *reinterpret_cast<uint4*>(h) = make_uint4(uint32_t(e.base), uint32_t(e.first), e.word_off, e.bw);
      else if (E.codec == C_DELTA) *reinterpret_cast<uint4*>(h) = make_uint4(uint32_t(e.first), uint32_t(e.base), wob, 0u);
      else *reinterpret_cast<uint2*>(h) = make_uint2(uint32_t(e.base), wob);
      if (E.codec == C_STR)
        *reinterpret_cast<uint32_t*>(pg + kPageHdr + uint64_t(nmb) * 8 + uint64_t(m) * 4) = uint32_t(E.mb_bytes[g]);
    }
    const unsigned long long base64 = (unsigned long long)uint32_t(e.base) | ((unsigned long long)uint32_t(e.first) << 32);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t j = uint32_t(32 * k + lane);
      unsigned long long x = 0;  // rows past the page's last pack 0
      if (j < cnt)
        x = E.codec == C_FOR64 ? (unsigned long long)E.v64[a + j] - base64
                               : (unsigned long long)(field32(E, a, j) - uint32_t(e.base));
      q[j] = x;
    }
    __syncwarp();
    // a lane per packed word: the fields that overlap its bits, LSB first
    const uint32_t bits = E.codec == C_FOR64 ? 64u : 32u, nw = kMB * e.bw / bits;
    for (uint32_t w = lane; w < nw; w += 32) {
      const uint32_t first = w * bits;
      unsigned long long x = 0;
      for (uint32_t j = first / e.bw; j < kMB && j * e.bw < first + bits; ++j) {
        const uint32_t at = j * e.bw;
        x |= at >= first ? q[j] << (at - first) : q[j] >> (first - at);
      }
      if (bits == 64) reinterpret_cast<unsigned long long*>(pg + poff)[e.word_off + w] = x;
      else reinterpret_cast<uint32_t*>(pg + poff)[e.word_off + w] = uint32_t(x);
    }
    __syncwarp();
  }
}

// String bytes of page blockIdx.x into its byte region (16-aligned): a thread
// per 16 bytes, read as aligned words and shifted to the source's alignment.
__global__ void copy_strings(EncodeDev E) {
  const uint64_t p = blockIdx.x, r0 = p * E.page_rows, r1 = min_u64(E.nrows, r0 + E.page_rows);
  const uint64_t from = E.offs[r0] - E.offs[0], n = E.offs[r1] - E.offs[r0];
  uint8_t* dst = E.blob + E.page_off[p] + E.pages[p].extra;
  const uint8_t* src = E.bytes + from;
  const uint32_t sh = 8 * uint32_t(reinterpret_cast<uintptr_t>(src) & 3u);
  const uint32_t* w = reinterpret_cast<const uint32_t*>(src - sh / 8);
  const uint64_t chunks = (n + 15) / 16;
  for (uint64_t c = uint64_t(blockIdx.y) * blockDim.x + threadIdx.x; c < chunks; c += uint64_t(gridDim.y) * blockDim.x) {
    if (16 * c + 16 > n) {  // the last, partial chunk: byte by byte (zeros follow it)
      for (uint64_t i = 16 * c; i < n; ++i) dst[i] = src[i];
      continue;
    }
    uint32_t x[5];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = __ldg(w + 4 * c + i);
    x[4] = sh ? __ldg(w + 4 * c + 4) : 0u;
    reinterpret_cast<uint4*>(dst)[c] = make_uint4(__funnelshift_r(x[0], x[1], sh), __funnelshift_r(x[1], x[2], sh),
                                                  __funnelshift_r(x[2], x[3], sh), __funnelshift_r(x[3], x[4], sh));
  }
}

// ---- dictionaries: the distinct values as a bitmap over [lo, lo + range)
__global__ void minmax_kernel(const int32_t* v, uint64_t n, uint32_t* hi, uint32_t* lo) {
  uint32_t a = 0, b = 0;  // BuildStat's ranks: the largest rank and the largest ~rank
  for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t r = BuildStat::rank(__ldg(v + i));
    a = max(a, r);
    b = max(b, ~r);
  }
  a = __reduce_max_sync(kFull, a);
  b = __reduce_max_sync(kFull, b);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(hi, a);
    atomicMax(lo, b);
  }
}

__global__ void mark_kernel(const int32_t* v, uint64_t n, int32_t lo, uint32_t* bitmap) {
  for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t off = uint32_t(__ldg(v + i)) - uint32_t(lo), bit = 1u << (off & 31u);
    if (!(bitmap[off >> 5] & bit)) atomicOr(bitmap + (off >> 5), bit);  // a stale word costs one atomic more
  }
}

// One CTA: each word's rank (values below it), the values in ascending order
// (at most cap are written) and, in *count, how many there are.
__global__ void __launch_bounds__(32 * kWarps) rank_values(const uint32_t* bitmap, uint32_t nwords, int32_t lo,
                                                           uint32_t* rank, int32_t* values, uint32_t cap,
                                                           unsigned long long* count) {
  unsigned long long carry = 0;
  for (uint32_t w0 = 0; w0 < nwords; w0 += 32 * kWarps) {
    const uint32_t w = w0 + threadIdx.x;
    uint32_t x = w < nwords ? bitmap[w] : 0u;
    unsigned long long total;
    const uint32_t n = uint32_t(__popc(x));
    unsigned long long at = carry + block_scan(n, &total) - n;
    if (w < nwords) rank[w] = uint32_t(at);
    for (; x; x &= x - 1, ++at)
      if (at < cap) values[at] = int32_t(uint32_t(lo) + w * 32u + uint32_t(__ffs(x) - 1));
    carry += total;
  }
  if (threadIdx.x == 0) *count = carry;
}

__global__ void codes_kernel(int32_t* v, uint64_t n, int32_t lo, const uint32_t* bitmap, const uint32_t* rank) {
  for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += uint64_t(gridDim.x) * blockDim.x) {
    const uint32_t off = uint32_t(v[i]) - uint32_t(lo);
    v[i] = int32_t(rank[off >> 5] + uint32_t(__popc(bitmap[off >> 5] & ((1u << (off & 31u)) - 1u))));
  }
}

int grid_of(uint64_t items, uint64_t per_block) {
  return int(tmin<uint64_t>(tmax<uint64_t>((items + per_block - 1) / per_block, 1), 152ull * 16));
}

}  // namespace

cudaError_t launch_encode_plan(const EncodeDev& E, cudaStream_t s) {
  plan_kernel<<<grid_of(E.nmb, kWarps), 32 * kWarps, 0, s>>>(E);
  page_kernel<<<unsigned(E.npages), 32 * kWarps, 0, s>>>(E);
  return cudaGetLastError();
}

cudaError_t launch_encode_write(const EncodeDev& E, cudaStream_t s) {
  write_kernel<<<grid_of(E.nmb, kWarps), 32 * kWarps, 0, s>>>(E);
  if (E.codec == C_STR) {
    const unsigned y = unsigned(tmin<uint64_t>(16, tmax<uint64_t>(1, 152ull * 8 / E.npages)));
    copy_strings<<<dim3(unsigned(E.npages), y), 256, 0, s>>>(E);
  }
  return cudaGetLastError();
}

cudaError_t launch_dict_range(const int32_t* v, uint64_t n, uint32_t* hi, uint32_t* lo, cudaStream_t s) {
  minmax_kernel<<<grid_of(n, 256 * 8), 256, 0, s>>>(v, n, hi, lo);
  return cudaGetLastError();
}

cudaError_t launch_dict_values(const int32_t* v, uint64_t n, int32_t lo, uint32_t nwords, uint32_t* bitmap, uint32_t* rank,
                               int32_t* values, uint32_t cap, unsigned long long* count, cudaStream_t s) {
  mark_kernel<<<grid_of(n, 256 * 8), 256, 0, s>>>(v, n, lo, bitmap);
  rank_values<<<1, 32 * kWarps, 0, s>>>(bitmap, nwords, lo, rank, values, cap, count);
  return cudaGetLastError();
}

cudaError_t launch_dict_codes(int32_t* v, uint64_t n, int32_t lo, const uint32_t* bitmap, const uint32_t* rank,
                              cudaStream_t s) {
  codes_kernel<<<grid_of(n, 256 * 8), 256, 0, s>>>(v, n, lo, bitmap, rank);
  return cudaGetLastError();
}

}  // namespace dpf
