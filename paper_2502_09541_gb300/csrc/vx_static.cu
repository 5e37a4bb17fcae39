// Allocation-free variant of the ordered filter (vx_filter_device_static).
//
// Some callers cannot let a library allocate device memory: code that runs
// inside another framework's memory manager, which owns all device memory and
// hands out only the input and output buffers of each call, and
// latency-critical paths where a cudaMalloc or cudaFree (which may synchronise
// the device) is not acceptable.  For them this entry point keeps its scratch
// — one look-back word per tile, tickets and the total — in one file-scope
// __device__ array of fixed size instead of an arena.  Every GPU that loads the
// library holds that array (kStaticScratchWords 32-bit words, 256 KiB + 256 B)
// until the process exits.
//
// Host code must not pass the array's name to a kernel: on the host the name
// is a stand-in object, not a device address, and a kernel given it would
// fault or, where the GPU can reach host memory, silently use the wrong
// memory.  The device address is looked up once per device with
// cudaGetSymbolAddress (with that device current) and passed to the kernels.
#include <mutex>

#include "vx_internal.h"

namespace vx {

constexpr uint64_t kStaticMaxRows = 1ull << 26;  // rows per call (67,108,864)
constexpr int kSfThreads = 256;
constexpr int kSfWarps = kSfThreads / 32;
constexpr uint32_t kSfGroupRows = kSfThreads * 4;  // a group: four consecutive rows of every thread
// Groups per tile, and when the tiles' prefixes come from a scan block instead
// of each tile's own look-back.  Whole calls measured, rows x columns (share
// qualifying), tiles of 4 / 8 / 16 groups with the scan block:
//   1,000,003 x 2 (0.5)      24.6 /  24.9 /  28.9 us; 29 us with look-backs
//   8,388,608 x 4 (0.8)      60.3 /  66.1 /  69.3 us; 88 us with look-backs
//   67,107,861 x 3 (0.02)   183   / 170   / 171 us;  270 us with look-backs
//   67,108,864 x 2 (0.001)  141   / 123   / 113 us;  232 us with look-backs
// so tiles are small while they are few thousand, and large above.  With at
// most 32 tiles a look-back is a single window and the scan block would only add
// a hand-over (10,007 rows: 21 us).
constexpr int kSfSmall = 4, kSfLarge = 16;
constexpr uint64_t kSfLargeRows = 1ull << 24;
constexpr uint32_t kSfLookBackTiles = 32;
constexpr uint32_t kStaticMaxTiles = (uint32_t)(kStaticMaxRows / (kSfSmall * kSfGroupRows));  // at most: 16,384
constexpr uint32_t kStaticScratchWords = 65536 + 64;
// scratch: the tiles' look-back words (64 bits each), then from kSfControl on
// the tickets (call number and count) and the result: count, error (64 bits each)
constexpr uint32_t kSfControl = 65536;
constexpr uint32_t kSfSpinLimit = 1u << 20;  // polls of a window of predecessor words before giving up
// Polls after which a tile stops counting on the scan block and looks back
// itself (about 0.1 ms; a tile of a call that has the GPU waits some 10 us), and
// after which the scan block gives its place up (about 50 ms: it waits for
// tiles that may not have started, which only costs time where it holds the
// last free place).
constexpr uint32_t kSfOwnPolls = 128, kSfScanPolls = 1u << 16;
static_assert(2 * kStaticMaxTiles <= kSfControl, "a look-back word per tile");
static_assert(kSfLarge * kSfGroupRows <= 65536, "tile rows fit 16 bits");

// Shared by every call on a device.  Look-back words and tickets count only if
// they carry the call's own number, and later calls have larger numbers, so
// nothing has to be cleared between calls (after 2^35 of them everything is).
static __device__ __align__(256) uint32_t g_filter_scratch[kStaticScratchWords];

namespace {

// a predicate as one range test: (uint32)(v - lo) <= span, complemented if neg
struct SfParams {
  int n_preds;
  const int32_t *col[VX_MAX_PREDS];
  uint32_t lo[VX_MAX_PREDS], span[VX_MAX_PREDS], neg[VX_MAX_PREDS];
  uint64_t row0, n, cap;
  uint64_t call;       // number of this call, in bits 29.. of its look-back words
  uint64_t *result;    // [0] count, [1] nonzero: a look-back wait gave up
  uint32_t n_tiles;
};

// look-back word: call number (35 bits) | flag (2) | value (27: at most 2^26)
constexpr uint32_t kSfAgg = 1, kSfIncl = 2;
constexpr uint64_t kSfCalls = 1ull << 35;
__device__ __forceinline__ uint64_t sf_word(uint64_t call, uint32_t flag, uint32_t v) {
  return call << 29 | (uint64_t)flag << 27 | v;
}
__device__ __forceinline__ uint32_t sf_flag(uint64_t w, uint64_t call) {
  return w >> 29 == call ? (uint32_t)(w >> 27) & 3u : 0u;
}
__device__ __forceinline__ uint32_t sf_value(uint64_t w) { return (uint32_t)w & ((1u << 27) - 1u); }

// Survivors in the tiles before `tile`, by one warp: a window of 32
// predecessors at a time (the nearest in lane 0), up to the nearest tile whose
// word holds the count of everything up to itself.
__device__ __forceinline__ uint32_t sf_look_back(const volatile uint64_t *words, uint64_t call, uint32_t tile,
                                                 uint32_t lane, bool *gave_up) {
  uint32_t prefix = 0;
  for (int64_t base = (int64_t)tile - 1; base >= 0; base -= 32) {
    const int64_t t = base - lane;
    for (uint32_t polls = 0;; ++polls) {
      const uint64_t w = t >= 0 ? words[t] : sf_word(call, kSfIncl, 0);  // before the first tile: nothing
      const uint32_t flag = sf_flag(w, call);
      const uint32_t have = __ballot_sync(0xffffffffu, flag != 0), inc = __ballot_sync(0xffffffffu, flag == kSfIncl);
      const uint32_t need = inc ? (inc & -inc) | ((inc & -inc) - 1u) : 0xffffffffu;
      if ((have & need) == need) {  // every word up to the nearest inclusive one is there
        prefix += __reduce_add_sync(0xffffffffu, need >> lane & 1u ? sf_value(w) : 0u);
        if (inc) return prefix;
        break;
      }
      if (polls > kSfSpinLimit) {
        *gave_up = true;
        return prefix;
      }
    }
  }
  return prefix;
}

// The scan block of a call with many tiles: its warps take windows of 32
// tiles in turn, wait for the tiles' words, add their counts up behind the window
// before (a carry handed from warp to warp in shared memory) and replace every
// word by the count of everything up to the tile, so that the prefixes advance by
// a window per hand-over instead of a window per round trip to memory.  A tile
// that has looked back itself has left that count already.
__device__ __forceinline__ void sf_scan_block(const SfParams &p, volatile uint64_t *words) {
  // carry into window k at [k % 16], tagged with k + 1 (at most 8 windows are in work)
  __shared__ uint64_t s_carry[2 * kSfWarps];
  if (threadIdx.x < 2 * kSfWarps) s_carry[threadIdx.x] = threadIdx.x == 0 ? 1ull << 32 : 0ull;
  __syncthreads();
  volatile uint64_t *carry = s_carry;
  constexpr uint32_t kWhole = 1u << 31;  // the sum counts from the first tile on, not from the window's
  const uint32_t lane = threadIdx.x & 31, n_win = (p.n_tiles + 31) / 32;
  for (uint32_t k = threadIdx.x >> 5; k < n_win; k += kSfWarps) {
    const uint32_t t = 32 * k + lane;
    uint32_t x = 0;
    for (uint32_t polls = 0;; ++polls) {
      const uint64_t w = t < p.n_tiles ? words[t] : sf_word(p.call, kSfAgg, 0);
      const uint32_t flag = sf_flag(w, p.call);
      x = sf_value(w) | (flag == kSfIncl ? kWhole : 0u);
      if (__all_sync(0xffffffffu, flag != 0)) break;
      if (polls > kSfScanPolls) return;  // the tiles manage without
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o && !(x & kWhole)) x += y;
    }
    uint64_t c = carry[k % (2 * kSfWarps)];
    for (uint32_t polls = 0; (uint32_t)(c >> 32) != k + 1; c = carry[k % (2 * kSfWarps)])
      if (++polls > 64 * kSfScanPolls) return;
    x = x & kWhole ? x & ~kWhole : (uint32_t)c + x;
    __syncwarp();
    if (lane == 31) carry[(k + 1) % (2 * kSfWarps)] = (uint64_t)(k + 2) << 32 | x;
    if (t < p.n_tiles) words[t] = sf_word(p.call, kSfIncl, x);
  }
}

// Ordered filter in one pass.  What bounds it is reading the predicate columns
// once.  A tile per block (taken by ticket, so that a tile only ever waits for
// tiles that already run): each thread tests kG groups of four consecutive
// rows with one 16-byte load per group and column, the loads of four groups
// issued together, and a column after the first is read only where a row of the
// group still qualifies.  Survivor counts are scanned over the block (four
// groups' counts packed into one word per thread) and staged in shared memory
// in order; the tile's first output position comes from a look-back over its
// predecessors' words, or with kScan from the block with the first ticket, which
// does nothing but turn the tiles' counts into prefixes; then the survivors leave
// as one contiguous run.  The scan block works on whole windows, whose later
// tiles may not have a place on the GPU yet, so a tile whose prefix does not come
// looks back itself: no tile needs one that has not started.  Three columns of
// 2^26 rows, 2 % qualifying: 171 us for the call, of which 20 us are not the
// kernel (5.4 TB/s, 0.79 of the measured copy bandwidth); 907 us when a count pass,
// a scan of the tiles and a write pass read the columns twice in 4-byte loads.
// 10,007 rows, two columns: 21 us, 42 us before.
template <bool kVec, int kG, bool kScan>
__global__ void __launch_bounds__(kSfThreads) sf_filter_kernel(const SfParams p, uint32_t *scratch, uint64_t *out) {
  constexpr int kB = kG / 4;  // batches of four groups
  __shared__ uint32_t s_tile;
  __shared__ uint32_t s_cnt[kG * kSfWarps];  // survivors before (group, warp) in the tile
  __shared__ uint32_t s_prefix, s_total;
  __shared__ uint16_t s_row[kG * kSfGroupRows];
  unsigned long long *ticket = (unsigned long long *)(scratch + kSfControl);
  if (threadIdx.x == 0) {
    atomicMax(ticket, (unsigned long long)p.call << 20);
    const uint64_t t = atomicAdd(ticket, 1ull);
    s_tile = t >> 20 == p.call ? (uint32_t)t & 0xFFFFFu : 0xFFFFFu;
  }
  __syncthreads();
  if (s_tile >= p.n_tiles + (kScan ? 1 : 0)) {  // another call's tickets: calls must not overlap
    if (threadIdx.x == 0) p.result[1] = 1;
    return;
  }
  volatile uint64_t *words = (volatile uint64_t *)scratch;
  if (kScan && s_tile == 0) {
    sf_scan_block(p, words);
    return;
  }
  const uint32_t tile = kScan ? s_tile - 1 : s_tile, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t t0 = tile * (kG * kSfGroupRows), n = (uint32_t)p.n;  // n is at most 2^26
  uint32_t keep[kB];    // 4 bits per group: rows that qualify
  uint32_t before[kB];  // 8 bits per group: survivors of the warp's lower lanes
#pragma unroll
  for (int b = 0; b < kB; ++b) {
    const uint32_t r0 = t0 + b * 4 * kSfGroupRows + threadIdx.x * 4;
    uint32_t alive[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const uint32_t r = r0 + g * kSfGroupRows;
      alive[g] = r + 4 <= n ? 0xFu : r < n ? (1u << (n - r)) - 1u : 0u;
    }
    for (int q = 0; q < p.n_preds; ++q) {
      const int32_t *c = p.col[q];
      int4 v[4];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const uint32_t r = r0 + g * kSfGroupRows;
        v[g] = make_int4(0, 0, 0, 0);
        if (kVec && r + 4 <= n) {
          if (alive[g]) v[g] = __ldg(reinterpret_cast<const int4 *>(c + r));
        } else {
          if (alive[g] & 1u) v[g].x = __ldg(c + r);
          if (alive[g] & 2u) v[g].y = __ldg(c + r + 1);
          if (alive[g] & 4u) v[g].z = __ldg(c + r + 2);
          if (alive[g] & 8u) v[g].w = __ldg(c + r + 3);
        }
      }
      const uint32_t lo = p.lo[q], span = p.span[q], neg = p.neg[q];
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const uint32_t in =
            (uint32_t)((uint32_t)v[g].x - lo <= span) | (uint32_t)((uint32_t)v[g].y - lo <= span) << 1 |
            (uint32_t)((uint32_t)v[g].z - lo <= span) << 2 | (uint32_t)((uint32_t)v[g].w - lo <= span) << 3;
        alive[g] &= neg ? ~in : in;
      }
    }
    keep[b] = alive[0] | alive[1] << 4 | alive[2] << 8 | alive[3] << 12;
    uint32_t own = 0;  // four counts of at most 128 over the warp
#pragma unroll
    for (int g = 0; g < 4; ++g) own |= __popc(alive[g]) << (8 * g);
    uint32_t incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= (uint32_t)o) incl += y;
    }
    before[b] = incl - own;
    if (lane == 31)
#pragma unroll
      for (int g = 0; g < 4; ++g) s_cnt[(4 * b + g) * kSfWarps + warp] = incl >> (8 * g) & 0xFFu;
  }
  __syncthreads();
  if (warp == 0) {
    uint32_t total = 0;
#pragma unroll
    for (int k = 0; k < kG * kSfWarps / 32; ++k) {
      const uint32_t c = s_cnt[32 * k + lane];
      uint32_t x = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
      }
      s_cnt[32 * k + lane] = total + x - c;
      total += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) {
      s_total = total;
      words[tile] = sf_word(p.call, tile ? kSfAgg : kSfIncl, total);
    }
    if (!kScan) {
      bool gave_up = false;
      const uint32_t prefix = sf_look_back(words, p.call, tile, lane, &gave_up);
      if (lane == 0) {
        if (tile) words[tile] = sf_word(p.call, kSfIncl, (prefix + total) & ((1u << 27) - 1u));
        if (gave_up) p.result[1] = 1;
        if (tile == p.n_tiles - 1) p.result[0] = prefix + total;
        s_prefix = prefix;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < kB; ++b)
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      uint32_t at = s_cnt[(4 * b + g) * kSfWarps + warp] + (before[b] >> (8 * g) & 0xFFu);
      const uint32_t r = (4 * b + g) * kSfGroupRows + threadIdx.x * 4;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (keep[b] >> (4 * g + j) & 1u) s_row[at++] = (uint16_t)(r + j);
    }
  if (kScan && warp == 0) {
    const uint32_t total = s_total;
    uint64_t w = 0;
    for (uint32_t polls = 0; polls < kSfOwnPolls; ++polls) {
      w = __shfl_sync(0xffffffffu, words[tile], 0);
      if (sf_flag(w, p.call) == kSfIncl) break;
      __nanosleep(200);
    }
    uint32_t prefix = sf_value(w) - total;
    if (sf_flag(w, p.call) != kSfIncl) {
      bool gave_up = false;
      prefix = sf_look_back(words, p.call, tile, lane, &gave_up);
      if (lane == 0) {
        if (gave_up) {
          p.result[1] = 1;
          s_total = 0;  // nothing is written
        } else {
          words[tile] = sf_word(p.call, kSfIncl, prefix + total);
        }
      }
    }
    if (lane == 0) {
      if (tile == p.n_tiles - 1) p.result[0] = prefix + total;
      s_prefix = prefix;
    }
  }
  __syncthreads();
  const uint64_t pos0 = s_prefix;
  const uint32_t m = pos0 >= p.cap ? 0 : (uint32_t)(p.cap - pos0 < s_total ? p.cap - pos0 : s_total);
  const uint64_t id0 = p.row0 + t0;
  for (uint32_t i = threadIdx.x; i < m; i += kSfThreads) out[pos0 + i] = id0 + s_row[i];
}

// device address of g_filter_scratch and whether the GPU writes pageable host
// memory, looked up once per device, and the number of the device's last call
std::mutex g_addr_mu;
uint32_t *g_addr[64] = {};
uint64_t g_calls[64] = {};
int g_pageable[64] = {};  // the device accesses pageable host memory through the host's page tables
// Where a device with g_pageable stores the last call's count and error.  They
// outlive the call: a kernel whose call returned early (a wait for the stream
// that failed, say because the stream is being captured) may still store them.
struct alignas(64) HostResult {
  volatile uint64_t w[2];
};
HostResult g_result[64];

vx_status scratch_address(uint32_t **out, uint64_t *call, volatile uint64_t **host_res) {
  int dev = 0;
  VX_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("vx_filter_device_static: device ordinal %d out of range", dev);
    return VX_E_UNSUPPORTED;
  }
  std::lock_guard<std::mutex> g(g_addr_mu);
  if (!g_addr[dev]) {
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_filter_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      set_error("vx_filter_device_static: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
      return VX_E_CUDA;
    }
    VX_CUDA_TRY(cudaDeviceGetAttribute(&g_pageable[dev], cudaDevAttrPageableMemoryAccessUsesHostPageTables, dev));
    g_addr[dev] = (uint32_t *)p;
  }
  *out = g_addr[dev];
  *host_res = g_pageable[dev] ? g_result[dev].w : nullptr;
  *call = g_calls[dev] = (g_calls[dev] + 1) % kSfCalls;
  return VX_OK;
}

// v passes op: (uint32)(v - lo) <= span, complemented if neg
void range_of(const vx_pred &q, uint32_t *lo, uint32_t *span, uint32_t *neg) {
  int64_t a = INT32_MIN, b = INT32_MAX;
  *neg = 0;
  switch (q.op) {
    case VX_BETWEEN: a = q.lo, b = q.hi; break;
    case VX_NE: *neg = 1;  // fall through: complement of EQ
    case VX_EQ: a = b = q.lo; break;
    case VX_LT: b = (int64_t)q.lo - 1; break;
    case VX_LE: b = q.lo; break;
    case VX_GT: a = (int64_t)q.lo + 1; break;
    case VX_GE: a = q.lo; break;
  }
  if (a > b) {  // no value passes
    a = INT32_MIN;
    b = INT32_MAX;
    *neg = 1;
  }
  *lo = (uint32_t)a;
  *span = (uint32_t)(b - a);
}

}  // namespace
}  // namespace vx

using namespace vx;

VX_API vx_status vx_filter_device_static(const int32_t *const *cols, int32_t n_cols, const vx_pred *preds,
                                         int32_t n_preds, uint64_t n_rows, uint64_t row0, uint64_t *out_rows,
                                         uint64_t cap, uint64_t *out_count, void *stream) {
  clear_error();
  if (!cols || !preds || !out_count || n_cols < 1 || n_preds < 1 || n_preds > VX_MAX_PREDS || (cap && !out_rows)) {
    set_error("vx_filter_device_static: bad argument");
    return VX_E_INVAL;
  }
  if (n_rows > kStaticMaxRows) {
    set_error("vx_filter_device_static: %llu rows exceed the static scratch limit of %llu rows per call",
              (unsigned long long)n_rows, (unsigned long long)kStaticMaxRows);
    return VX_E_INVAL;
  }
  SfParams p{};
  bool vec = true;  // 16-byte loads need every column on a 16-byte boundary
  p.n_preds = n_preds;
  for (int q = 0; q < n_preds; ++q) {
    if (preds[q].col < 0 || preds[q].col >= n_cols || !cols[preds[q].col] || preds[q].op < VX_BETWEEN ||
        preds[q].op > VX_GE) {
      set_error("vx_filter_device_static: predicate %d: bad column index or op", q);
      return VX_E_INVAL;
    }
    p.col[q] = cols[preds[q].col];
    range_of(preds[q], &p.lo[q], &p.span[q], &p.neg[q]);
    vec = vec && ((uintptr_t)p.col[q] & 15) == 0;
  }
  p.row0 = row0;
  p.n = n_rows;
  p.cap = cap;
  *out_count = 0;
  if (n_rows == 0) return VX_OK;
  uint32_t *scratch = nullptr;
  volatile uint64_t *host_res = nullptr;
  VX_TRY(scratch_address(&scratch, &p.call, &host_res));
  cudaStream_t s = (cudaStream_t)stream;
  if (p.call == 0) VX_CUDA_TRY(cudaMemsetAsync(scratch, 0, 4ull * kStaticScratchWords, s));  // the numbers start again
  const bool large = n_rows > kSfLargeRows;
  const uint64_t tile = (large ? kSfLarge : kSfSmall) * kSfGroupRows;
  p.n_tiles = (uint32_t)((n_rows + tile - 1) / tile);
  const bool scan = p.n_tiles > kSfLookBackTiles;
  // the kernel writes the count to host memory itself where the GPU reads and
  // writes pageable host memory through the host's page tables (a copy of 16
  // bytes back from the device took 8 us more of a 21 us call)
  if (host_res) host_res[0] = host_res[1] = 0;
  p.result = host_res ? (uint64_t *)host_res : (uint64_t *)(scratch + kSfControl + 4);
  auto kernel = large  ? (vec ? sf_filter_kernel<true, kSfLarge, true> : sf_filter_kernel<false, kSfLarge, true>)
                : scan ? (vec ? sf_filter_kernel<true, kSfSmall, true> : sf_filter_kernel<false, kSfSmall, true>)
                       : (vec ? sf_filter_kernel<true, kSfSmall, false> : sf_filter_kernel<false, kSfSmall, false>);
  cudaGetLastError();  // an error that an earlier call of this thread left is not this launch's
  kernel<<<p.n_tiles + (scan ? 1 : 0), kSfThreads, 0, s>>>(p, scratch, out_rows);
  VX_CUDA_TRY(cudaGetLastError());
  uint64_t res[2] = {0, 0};
  if (!host_res) VX_CUDA_TRY(cudaMemcpyAsync(res, p.result, sizeof res, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  const uint64_t total = host_res ? host_res[0] : res[0];
  if (host_res ? host_res[1] : res[1]) {
    if (!host_res) VX_CUDA_TRY(cudaMemsetAsync(p.result, 0, sizeof res, s));
    set_error("vx_filter_device_static: a look-back wait gave up");
    return VX_E_TIMEOUT;
  }
  *out_count = total;
  if (total > cap) {
    set_error("vx_filter_device_static: %llu rows qualify; capacity %llu", (unsigned long long)total,
              (unsigned long long)cap);
    return VX_E_CAPACITY;
  }
  return VX_OK;
}
