// Out-of-core sort: range partition + per-partition LSD radix sort.
//
// Section 6.1 sorts chunks and merges them; here the partition step comes
// first (the two-phase layout of Section 6.2.1: per-chunk clustering with a
// boundary array, then per-group processing of the multi-extent partitions),
// with a monotone range function so that sorted partitions concatenate into
// the sorted output:
//   pass 1 (ExKernel over input chunks): stable scatter of each chunk by
//           partition id into a host intermediate at the chunk's own offset,
//           plus the chunk's P+1 boundary array;
//   pass 2 (ExKernel over partitions): gather partition p's extents (one per
//           chunk), LSD radix sort in HBM, store at the partition's final
//           offset.
// Both passes run on the pipelined executor, so host->device loads and
// device->host stores overlap with the kernels.  Partitions of one key value
// are already in input order and are copied through; a multi-key partition
// above the slot capacity is sorted recursively.
#include <algorithm>
#include <cstddef>
#include <deque>
#include <cmath>
#include <thread>

#include "vx_internal.h"
#include "vx_prefix.cuh"
#include "vx_radix.cuh"
#include "vx_sort.cuh"

namespace vx {

// ================================================================== kernels

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// partition of a key: the number of splitters <= key
__device__ __forceinline__ uint32_t key_range(uint64_t k, const uint64_t *s_spl, int n_spl) {
  int lo = 0, hi = n_spl;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (s_spl[mid] <= k) lo = mid + 1;
    else hi = mid;
  }
  return (uint32_t)lo;
}

__global__ void __launch_bounds__(kRxThreads) rx_upsweep(const uint64_t *__restrict__ keys, uint64_t n,
                                                         const uint64_t *spl, int n_spl, uint32_t *hist,
                                                         uint32_t ntiles) {
  __shared__ uint32_t wcnt[kRxWarps][kRxDigits];
  __shared__ uint64_t s_spl[kRxDigits];
  for (int i = threadIdx.x; i < kRxWarps * kRxDigits; i += blockDim.x) (&wcnt[0][0])[i] = 0;
  for (int i = threadIdx.x; i < n_spl; i += blockDim.x) s_spl[i] = spl[i];
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t wbase = (uint64_t)blockIdx.x * kRxTile + (uint64_t)w * (32 * kRxItems);
#pragma unroll 4
  for (int r = 0; r < kRxItems; ++r) {
    const uint64_t i = wbase + (uint64_t)r * 32 + lane;
    if (i < n) atomicAdd(&wcnt[w][key_range(keys[i], s_spl, n_spl)], 1u);  // counting needs no order
  }
  __syncthreads();
  for (int d = threadIdx.x; d < kRxDigits; d += blockDim.x) {
    uint32_t s = 0;
    for (int q = 0; q < kRxWarps; ++q) s += wcnt[q][d];
    hist[(uint64_t)d * ntiles + blockIdx.x] = s;
  }
}

// block d: exclusive scan of hist[d][0..ntiles) in place; row total -> totals[d]
__global__ void __launch_bounds__(1024) rx_scan_rows(uint32_t *hist, uint32_t ntiles, RadixState *st) {
  __shared__ uint32_t wsum[32];
  __shared__ uint64_t carry;
  uint32_t *row = hist + (uint64_t)blockIdx.x * ntiles;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (uint32_t base = 0; base < ntiles; base += blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    const uint32_t v = i < ntiles ? row[i] : 0;
    uint32_t x = v;
    for (int off = 1; off < 32; off <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
      if ((threadIdx.x & 31) >= (unsigned)off) x += y;
    }
    if ((threadIdx.x & 31) == 31) wsum[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) {
      uint32_t wv = threadIdx.x < (blockDim.x >> 5) ? wsum[threadIdx.x] : 0;
      for (int off = 1; off < 32; off <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, wv, off);
        if (threadIdx.x >= (unsigned)off) wv += y;
      }
      wsum[threadIdx.x] = wv;
    }
    __syncthreads();
    const uint32_t wpre = (threadIdx.x >> 5) ? wsum[(threadIdx.x >> 5) - 1] : 0;
    if (i < ntiles) row[i] = (uint32_t)carry + wpre + x - v;
    __syncthreads();
    if (threadIdx.x == 0) carry += wsum[(blockDim.x >> 5) - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) st->totals[blockIdx.x] = carry;
}

// one block of 256 threads: partition starts (exclusive scan of totals,
// base[256] = n)
__global__ void __launch_bounds__(kRxDigits) rx_scan_totals(RadixState *st, uint64_t n) {
  __shared__ uint64_t s[kRxDigits];
  const int d = threadIdx.x;
  const uint64_t t = st->totals[d];
  s[d] = t;
  __syncthreads();
  for (int off = 1; off < kRxDigits; off <<= 1) {
    uint64_t y = d >= off ? s[d - off] : 0;
    __syncthreads();
    s[d] += y;
    __syncthreads();
  }
  st->base[d] = s[d] - t;
  if (d == 0) st->base[kRxDigits] = n;
}

// Resident partitions: where each partition's region of the arena starts, how
// many pairs it takes and how many it holds.
struct RxRegions {
  uint64_t off[kRxDigits], cap[kRxDigits], used[kRxDigits];
  uint64_t dest[kRxDigits];  // of the chunk in work: position of the partition's first pair
  uint32_t full;             // a region was too small: nothing is scattered any more
};

// one block of 256 threads: the chunk's partitions go behind what their
// regions hold
__global__ void __launch_bounds__(kRxDigits) rx_place(const RadixState *st, RxRegions *rg, uint32_t P) {
  const uint32_t d = threadIdx.x;
  const uint64_t t = d < P ? st->totals[d] : 0, u = d < P ? rg->used[d] : 0;
  const int over = __syncthreads_or(d < P && t > rg->cap[d] - u);
  if (over) {
    if (d == 0) rg->full = 1;
    return;
  }
  if (d < P) {
    rg->dest[d] = rg->off[d] + u;
    rg->used[d] = u + t;
  }
}

// histograms of the key bytes kFirst .. kFirst + kP - 1 in one read (constant
// digits are skipped later)
template <int kP, int kFirst = 0>
__global__ void __launch_bounds__(kRxThreads) rx_byte_hist(const uint64_t *__restrict__ keys, uint64_t n,
                                                           unsigned long long *bh) {
  __shared__ uint32_t h[kP][kRxDigits];
  for (int i = threadIdx.x; i < kP * kRxDigits; i += blockDim.x) (&h[0][0])[i] = 0;
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  for (; i + 3 * stride < n; i += 4 * stride) {
    uint64_t k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) k[u] = keys[i + u * stride];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int p = 0; p < kP; ++p) atomicAdd(&h[p][(k[u] >> (8 * (kFirst + p))) & 0xFF], 1u);
  }
  for (; i < n; i += stride)
#pragma unroll
    for (int p = 0; p < kP; ++p) atomicAdd(&h[p][(keys[i] >> (8 * (kFirst + p))) & 0xFF], 1u);
  __syncthreads();
  for (int i = threadIdx.x; i < kP * kRxDigits; i += blockDim.x)
    if ((&h[0][0])[i]) atomicAdd(&bh[kFirst * kRxDigits + i], (unsigned long long)(&h[0][0])[i]);
}

// one block of 256 threads per LSD pass: exclusive scan of the pass's digit
// histogram (the global position of each digit's first pair) and whether one
// digit holds all n pairs (the pass is skipped)
__global__ void __launch_bounds__(kRxDigits) rx_init(RadixState *st, const unsigned long long *bh, uint64_t *bases,
                                                     uint64_t n, uint32_t spin_limit, int first) {
  __shared__ uint64_t wsum[kRxDigits / 32];
  const int p = first + blockIdx.x, d = threadIdx.x, lane = d & 31, w = d >> 5;
  const uint64_t t = bh[p * kRxDigits + d];
  uint64_t x = t;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[w] = x;
  const int full = __syncthreads_or(t == n);
  for (int q = 0; q < w; ++q) x += wsum[q];
  bases[p * kRxDigits + d] = x - t;
  if (d == 0) {
    st->skip[p] = full;
    if (p == first) {
      for (int q = 0; q < first; ++q) st->skip[q] = 1;
      st->cur[first] = 0;
      st->err = st->n_fix = st->redo = 0;
      st->spin_limit = spin_limit;
    }
  }
}

// dynamic shared memory of the scatter: the tile's pairs regrouped by digit
// (keys, values, digits), per-warp digit counters, per-digit offsets
struct RxScatterSmem {
  uint64_t k[kRxTile];
  uint32_t v[kRxTile];
  uint32_t wcnt[kRxWarps][kRxDigits];
  uint64_t off[kRxDigits];  // global position of local position 0 of each digit
  uint32_t tstart[kRxDigits];
  uint32_t wsum[kRxWarps];
  uint8_t d[kRxTile];
};

// One-sweep LSD passes: per-(tile, digit) status words carry a flag (0 not
// ready, 1 the tile's own count, 2 the inclusive prefix over tiles 0..t), the
// pass number (so one clearing serves all eight passes) and the value.
constexpr uint64_t kRxFlagAgg = 1ull << 62, kRxFlagIncl = 2ull << 62;
constexpr uint64_t kRxValueMask = (1ull << 59) - 1;
constexpr uint32_t kRxSpinLimit = 1u << 20;  // polls of one predecessor word before giving up

__device__ __forceinline__ uint64_t rx_status_word(uint64_t flag, int pass, uint64_t value) {
  return flag | (uint64_t)pass << 59 | value;
}

// Stable scatter of one tile: rank every pair inside its warp (match_any over
// 16 rounds of 32 consecutive pairs), regroup the tile by digit in shared
// memory, then write each digit's run with consecutive threads on consecutive
// output positions, so stores leave the SM as contiguous runs.
// The tile's digit offsets come from the scanned per-tile histograms, behind
// the partitions' starts in the chunk (rg null) or in their regions.
__global__ void __launch_bounds__(kRxThreads, 2) rx_range_scatter(RadixBufs b, const RadixState *st, uint64_t n,
                                                                  const uint64_t *spl, int n_spl, const uint32_t *hist,
                                                                  uint32_t ntiles, const RxRegions *rg) {
  if (rg && rg->full) return;
  extern __shared__ __align__(16) unsigned char rx_smem[];
  RxScatterSmem &sm = *reinterpret_cast<RxScatterSmem *>(rx_smem);
  __shared__ uint64_t s_spl[kRxDigits];
  const uint64_t *kin = b.keys[0];
  const uint32_t *vin = b.vals[0];
  uint64_t *kout = b.keys[1];
  uint32_t *vout = b.vals[1];
  for (int i = threadIdx.x; i < kRxWarps * kRxDigits; i += blockDim.x) (&sm.wcnt[0][0])[i] = 0;
  for (int i = threadIdx.x; i < n_spl; i += blockDim.x) s_spl[i] = spl[i];
  __syncthreads();
  const uint32_t tile = blockIdx.x;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t tbase = (uint64_t)tile * kRxTile;
  const uint64_t wbase = tbase + (uint64_t)w * (32 * kRxItems);
  uint64_t k[kRxItems];
  uint32_t v[kRxItems], dr[kRxItems];  // dr = rank inside the warp << 9 | digit
#pragma unroll
  for (int r = 0; r < kRxItems; ++r) {
    const uint64_t i = wbase + (uint64_t)r * 32 + lane;
    k[r] = i < n ? kin[i] : 0;
    v[r] = i < n ? vin[i] : 0;
  }
#pragma unroll
  for (int r = 0; r < kRxItems; ++r) {
    const uint64_t i = wbase + (uint64_t)r * 32 + lane;
    const uint32_t d = i < n ? key_range(k[r], s_spl, n_spl) : kRxInvalid;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    uint32_t before = 0;
    if (d != kRxInvalid) before = sm.wcnt[w][d];
    __syncwarp();
    dr[r] = (before + __popc(peers & lanemask_lt())) << 9 | d;
    if (d != kRxInvalid && lane == (uint32_t)(__ffs(peers) - 1)) sm.wcnt[w][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {  // thread d: warp offsets within digit d, then the tile's digit starts (exclusive scan over digits)
    const int d = threadIdx.x;
    uint32_t run = 0;
#pragma unroll
    for (int q = 0; q < kRxWarps; ++q) {
      const uint32_t cq = sm.wcnt[q][d];
      sm.wcnt[q][d] = run;
      run += cq;
    }
    // position of the tile's first pair of digit d
    const uint64_t before_tile =
        d <= n_spl ? (rg ? rg->dest[d] : st->base[d]) + hist[(uint64_t)d * ntiles + tile] : 0;
    uint32_t x = run;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, off);
      if (lane >= (uint32_t)off) x += y;
    }
    if (lane == 31) sm.wsum[w] = x;
    __syncthreads();
    uint32_t wpre = 0;
#pragma unroll
    for (int q = 0; q < kRxWarps; ++q) wpre += q < (int)w ? sm.wsum[q] : 0u;
    const uint32_t excl = wpre + x - run;
    sm.tstart[d] = excl;
    sm.off[d] = before_tile - excl;  // wraps back when added to a position
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kRxItems; ++r) {
    const uint32_t d = dr[r] & 0x1FFu;
    if (d == kRxInvalid) continue;
    const uint32_t lp = sm.tstart[d] + sm.wcnt[w][d] + (dr[r] >> 9);
    sm.k[lp] = k[r];
    sm.v[lp] = v[r];
    sm.d[lp] = (uint8_t)d;
  }
  __syncthreads();
  const uint32_t valid = n - tbase < (uint64_t)kRxTile ? (uint32_t)(n - tbase) : (uint32_t)kRxTile;
  for (uint32_t t = threadIdx.x; t < valid; t += blockDim.x) {
    const uint64_t pos = sm.off[sm.d[t]] + t;
    kout[pos] = sm.k[t];
    vout[pos] = sm.v[t];
  }
}

// Lanes of the warp with the same 8-bit digit, from one vote per bit
// (match_any takes a step per distinct value, about 30 of them for random
// digits: 0.98 against 0.74 ms for the eight passes over 9.6M random pairs,
// and 0.70 with the matches found through shared-memory words, which falls to
// 0.78 on skewed digits where votes take 0.69).
__device__ __forceinline__ uint32_t same_digit(uint32_t d) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const uint32_t on = (uint32_t)((int32_t)(d << (31 - b)) >> 31);  // all ones where the bit is set
    peers &= ~(__ballot_sync(0xffffffffu, on != 0) ^ on);
  }
  return peers;
}

// One LSD pass: a stable scatter of the pairs by one key byte.  The tile is
// the block's ticket; its digits' positions come from the one-read histogram
// (bases) plus a look-back over the status words of the tiles before it.
//   rank: a warp owns kI * 32 consecutive pairs.  The lanes of a round that
// share a digit find one another (same_digit), their first lane adds them to the
// warp's counter of the digit and hands the count before them to the others;
// the rounds' matches and shared-memory atomics are issued back to back, so
// that the warp waits for one round trip per kB rounds and not for each.
//   place: keys are regrouped by digit in shared memory while the tiles before
// publish, then written as runs of consecutive positions; the values follow
// through the same shared memory.  Holding only one of the two at a time lets
// 28 warps share an SM, which the latencies here need.
// Bound by shared-memory wavefronts, barriers and issue rather than by HBM: 24
// bytes a pair and pass at 3.25 TB/s (0.48 of the measured copy bandwidth, 40M
// pairs); 1.67 TB/s before, when every round waited for its match_any and its
// counter, and keys and values together left 16 warps an SM.
template <int kT, int kI, class Off>
struct RxSweepSmem {
  uint64_t k[kT * kI];                 // the keys by digit, then the values
  uint32_t wcnt[kT / 32][kRxDigits];
  Off off[kRxDigits];  // global position of local position 0 of each digit
  uint32_t wsum[kRxDigits / 32];
  uint32_t tile;
};

template <int kT, int kI, class Off>
__global__ void __launch_bounds__(kT, 2) rx_sweep(RadixBufs b, RadixState *st, int pass, uint64_t n,
                                                          const uint64_t *bases, unsigned int *tickets,
                                                          unsigned long long *status, bool iota) {
  constexpr int kTile = kT * kI, kB = 4;
  static_assert(kT >= kRxDigits && kI % kB == 0 && kTile <= 65536, "a thread per digit, whole batches, 16-bit places");
  if (st->skip[pass]) {
    if (blockIdx.x == 0 && threadIdx.x == 0) st->cur[pass + 1] = st->cur[pass];
    return;
  }
  extern __shared__ __align__(16) unsigned char rx_smem[];
  RxSweepSmem<kT, kI, Off> &sm = *reinterpret_cast<RxSweepSmem<kT, kI, Off> *>(rx_smem);
  const int c = st->cur[pass];
  if (threadIdx.x == 0) sm.tile = atomicAdd(&tickets[pass], 1u);
  for (int i = threadIdx.x; i < kT / 32 * kRxDigits; i += kT) (&sm.wcnt[0][0])[i] = 0;
  __syncthreads();
  const uint32_t tile = sm.tile;
  if (tile == 0 && threadIdx.x == 0) st->cur[pass + 1] = 1 - c;  // read by the next pass only
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t tbase = (uint64_t)tile * kTile;
  const uint32_t valid = n - tbase < (uint64_t)kTile ? (uint32_t)(n - tbase) : (uint32_t)kTile;
  const uint32_t first = w * (32 * kI) + lane;  // the thread's pairs: first + 32 r of the tile
  const uint64_t *kin = (c ? b.keys[1] : b.keys[0]) + tbase;
  auto digit = [&](uint64_t k) { return __byte_perm((uint32_t)k, (uint32_t)(k >> 32), pass) & 0xFFu; };
  // keys past the end are all ones: the last pairs of the tile's last digit
  uint64_t k[kI];
#pragma unroll
  for (int r = 0; r < kI; ++r) k[r] = first + 32 * r < valid ? kin[first + 32 * r] : ~0ull;
  // rank inside the warp's pairs of the digit, then the place in the tile: two
  // 16-bit ones per word (registers are what limits the warps here)
  uint32_t place[kI / 2];
#pragma unroll
  for (int r0 = 0; r0 < kI; r0 += kB) {
    uint32_t peers[kB], before[kB];
#pragma unroll
    for (int r = 0; r < kB; ++r) peers[r] = same_digit(digit(k[r0 + r]));
#pragma unroll
    for (int r = 0; r < kB; ++r) {
      before[r] = 0;
      if ((peers[r] & lanemask_lt()) == 0) before[r] = atomicAdd(&sm.wcnt[w][digit(k[r0 + r])], __popc(peers[r]));
      __syncwarp();
    }
#pragma unroll
    for (int r = 0; r < kB; ++r) {
      const uint32_t rank =
          __shfl_sync(0xffffffffu, before[r], __ffs(peers[r]) - 1) + __popc(peers[r] & lanemask_lt());
      place[(r0 + r) / 2] = r % 2 ? place[(r0 + r) / 2] | rank << 16 : rank;
    }
  }
  __syncthreads();
  const uint32_t d = threadIdx.x;
  uint32_t run = 0, start = 0;  // the tile's pairs of digit d, their first place
  volatile unsigned long long *sw = status + (uint64_t)tile * kRxDigits + d;
  uint32_t cnt[kT / 32];
  if (d < kRxDigits) {
#pragma unroll
    for (int q = 0; q < kT / 32; ++q) {
      cnt[q] = sm.wcnt[q][d];
      run += cnt[q];
    }
    uint32_t x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) sm.wsum[w] = x;
    start = x - run;
    if (d == kRxDigits - 1) run -= kTile - valid;
    *sw = rx_status_word(tile == 0 ? kRxFlagIncl : kRxFlagAgg, pass, run);
  }
  __syncthreads();
  if (d < kRxDigits) {  // where each warp's pairs of the digit go
#pragma unroll
    for (int q = 0; q < kRxDigits / 32; ++q) start += q < (int)w ? sm.wsum[q] : 0u;
    uint32_t at = start;
#pragma unroll
    for (int q = 0; q < kT / 32; ++q) {
      sm.wcnt[q][d] = at;
      at += cnt[q];
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kI; ++r) {
    place[r / 2] += sm.wcnt[w][digit(k[r])] << (r % 2 * 16);
    sm.k[r % 2 ? place[r / 2] >> 16 : place[r / 2] & 0xFFFFu] = k[r];
  }
  const uint32_t *vin = (c ? b.vals[1] : b.vals[0]) + tbase;
  uint32_t v[kI];
  if (iota)  // the values are the positions, which nobody has written, until a pass has moved them
    for (int q = 0; q < pass; ++q) iota = iota && st->skip[q];
#pragma unroll
  for (int r = 0; r < kI; ++r)
    v[r] = iota ? (uint32_t)tbase + first + 32 * r : first + 32 * r < valid ? vin[first + 32 * r] : 0u;
  if (d < kRxDigits) {
    uint64_t prefix = 0;  // pairs of digit d in the tiles before this one
    const uint32_t limit = st->spin_limit;
    bool done = tile == 0;
    for (uint32_t t = tile; !done;) {  // look back over the predecessors' words, kL of them read at once
      constexpr uint32_t kL = 4;
      uint64_t word[kL];
#pragma unroll
      for (uint32_t j = 0; j < kL; ++j)
        word[j] = *(const volatile unsigned long long *)(status + (uint64_t)(t > j ? t - 1 - j : 0) * kRxDigits + d);
#pragma unroll
      for (uint32_t j = 0; j < kL; ++j) {
        if (done) break;
        uint32_t spins = 0;
        while ((word[j] >> 62) == 0 || (int)((word[j] >> 59) & 7u) != pass) {
          // give up after the limit, or at once when another tile already gave up
          if (++spins > limit || ((spins & 1023u) == 0 && *(volatile uint32_t *)&st->err)) {
            spins = limit + 1;
            break;
          }
          __nanosleep(32);
          word[j] = *(const volatile unsigned long long *)(status + (uint64_t)(t - 1 - j) * kRxDigits + d);
        }
        if (spins > limit) {  // a predecessor never published: report, keep going (a partial
                              // prefix only lowers this tile's positions, all inside the pass's n)
          atomicOr(&st->err, 1u);
          done = true;
          break;
        }
        prefix += word[j] & kRxValueMask;
        done = (word[j] >> 62) == 2;  // tile 0's word is always inclusive
      }
      t = t > kL ? t - kL : 0;
      if (t == 0) done = true;
    }
    if (tile > 0) *sw = rx_status_word(kRxFlagIncl, pass, prefix + run);
    sm.off[d] = (Off)(bases[pass * kRxDigits + d] + prefix - start);  // wraps back when added to a position
  }
  __syncthreads();
  uint64_t *kout = c ? b.keys[0] : b.keys[1];
  uint32_t *vout = c ? b.vals[0] : b.vals[1];
  uint32_t dg[kI / 4];  // the digits of the places this thread writes
#pragma unroll
  for (int j = 0; j < kI; ++j) {
    const uint32_t t = threadIdx.x + j * kT;
    const uint64_t key = sm.k[t];
    const uint32_t g = digit(key);
    dg[j / 4] = j % 4 ? dg[j / 4] | g << (8 * (j % 4)) : g;
    if (t < valid) kout[(Off)(sm.off[g] + t)] = key;
  }
  __syncthreads();
  uint32_t *sv = reinterpret_cast<uint32_t *>(sm.k);
#pragma unroll
  for (int r = 0; r < kI; ++r) sv[r % 2 ? place[r / 2] >> 16 : place[r / 2] & 0xFFFFu] = v[r];
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kI; ++j) {
    const uint32_t t = threadIdx.x + j * kT;
    if (t < valid) vout[(Off)(sm.off[dg[j / 4] >> (8 * (j % 4)) & 0xFFu] + t)] = sv[t];
  }
}

constexpr size_t kRxScatterSmem = sizeof(RxScatterSmem);

// 14 warps a block, two blocks an SM, 72 registers a thread: eight passes over
// 9.6M / 40M random pairs take 0.666 / 2.36 ms; 512 x 2 (64 registers, spilling
// more) 0.683 / 2.40, 384 x 3 0.750 / 2.59, 256 x 4 0.723 / 2.48.  16 pairs a
// thread, or 8 while that leaves no SM a second block: a small sort's time is a
// tile's chain of steps (8 passes over 100K / 500K pairs take 0.103 / 0.123 ms
// with 8, 0.119 / 0.142 with 16; over 1M 0.160 and 0.158).
constexpr int kSweepThreads = 448;
constexpr uint32_t kSweepTile = kSweepThreads * 16, kSweepSmallTile = kSweepThreads * 8;
constexpr uint32_t kSweepSmallTiles = 160;  // small tiles a sort may have, by num_sms or at most so many

static bool sweep_small(uint64_t n, int num_sms) {
  return n <= (uint64_t)kSweepSmallTile * std::min<uint32_t>(num_sms, kSweepSmallTiles);
}
static uint32_t sweep_tiles(uint64_t n, int num_sms) {
  const uint32_t t = sweep_small(n, num_sms) ? kSweepSmallTile : kSweepTile;
  return (uint32_t)((n + t - 1) / t);
}

template <int kI, class Off>
static vx_status launch_sweep(RadixBufs b, RadixState *st, int pass, uint64_t n, const uint64_t *bases,
                              unsigned int *tickets, unsigned long long *status, bool iota, uint32_t tiles,
                              cudaStream_t s) {
  constexpr size_t smem = sizeof(RxSweepSmem<kSweepThreads, kI, Off>);
  static OncePerDevice once;
  VX_TRY(raise_smem_limit(once, rx_sweep<kSweepThreads, kI, Off>, smem));
  rx_sweep<kSweepThreads, kI, Off><<<tiles, kSweepThreads, smem, s>>>(b, st, pass, n, bases, tickets, status, iota);
  return VX_OK;
}

// one pass; positions take 32 bits below 2^32 pairs
static vx_status enqueue_sweep(RadixBufs b, RadixState *st, int pass, uint64_t n, const uint64_t *bases,
                               unsigned int *tickets, unsigned long long *status, bool iota, int num_sms,
                               cudaStream_t s) {
  const uint32_t nt = sweep_tiles(n, num_sms);
  if (sweep_small(n, num_sms)) return launch_sweep<8, uint32_t>(b, st, pass, n, bases, tickets, status, iota, nt, s);
  if (n >> 32) return launch_sweep<16, uint64_t>(b, st, pass, n, bases, tickets, status, iota, nt, s);
  return launch_sweep<16, uint32_t>(b, st, pass, n, bases, tickets, status, iota, nt, s);
}

static vx_status rx_scatter_attr() {
  static OncePerDevice once;
  return raise_smem_limit(once, rx_range_scatter, kRxScatterSmem);
}

// publishes the buffer holding the result (low byte), the number of
// executed (not skipped) passes (next byte) and the error word (bit 16) to a
// mapped host word
__global__ void rx_publish(const RadixState *st, int pass, uint64_t *host_word) {
  uint64_t executed = 0;
  for (int p = 0; p < pass; ++p) executed += st->skip[p] ? 0u : 1u;
  *host_word = (uint64_t)st->cur[pass] | executed << 8 | (uint64_t)(st->err != 0) << 16 |
               (uint64_t)(st->redo != 0) << 17;
}

// ---- prefix sort: what the passes over the upper key bytes left out of order
// (vx_prefix.cuh)

// lists the first pair of every group to repair; a group of more than kFixGroup
// pairs, or a full list, asks for the sort in full
__global__ void rx_find_kernel(const RadixBufs b, RadixState *st, uint64_t n, int shift, uint32_t *list, uint32_t cap) {
  const uint64_t *k = st->cur[8] ? b.keys[1] : b.keys[0];
  for (PrefixWalk w{blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, n, (uint64_t)gridDim.x * blockDim.x}; w.more();
       w.next()) {
    uint64_t first = 0;
    const PrefixFind what = prefix_find(k, n, w.i, shift, &first);
    if (what == kFixNone) continue;
    const uint32_t at = what == kFixList ? atomicAdd(&st->n_fix, 1u) : cap;
    if (at < cap) list[at] = (uint32_t)first;
    else st->redo = 1;
  }
}

// a thread per listed group
__global__ void rx_fix_kernel(const RadixBufs b, const RadixState *st, uint64_t n, int shift, const uint32_t *list,
                              uint32_t cap) {
  uint64_t *k = st->cur[8] ? b.keys[1] : b.keys[0];
  uint32_t *v = st->cur[8] ? b.vals[1] : b.vals[0];
  const uint32_t m = st->n_fix < cap ? st->n_fix : cap;
  for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < m; q += (uint64_t)gridDim.x * blockDim.x)
    prefix_fix(k, v, n, list[q], shift);
}

// ---- sampling and splitters -----------------------------------------------

// key of sample i at position mix64(base + i) mod n (the library's own
// counter-based positions), read through mapped host memory
__device__ __forceinline__ uint64_t mix64_dev(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void sample_keys_kernel(const uint64_t *keys, uint64_t n, uint64_t m, uint64_t seed, uint64_t *out,
                                   uint32_t *out_vals) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t pos = mix64_dev(seed * 0x9E3779B97F4A7C15ull + i) % n;
    out[i] = keys[pos];
    out_vals[i] = (uint32_t)i;
  }
}

// rank[i] = number of sample keys below splitter i (lower bound in the sorted
// sample): partition p (keys in [spl[p-1], spl[p])) holds rank[p] - rank[p-1]
// of the m sample keys
__global__ void sample_ranks_kernel(const uint64_t *sorted, uint64_t m, const uint64_t *spl, uint32_t n_spl,
                                    uint64_t *rank) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_spl; i += gridDim.x * blockDim.x) {
    uint64_t lo = 0, hi = m;
    while (lo < hi) {
      const uint64_t mid = (lo + hi) >> 1;
      if (sorted[mid] < spl[i]) lo = mid + 1;
      else hi = mid;
    }
    rank[i] = lo;
  }
}

// out[0] / out[1]: neighbours of the sorted sample that differ but agree in
// their upper four / five bytes; out[2]: keys that occur eight times or more;
// out[3]: equal neighbours
__global__ void sample_prefix_kernel(const uint64_t *sorted, uint64_t m, unsigned long long *out) {
  uint32_t c4 = 0, c5 = 0, heavy = 0, same = 0;
  for (uint64_t i = 1 + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t a = sorted[i - 1], b = sorted[i];
    c4 += a != b && a >> 32 == b >> 32;
    c5 += a != b && a >> 24 == b >> 24;
    heavy += i >= 7 && sorted[i - 7] == b;
    same += a == b;
  }
  c4 = __reduce_add_sync(0xffffffffu, c4);
  c5 = __reduce_add_sync(0xffffffffu, c5);
  heavy = __reduce_add_sync(0xffffffffu, heavy);
  same = __reduce_add_sync(0xffffffffu, same);
  if ((threadIdx.x & 31) == 0) {
    if (c4) atomicAdd(&out[0], (unsigned long long)c4);
    if (c5) atomicAdd(&out[1], (unsigned long long)c5);
    if (heavy) atomicAdd(&out[2], (unsigned long long)heavy);
    if (same) atomicAdd(&out[3], (unsigned long long)same);
  }
}

// The same counts for keys that have not been sampled: one block hashes m rows
// spread over the n into shared memory, once by the whole key, then its distinct
// keys by their upper five bytes and those distinct in that by their upper four.
constexpr uint32_t kPairSample = 4096, kPairSlots = 2 * kPairSample;
struct PairSampleSmem {
  unsigned long long slot[kPairSlots];
  uint32_t count[kPairSlots];
  uint32_t out[4];
};
__global__ void __launch_bounds__(1024) pair_prefix_kernel(const uint64_t *keys, uint64_t n, uint32_t m, uint64_t *out) {
  extern __shared__ __align__(16) unsigned char pair_smem[];
  PairSampleSmem &sm = *reinterpret_cast<PairSampleSmem *>(pair_smem);
  constexpr int kPer = kPairSample / 1024;
  constexpr unsigned long long kNone = ~0ull;
  unsigned long long k[kPer];
  bool live[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const uint32_t i = threadIdx.x + j * 1024;
    live[j] = i < m;
    k[j] = live[j] ? keys[(uint64_t)i * n / m] : 0;
    if (k[j] == kNone) --k[j];  // the empty slot's word
  }
  if (threadIdx.x < 4) sm.out[threadIdx.x] = 0;
  for (uint32_t i = threadIdx.x; i < kPairSlots; i += 1024) sm.count[i] = 0;
#pragma unroll 1
  for (int round = 0; round < 3; ++round) {
    const int shift = round == 0 ? 0 : round == 1 ? 24 : 32;
    for (uint32_t i = threadIdx.x; i < kPairSlots; i += 1024) sm.slot[i] = kNone;
    __syncthreads();
    uint32_t repeats = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      if (!live[j]) continue;
      const unsigned long long x = k[j] >> shift;
      uint32_t h = (uint32_t)((x * 0x9E3779B97F4A7C15ull) >> 40) % kPairSlots;
      for (;;) {  // at most half of the slots are taken
        const unsigned long long was = atomicCAS(&sm.slot[h], kNone, x);
        if (was == kNone) break;
        if (was == x) {
          if (round == 0 && atomicAdd(&sm.count[h], 1u) == 6) atomicAdd(&sm.out[2], 1u);
          ++repeats;
          live[j] = false;
          break;
        }
        h = (h + 1) % kPairSlots;
      }
    }
    repeats = __reduce_add_sync(0xffffffffu, repeats);
    if ((threadIdx.x & 31) == 0 && repeats) atomicAdd(&sm.out[round == 0 ? 3 : round == 1 ? 1 : 0], repeats);
    __syncthreads();
  }
  // keys that agree in five bytes agree in four
  if (threadIdx.x < 4) out[threadIdx.x] = sm.out[threadIdx.x] + (threadIdx.x == 0 ? sm.out[1] : 0u);
}

// splitters from the sorted sample: s_p = sample[p*m/P]
__global__ void sample_splitters_kernel(const uint64_t *sorted, uint64_t m, uint32_t P, uint64_t *spl) {
  for (uint32_t p = 1 + blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x)
    spl[p - 1] = sorted[(uint64_t)p * m / P];
}

// piecewise-linear CDF model: knot j = sorted[j*(m-1)/S], CDF(knot j) = j/S;
// splitter p = model inverse at p/P, exact integer interpolation
__global__ void pl_knots_kernel(const uint64_t *sorted, uint64_t m, uint32_t S, uint64_t *knots) {
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j <= S; j += gridDim.x * blockDim.x)
    knots[j] = sorted[(uint64_t)j * (m - 1) / S];
}

__global__ void pl_splitters_kernel(const uint64_t *knots, uint32_t S, uint32_t P, uint64_t *spl) {
  for (uint32_t p = 1 + blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
    const uint64_t num = (uint64_t)p * S;
    const uint64_t j = num / P, rem = num % P;
    if (j >= S) {
      spl[p - 1] = knots[S];
      continue;
    }
    const uint64_t gap = knots[j + 1] - knots[j];
    // floor(gap * rem / P) without 128-bit arithmetic: gap = q*P + r
    spl[p - 1] = knots[j] + (gap / P) * rem + ((gap % P) * rem) / P;
  }
}

// Keys of the sorted sample that occur at least m / (2P) times (up to cap of
// them, in no particular order; *n counts them all).  Thread i looks at run
// starts only and finds the run's end by binary search.
__global__ void heavy_keys_kernel(const uint64_t *sorted, uint64_t m, uint32_t P, uint64_t *keys, uint32_t *n,
                                  uint32_t cap) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t v = sorted[i];
    if (i > 0 && sorted[i - 1] == v) continue;
    uint64_t a = i, b = m;  // first index with sorted[] > v
    while (a < b) {
      const uint64_t mid = (a + b) >> 1;
      if (sorted[mid] <= v) a = mid + 1;
      else b = mid;
    }
    if ((a - i) * 2 * (uint64_t)P >= m) {
      const uint32_t j = atomicAdd(n, 1u);
      if (j < cap) keys[j] = v;
    }
  }
}

// raw (n_raw non-decreasing splitters of a smooth model) merged with the heavy
// keys (sorted here, at most cap_heavy of them), duplicates dropped, at most
// cap_out entries: every heavy key becomes a splitter, so the isolation below
// gives it a partition of its own as the sample's quantiles do.  One thread.
__global__ void merge_heavy_kernel(const uint64_t *raw, uint32_t n_raw, uint64_t *heavy, const uint32_t *n_heavy,
                                   uint32_t cap_heavy, uint64_t *out, uint32_t *n_out, uint32_t cap_out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const uint32_t nh = *n_heavy < cap_heavy ? *n_heavy : cap_heavy;
  for (uint32_t i = 1; i < nh; ++i) {  // insertion sort of a few dozen keys
    const uint64_t x = heavy[i];
    uint32_t j = i;
    while (j > 0 && heavy[j - 1] > x) {
      heavy[j] = heavy[j - 1];
      --j;
    }
    heavy[j] = x;
  }
  uint32_t a = 0, b = 0, k = 0;
  // the model's splitters all stay; heavy keys fill what room is left
  uint32_t room = cap_out > n_raw ? cap_out - n_raw : 0;
  while ((a < n_raw || b < nh) && k < cap_out) {
    uint64_t v;
    if (b >= nh || (a < n_raw && raw[a] <= heavy[b])) {
      v = raw[a++];
    } else {
      v = heavy[b++];
      if (room == 0) continue;
      --room;
    }
    if (k > 0 && out[k - 1] == v) continue;
    out[k++] = v;
  }
  *n_out = k;
}

// Heavy keys.  A value repeated among consecutive splitters would leave empty
// partitions, and one partition [v, next) would hold all copies of v plus
// other keys.  Walking left to right, a splitter not above the last kept one
// becomes that one + 1 (dropped at UINT64_MAX); a kept value v that occurs at
// least m / (2P) times in the sorted sample (half a partition's share) is
// followed by the boundary v + 1, so [v, v + 1) holds v alone.  At most
// 2 n_raw splitters result; their count goes to *n_out.
// One block: a thread per raw splitter counts its value in the sample (one
// thread walking all of them took 81 us for eight), then one thread walks.
constexpr uint32_t kMaxRawSplitters = 128;
__global__ void __launch_bounds__(kMaxRawSplitters) isolate_splitters_kernel(const uint64_t *raw, uint32_t n_raw,
                                                                            const uint64_t *sorted, uint64_t m,
                                                                            uint32_t P, uint64_t *out, uint32_t *n_out) {
  __shared__ uint64_t count[kMaxRawSplitters];
  auto occurrences = [&](uint64_t v) {
    uint64_t a = 0, b = m, c = 0, d = m;  // lower bound in [a, b), upper bound in [c, d)
    while (a < b || c < d) {
      const uint64_t p = (a + b) >> 1, q = (c + d) >> 1;
      const bool lo = a < b && sorted[p] < v, hi = c < d && sorted[q] <= v;
      if (a < b) (lo ? a : b) = lo ? p + 1 : p;
      if (c < d) (hi ? c : d) = hi ? q + 1 : q;
    }
    return c - a;
  };
  if (threadIdx.x < n_raw) count[threadIdx.x] = occurrences(raw[threadIdx.x]);
  __syncthreads();
  if (threadIdx.x != 0) return;
  uint32_t k = 0;
  for (uint32_t j = 0; j < n_raw; ++j) {
    uint64_t v = raw[j];
    uint64_t c = count[j];
    if (k > 0 && v <= out[k - 1]) {
      if (out[k - 1] == UINT64_MAX) continue;
      v = out[k - 1] + 1;
      c = occurrences(v);
    }
    out[k++] = v;
    if (c * 2 * (uint64_t)P >= m && v != UINT64_MAX) out[k++] = v + 1;
  }
  *n_out = k;
}

// ================================================================== host helpers

vx_status radix_publish_enqueue(char *temp, uint64_t *host_word, cudaStream_t s, int npass) {
  rx_publish<<<1, 1, 0, s>>>(radix_state_of(temp), npass, host_word);
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

static uint32_t ntiles_of(uint64_t n) { return (uint32_t)((n + kRxTile - 1) / kRxTile); }

// temp layout: [RadixState | 8 byte histograms (u64) | per-tile region]; the
// per-tile region holds the range partition's per-tile histograms (u32), or
// for an LSD sort the 8 digit bases (u64), 8 tickets and the look-back status
// words (u64 per tile and digit)
constexpr uint64_t kStateBytes = (sizeof(RadixState) + 255) & ~255ull;
constexpr uint64_t kByteHistBytes = 8ull * kRxDigits * 8;
constexpr uint64_t kBasesBytes = 8ull * kRxDigits * 8;
constexpr uint64_t kTicketBytes = 256;

uint64_t radix_temp_bytes(uint64_t cap) {
  // the sweep's tiles hold more, but for a small sort's
  const uint64_t nt = std::max<uint64_t>(
      {ntiles_of(cap), 1, std::min<uint64_t>((cap + kSweepSmallTile - 1) / kSweepSmallTile, kSweepSmallTiles)});
  return kStateBytes + kByteHistBytes + kBasesBytes + kTicketBytes + (uint64_t)kRxDigits * nt * 8 + 256;
}

RadixState *radix_state_of(char *temp) { return (RadixState *)temp; }

// after a radix sort on s: the buffer holding the result, or VX_E_TIMEOUT when
// a look-back wait gave up
static vx_status radix_result(char *temp, cudaStream_t s, int *cur, bool *redo = nullptr) {
  RadixState h;
  VX_CUDA_TRY(cudaMemcpyAsync(&h, radix_state_of(temp), offsetof(RadixState, totals), cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  if (h.err) {
    set_error("radix sort: a look-back wait gave up");
    return VX_E_TIMEOUT;
  }
  *cur = h.cur[8];
  if (redo) *redo = h.redo != 0;
  return VX_OK;
}

// Enqueues a stable LSD radix sort of b.keys[0]/b.vals[0] (n pairs) on s by
// the key bytes first .. npass - 1 (0 and 8: the whole key).  The sorted pairs end in
// buffer st->cur[npass] (0 or 1).
vx_status radix_sort_enqueue(RadixBufs b, uint64_t n, char *temp, cudaStream_t s, int num_sms, int npass,
                             uint32_t spin_limit, bool iota, cudaEvent_t vals, int first) {
  const uint32_t nt = sweep_tiles(n, num_sms);
  RadixState *st = radix_state_of(temp);
  unsigned long long *bh = (unsigned long long *)(temp + kStateBytes);
  uint64_t *bases = (uint64_t *)(temp + kStateBytes + kByteHistBytes);
  unsigned int *tickets = (unsigned int *)((char *)bases + kBasesBytes);
  unsigned long long *status = (unsigned long long *)((char *)tickets + kTicketBytes);
  if (n == 0) {
    VX_CUDA_TRY(cudaMemsetAsync(temp, 0, kStateBytes + kByteHistBytes, s));
    return VX_OK;
  }
  VX_TRY(rx_scatter_attr());
  // histograms, tickets and status words (the words carry their pass number)
  VX_CUDA_TRY(cudaMemsetAsync(bh, 0, kByteHistBytes + kBasesBytes + kTicketBytes + (uint64_t)kRxDigits * nt * 8, s));
  const int g = (int)std::min<uint64_t>((n + kRxThreads - 1) / kRxThreads, (uint64_t)num_sms * 6);
  auto hist = first == 1   ? (npass == 2 ? rx_byte_hist<1, 1> : rx_byte_hist<2, 1>)
              : first == 2 ? rx_byte_hist<1, 2>
              : npass == 1 ? rx_byte_hist<1>
              : npass == 2 ? rx_byte_hist<2>
              : npass == 3 ? rx_byte_hist<3>
                           : rx_byte_hist<8>;
  hist<<<g, kRxThreads, 0, s>>>(b.keys[0], n, bh);
  rx_init<<<npass - first, kRxDigits, 0, s>>>(st, bh, bases, n, spin_limit ? spin_limit : kRxSpinLimit, first);
  if (vals) VX_CUDA_TRY(cudaStreamWaitEvent(s, vals, 0));
  for (int pass = first; pass < npass; ++pass)  // a skipped pass returns at once and keeps the buffer
    VX_TRY(enqueue_sweep(b, st, pass, n, bases, tickets, status, iota, num_sms, s));
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

vx_status radix_prefix_sort_enqueue(RadixBufs b, uint64_t n, char *temp, cudaStream_t s, int num_sms, int first,
                                    uint32_t spin_limit, cudaEvent_t vals) {
  if (n < 2 || n >> 32 || (first != 3 && first != 4))
    return radix_sort_enqueue(b, n, temp, s, num_sms, 8, spin_limit, false, vals);
  const uint32_t nt = sweep_tiles(n, num_sms);
  RadixState *st = radix_state_of(temp);
  unsigned long long *bh = (unsigned long long *)(temp + kStateBytes);
  uint64_t *bases = (uint64_t *)(temp + kStateBytes + kByteHistBytes);
  unsigned int *tickets = (unsigned int *)((char *)bases + kBasesBytes);
  unsigned long long *status = (unsigned long long *)((char *)tickets + kTicketBytes);
  VX_TRY(rx_scatter_attr());
  VX_CUDA_TRY(cudaMemsetAsync(bh, 0, kByteHistBytes + kBasesBytes + kTicketBytes + (uint64_t)kRxDigits * nt * 8, s));
  const int g = (int)std::min<uint64_t>((n + kRxThreads - 1) / kRxThreads, (uint64_t)num_sms * 6);
  (first == 4 ? rx_byte_hist<4, 4> : rx_byte_hist<5, 3>)<<<g, kRxThreads, 0, s>>>(b.keys[0], n, bh);
  rx_init<<<8 - first, kRxDigits, 0, s>>>(st, bh, bases, n, spin_limit ? spin_limit : kRxSpinLimit, first);
  if (vals) VX_CUDA_TRY(cudaStreamWaitEvent(s, vals, 0));
  for (int pass = first; pass < 8; ++pass)
    VX_TRY(enqueue_sweep(b, st, pass, n, bases, tickets, status, false, num_sms, s));
  // the list takes the place of the look-back words: 256 * 8 bytes a tile
  const uint32_t cap = nt * (kRxDigits * 8 / 4);
  const int gf = (int)std::min<uint64_t>((n + 255) / 256, (uint64_t)num_sms * 8);
  rx_find_kernel<<<gf, 256, 0, s>>>(b, st, n, 8 * first, (uint32_t *)status, cap);
  rx_fix_kernel<<<num_sms * 2, 256, 0, s>>>(b, st, n, 8 * first, (const uint32_t *)status, cap);
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

// Enqueues a stable scatter of b.keys[0]/b.vals[0] into b.keys[1]/b.vals[1] by
// partition id (splitters spl[0..P-2] on the device); the P+1 boundary array
// is left in st->base[0..P] with base[P] = n.
vx_status range_partition_enqueue(RadixBufs b, uint64_t n, const uint64_t *spl, uint32_t P, char *temp,
                                  cudaStream_t s) {
  uint32_t nt = std::max<uint32_t>(ntiles_of(n), 1);
  RadixState *st = radix_state_of(temp);
  uint32_t *hist = (uint32_t *)(temp + kStateBytes + kByteHistBytes);
  VX_TRY(rx_scatter_attr());
  VX_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(RadixState), s));
  if (n) {
    rx_upsweep<<<nt, kRxThreads, 0, s>>>(b.keys[0], n, spl, (int)P - 1, hist, nt);
    rx_scan_rows<<<kRxDigits, 1024, 0, s>>>(hist, nt, st);
  }
  rx_scan_totals<<<1, kRxDigits, 0, s>>>(st, n);
  if (n) rx_range_scatter<<<nt, kRxThreads, kRxScatterSmem, s>>>(b, st, n, spl, (int)P - 1, hist, nt, nullptr);
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

// The same scatter of n > 0 pairs into the partitions' regions of b.keys[1] /
// b.vals[1], each behind what the region holds.
static vx_status region_partition_enqueue(RadixBufs b, uint64_t n, const uint64_t *spl, uint32_t P, RxRegions *rg,
                                          char *temp, cudaStream_t s) {
  const uint32_t nt = ntiles_of(n);
  RadixState *st = radix_state_of(temp);
  uint32_t *hist = (uint32_t *)(temp + kStateBytes + kByteHistBytes);
  VX_TRY(rx_scatter_attr());
  rx_upsweep<<<nt, kRxThreads, 0, s>>>(b.keys[0], n, spl, (int)P - 1, hist, nt);
  rx_scan_rows<<<kRxDigits, 1024, 0, s>>>(hist, nt, st);
  rx_place<<<1, kRxDigits, 0, s>>>(st, rg, P);
  rx_range_scatter<<<nt, kRxThreads, kRxScatterSmem, s>>>(b, st, n, spl, (int)P - 1, hist, nt, rg);
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}


// Splitters for P requested partitions from the sorted sample (device), then
// heavy-key isolation.  spl_buf has kSplitterBufBytes: [out 256 | raw 256 |
// knots 1025 | count]; returns the number of splitters in *n_spl (at most 254).
vx_status splitters_from_sample(vx_ctx *ctx, int32_t kind, const uint64_t *sorted, uint64_t m, uint32_t P,
                                uint64_t *spl_buf, uint32_t mlp_steps, double *ms_train, uint32_t *n_spl) {
  cudaStream_t s = ctx->s_compute;
  *n_spl = 0;
  if (P < 2) return VX_OK;
  if (P > kMaxRequestedPartitions) {
    set_error("at most %u partitions per pass", kMaxRequestedPartitions);
    return VX_E_UNSUPPORTED;
  }
  uint64_t *d_out = spl_buf, *d_raw = spl_buf + 256, *d_knots = spl_buf + 512;
  uint32_t *d_n = (uint32_t *)(spl_buf + 512 + kPLSegments + 1);
  if (kind == VX_PART_SAMPLE) {
    sample_splitters_kernel<<<1, 256, 0, s>>>(sorted, m, P, d_raw);
  } else if (kind == VX_PART_LEARNED_PL) {
    pl_knots_kernel<<<(kPLSegments + 256) / 256, 256, 0, s>>>(sorted, m, kPLSegments, d_knots);
    pl_splitters_kernel<<<1, 256, 0, s>>>(d_knots, kPLSegments, P, d_raw);
  } else if (kind == VX_PART_LEARNED_MLP) {
    VX_TRY(mlp_splitters(ctx, sorted, m, P, mlp_steps, d_raw, ms_train));
  } else {
    set_error("unknown partitioner %d", kind);
    return VX_E_INVAL;
  }
  uint32_t n_raw = P - 1;
  if (kind == VX_PART_LEARNED_MLP) {
    // a smooth CDF model steps over a heavy key's jump instead of landing a
    // splitter on it: add the sample's heavy keys to its splitters (the
    // knots area is free here: heavy keys, then the merged list, then counts)
    constexpr uint32_t kHeavyCap = 64, kMergedCap = 127;  // isolation doubles at most: <= 254 cuts
    uint64_t *d_heavy = d_knots, *d_merged = d_knots + kHeavyCap;
    uint32_t *d_cnt = (uint32_t *)(d_knots + kHeavyCap + kMergedCap);
    VX_CUDA_TRY(cudaMemsetAsync(d_cnt, 0, 8, s));
    heavy_keys_kernel<<<(unsigned)std::min<uint64_t>((m + 255) / 256, 1024), 256, 0, s>>>(sorted, m, P, d_heavy, d_cnt,
                                                                                      kHeavyCap);
    merge_heavy_kernel<<<1, 1, 0, s>>>(d_raw, P - 1, d_heavy, d_cnt, kHeavyCap, d_merged, d_cnt + 1, kMergedCap);
    VX_CUDA_TRY(cudaGetLastError());
    VX_CUDA_TRY(cudaMemcpyAsync(&n_raw, d_cnt + 1, 4, cudaMemcpyDeviceToHost, s));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    VX_CUDA_TRY(cudaMemcpyAsync(d_raw, d_merged, 8ull * n_raw, cudaMemcpyDeviceToDevice, s));
  }
  isolate_splitters_kernel<<<1, kMaxRawSplitters, 0, s>>>(d_raw, n_raw, sorted, m, P, d_out, d_n);
  VX_CUDA_TRY(cudaGetLastError());
  VX_CUDA_TRY(cudaMemcpyAsync(n_spl, d_n, 4, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  return VX_OK;
}

// samples m keys of a mapped column and sorts them on the device; m shrinks to
// what the free arena holds
vx_status sample_and_sort(vx_ctx *ctx, const uint64_t *dev_keys, uint64_t n, uint64_t &m, uint64_t seed,
                          DevBuf &sorted_out, uint64_t **sorted_ptr, const std::function<vx_status()> &sampled) {
  cudaStream_t s = ctx->s_compute;
  const uint64_t freeb = ctx->arena.largest_free();
  const uint64_t m_fit = freeb > (64u << 10) ? (freeb - (64u << 10)) / 25 : 0;
  m = std::min(m, m_fit);
  if (m == 0) {
    set_error("no room in the arena for a key sample");
    return VX_E_NOMEM;
  }
  uint64_t bytes = 2 * m * 12 + radix_temp_bytes(m) + 1024;
  sorted_out.arena = &ctx->arena;
  sorted_out.p = ctx->arena.alloc(bytes);
  if (!sorted_out.p) {
    set_error("sample of %llu keys does not fit the arena", (unsigned long long)m);
    return VX_E_NOMEM;
  }
  char *p = sorted_out.as<char>();
  RadixBufs b;
  b.keys[0] = (uint64_t *)p;
  b.keys[1] = (uint64_t *)(p + ((8 * m + 255) & ~255ull));
  char *q = p + 2 * ((8 * m + 255) & ~255ull);
  b.vals[0] = (uint32_t *)q;
  b.vals[1] = (uint32_t *)(q + ((4 * m + 255) & ~255ull));
  char *temp = q + 2 * ((4 * m + 255) & ~255ull);
  sample_keys_kernel<<<ctx->num_sms * 2, 256, 0, s>>>(dev_keys, n, m, seed, b.keys[0], b.vals[0]);
  VX_CUDA_TRY(cudaGetLastError());
  if (sampled) VX_TRY(sampled());
  VX_TRY(radix_sort_enqueue(b, m, temp, s, ctx->num_sms, 8, ctx->cfg.lookback_spin_limit));
  int cur = 0;
  VX_TRY(radix_result(temp, s, &cur));
  *sorted_ptr = b.keys[cur];
  return VX_OK;
}

// ================================================================== out-of-core sort

namespace {

void parallel_copy(void *dst, const void *src, uint64_t bytes) {
  const uint64_t kMin = 64ull << 20;
  unsigned nt = std::max(1u, std::min(16u, (unsigned)(bytes / kMin)));
  if (nt == 1) {
    memcpy(dst, src, bytes);
    return;
  }
  std::vector<std::thread> th;
  for (unsigned t = 0; t < nt; ++t) {
    uint64_t b = bytes * t / nt, e = bytes * (t + 1) / nt;
    th.emplace_back([=] { memcpy((char *)dst + b, (const char *)src + b, e - b); });
  }
  for (auto &x : th) x.join();
}

// pass 1: per-chunk stable partition into the intermediate + boundary arrays
// a run of one partition's pairs in host memory, in input order
struct Extent {
  const uint64_t *k;
  const uint32_t *v;
  uint64_t len;
};

// host memory registered for the call that holds spilled partition segments
struct Spill {
  std::unique_ptr<char[]> mem;
  HostReg reg;
  uint64_t cap = 0, used = 0;
};

// pass 1: range-partition each chunk on the device and store its partition
// segments to the host intermediate.  Contiguous layout: partition p owns
// [reg_off[p], reg_off[p] + reg_cap[p]) of the intermediate and each chunk's
// segment of p is appended there, so the sort pass loads a partition with one
// copy per column; what does not fit goes to the overflow area after the
// regions, then to spill buffers.  Blocked layout (an intermediate without room
// for the regions): chunk c keeps rows [c R, c R + R) and partition p is one
// extent per chunk.
struct PartitionPass : ExKernel {
  vx_ctx *ctx;
  const uint64_t *keys;
  const uint32_t *vals;
  uint64_t n, R;
  uint32_t P;
  const uint64_t *d_spl;
  uint64_t *mid_keys;
  uint32_t *mid_vals;
  uint64_t *h_bnd;  // page-locked host, chunks x (P+1): chunk-local partition starts
  bool contig = false;
  uint64_t C = 0;                          // pairs of the intermediate
  std::vector<uint64_t> reg_off, reg_cap;  // contiguous layout
  std::vector<uint64_t> used;
  uint64_t ovf = 0;                        // next free pair of the overflow area
  std::deque<Spill> *spills = nullptr;
  std::vector<std::vector<Extent>> ext;    // per partition, in input order

  uint64_t size() override { return (n + R - 1) / R; }
  uint64_t rows(uint64_t it) const { return std::min(R, n - it * R); }
  uint64_t kb() const { return (8 * R + 255) & ~255ull; }
  uint64_t vb() const { return (4 * R + 255) & ~255ull; }
  uint64_t slot_bytes() override { return 2 * kb() + 2 * vb() + radix_temp_bytes(R); }
  RadixBufs bufs(char *slot) const {
    RadixBufs b;
    b.keys[0] = (uint64_t *)slot;
    b.keys[1] = (uint64_t *)(slot + kb());
    b.vals[0] = (uint32_t *)(slot + 2 * kb());
    b.vals[1] = (uint32_t *)(slot + 2 * kb() + vb());
    return b;
  }
  char *temp(char *slot) const { return slot + 2 * kb() + 2 * vb(); }
  void inputs(uint64_t it, char *slot, std::vector<CopyOp> &h2d) override {
    RadixBufs b = bufs(slot);
    uint64_t r0 = it * R, m = rows(it);
    h2d.push_back({keys + r0, b.keys[0], 8 * m});
    h2d.push_back({vals + r0, b.vals[0], 4 * m});
  }
  vx_status kernel(char *slot, uint64_t it, cudaStream_t s) override {
    VX_TRY(range_partition_enqueue(bufs(slot), rows(it), d_spl, P, temp(slot), s));
    // the chunk's boundary array goes to page-locked host memory (a copy into
    // pageable memory would hold the issuing thread until the store queue
    // drains); outputs() reads it once the kernel has completed
    VX_CUDA_TRY(cudaMemcpyAsync(h_bnd + it * (P + 1), radix_state_of(temp(slot))->base, 8ull * (P + 1),
                                cudaMemcpyDeviceToHost, s));
    return VX_OK;
  }
  bool has_outputs() override { return true; }
  void add_extent(uint32_t p, const uint64_t *k, const uint32_t *v, uint64_t len) {
    std::vector<Extent> &e = ext[p];
    if (!e.empty() && e.back().k + e.back().len == k && e.back().v + e.back().len == v)
      e.back().len += len;  // right after the partition's previous segment
    else
      e.push_back({k, v, len});
  }
  // room for up to len pairs of partition p: its region, the overflow area,
  // then a spill buffer; *take pairs of it are handed out
  vx_status place(uint32_t p, uint64_t len, uint64_t **dk, uint32_t **dv, uint64_t *take) {
    if (used[p] < reg_cap[p]) {
      *take = std::min(len, reg_cap[p] - used[p]);
      *dk = mid_keys + reg_off[p] + used[p];
      *dv = mid_vals + reg_off[p] + used[p];
      used[p] += *take;
      return VX_OK;
    }
    if (ovf < C) {
      *take = std::min(len, C - ovf);
      *dk = mid_keys + ovf;
      *dv = mid_vals + ovf;
      ovf += *take;
      return VX_OK;
    }
    if (spills->empty() || spills->back().used == spills->back().cap) {
      spills->emplace_back();
      Spill &sp = spills->back();
      sp.cap = std::max(len, R);
      sp.mem.reset(new (std::nothrow) char[12 * sp.cap]);
      if (!sp.mem) {
        set_error("vx_sort: no host memory for %llu spilled pairs", (unsigned long long)sp.cap);
        return VX_E_NOMEM;
      }
      VX_TRY(sp.reg.add(sp.mem.get(), 12 * sp.cap));
    }
    Spill &sp = spills->back();
    *take = std::min(len, sp.cap - sp.used);
    *dk = (uint64_t *)sp.mem.get() + sp.used;
    *dv = (uint32_t *)(sp.mem.get() + 8 * sp.cap) + sp.used;
    sp.used += *take;
    return VX_OK;
  }
  vx_status outputs(uint64_t it, char *slot, std::vector<CopyOp> &d2h) override {
    RadixBufs b = bufs(slot);
    const uint64_t r0 = it * R, m = rows(it);
    const uint64_t *bd = h_bnd + it * (P + 1);  // copied before the kernel's completion event
    if (!contig) {
      d2h.push_back({b.keys[1], mid_keys + r0, 8 * m});
      d2h.push_back({b.vals[1], mid_vals + r0, 4 * m});
      for (uint32_t p = 0; p < P; ++p)
        if (bd[p + 1] > bd[p]) add_extent(p, mid_keys + r0 + bd[p], mid_vals + r0 + bd[p], bd[p + 1] - bd[p]);
      return VX_OK;
    }
    for (uint32_t p = 0; p < P; ++p) {
      uint64_t s0 = bd[p], len = bd[p + 1] - bd[p];
      while (len) {
        uint64_t *dk;
        uint32_t *dv;
        uint64_t take;
        VX_TRY(place(p, len, &dk, &dv, &take));
        d2h.push_back({b.keys[1] + s0, dk, 8 * take});
        d2h.push_back({b.vals[1] + s0, dv, 4 * take});
        add_extent(p, dk, dv, take);
        s0 += take;
        len -= take;
      }
    }
    return VX_OK;
  }
};

// pass 2: per-partition gather + radix sort + store
struct SortPass : ExKernel {
  vx_ctx *ctx;
  uint64_t cap;
  std::vector<std::vector<Extent>> ext;  // per job
  std::vector<uint64_t> job_n, job_off;
  uint64_t *out_keys;
  uint32_t *out_vals;
  int S;                    // slots of the ring (one published result word per slot)
  uint64_t pass_pairs = 0;  // pairs x executed passes

  uint64_t size() override { return job_n.size(); }
  int n_slots() override { return S; }
  int max_in_flight() override { return S; }
  uint64_t kb() const { return (8 * cap + 255) & ~255ull; }
  uint64_t vb() const { return (4 * cap + 255) & ~255ull; }
  uint64_t slot_bytes() override { return 2 * kb() + 2 * vb() + radix_temp_bytes(cap); }
  RadixBufs bufs(char *slot) const {
    RadixBufs b;
    b.keys[0] = (uint64_t *)slot;
    b.keys[1] = (uint64_t *)(slot + kb());
    b.vals[0] = (uint32_t *)(slot + 2 * kb());
    b.vals[1] = (uint32_t *)(slot + 2 * kb() + vb());
    return b;
  }
  char *temp(char *slot) const { return slot + 2 * kb() + 2 * vb(); }
  void inputs(uint64_t it, char *slot, std::vector<CopyOp> &h2d) override {
    RadixBufs b = bufs(slot);
    uint64_t at = 0;
    for (const Extent &e : ext[it]) {
      if (!e.len) continue;
      h2d.push_back({e.k, b.keys[0] + at, 8 * e.len});
      h2d.push_back({e.v, b.vals[0] + at, 4 * e.len});
      at += e.len;
    }
  }
  vx_status kernel(char *slot, uint64_t it, cudaStream_t s) override {
    VX_TRY(radix_sort_enqueue(bufs(slot), job_n[it], temp(slot), s, ctx->num_sms, 8, ctx->cfg.lookback_spin_limit));
    rx_publish<<<1, 1, 0, s>>>(radix_state_of(temp(slot)), 8, ctx->d_scalars + 64 + (it % S));
    VX_CUDA_TRY(cudaGetLastError());
    return VX_OK;
  }
  bool has_outputs() override { return true; }
  vx_status outputs(uint64_t it, char *slot, std::vector<CopyOp> &d2h) override {
    RadixBufs b = bufs(slot);
    const uint64_t word = ((volatile uint64_t *)ctx->h_scalars)[64 + (it % S)];
    if (word >> 16 & 1) {
      set_error("radix sort of partition job %llu: a look-back wait gave up", (unsigned long long)it);
      return VX_E_TIMEOUT;
    }
    const int c = (int)(word & 0xFF);
    pass_pairs += job_n[it] * ((word >> 8) & 0xFF);
    if (job_n[it] == 0) return VX_OK;
    d2h.push_back({b.keys[c], out_keys + job_off[it], 8 * job_n[it]});
    d2h.push_back({b.vals[c], out_vals + job_off[it], 4 * job_n[it]});
    return VX_OK;
  }
};

// ---- partitions that stay in the arena
// When the arena holds all pairs beside the slots of both passes, pass 1
// scatters the chunks straight into the partitions' regions and pass 2 sorts
// each partition where it is (the other buffer in a slot) and stores it: the
// pairs cross the link once in each direction instead of twice.  67M uniform
// pairs (805 MB) under 1 GiB: 10.3 ms, 13.7 through host memory (9.05 with the
// shorter sorts and the early loads below); 300M (3.6 GB) under 4.5 GiB: 37.5
// ms, about 62.  Bound by the link one way, then the other.
struct ResidentPlan {
  std::vector<uint64_t> off, cap;  // regions, pairs
  uint64_t pairs = 0;              // all regions
  uint64_t R = 0, jcap = 0;        // pairs per slot of pass 1 and pass 2
  int S1 = 0, S2 = 0;
  // pass 1's slots, which take what the regions leave of the arena; the first
  // chunks are loaded into them while the splitters are still being found (the
  // sample's sort, the model's training), and pass 2's slots follow in their
  // place.  50M pairs with the MLP partitioner, whose training takes 1.9 ms: 9.7
  // -> 8.1 ms; 67M with the sample's quantiles 9.3 -> 9.05.
  vx_ctx *ctx = nullptr;
  DevBuf ring;
  std::vector<cudaEvent_t> loaded;  // one per chunk, after its copies
  uint64_t bytes_loaded = 0;
  bool drain = false;
  void release() {
    if (!ring.p) return;
    if (ctx->poisoned) ring.arena = nullptr;  // work that never finished may still write there
    else if (drain) cudaStreamSynchronize(ctx->s_h2d);
    ring.release();
  }
  ~ResidentPlan() {
    release();
    for (cudaEvent_t e : loaded) cudaEventDestroy(e);
  }
};

struct ResidentPartitionPass : ExKernel {
  const uint64_t *keys;
  const uint32_t *vals;
  uint64_t n, R;
  int S;
  uint32_t P;
  const uint64_t *d_spl;
  uint64_t *res_keys;
  uint32_t *res_vals;
  RxRegions *rg;
  char *base;  // the ring
  const std::vector<cudaEvent_t> *loaded = nullptr;  // chunks whose copies have been issued
  uint64_t size() override { return (n + R - 1) / R; }
  int n_slots() override { return S; }
  int max_in_flight() override { return S; }
  char *ring() override { return base; }
  cudaEvent_t loaded_event(uint64_t it) override { return loaded && it < loaded->size() ? (*loaded)[it] : nullptr; }
  uint64_t rows(uint64_t it) const { return std::min(R, n - it * R); }
  uint64_t kb() const { return (8 * R + 255) & ~255ull; }
  uint64_t vb() const { return (4 * R + 255) & ~255ull; }
  static uint64_t bytes(uint64_t R) { return (8 * R + 255) / 256 * 256 + (4 * R + 255) / 256 * 256 + radix_temp_bytes(R); }
  uint64_t slot_bytes() override { return bytes(R); }
  void inputs(uint64_t it, char *slot, std::vector<CopyOp> &h2d) override {
    if (loaded_event(it)) return;
    h2d.push_back({keys + it * R, slot, 8 * rows(it)});
    h2d.push_back({vals + it * R, slot + kb(), 4 * rows(it)});
  }
  vx_status kernel(char *slot, uint64_t it, cudaStream_t s) override {
    RadixBufs b;
    b.keys[0] = (uint64_t *)slot;
    b.vals[0] = (uint32_t *)(slot + kb());
    b.keys[1] = res_keys;
    b.vals[1] = res_vals;
    return region_partition_enqueue(b, rows(it), d_spl, P, rg, slot + kb() + vb(), s);
  }
};

struct ResidentSortPass : ExKernel {
  vx_ctx *ctx;
  uint64_t cap;
  struct Job {
    uint64_t *k;
    uint32_t *v;
    uint64_t n, at;  // pairs, output position
    bool sorted;     // one key value: already in input order
  };
  std::vector<Job> jobs;
  uint64_t *out_keys;
  uint32_t *out_vals;
  int S;
  int first;  // sort by the key bytes first .. 7 and repair, 0: by all
  uint64_t pass_pairs = 0, launches = 0;
  uint64_t size() override { return jobs.size(); }
  int n_slots() override { return S; }
  int max_in_flight() override { return S; }
  uint64_t kb() const { return (8 * cap + 255) & ~255ull; }
  uint64_t vb() const { return (4 * cap + 255) & ~255ull; }
  uint64_t slot_bytes() override { return ResidentPartitionPass::bytes(cap); }
  void inputs(uint64_t, char *, std::vector<CopyOp> &) override {}
  RadixBufs bufs(const Job &j, char *slot) const {
    RadixBufs b;
    b.keys[0] = j.k;
    b.vals[0] = j.v;
    b.keys[1] = (uint64_t *)slot;
    b.vals[1] = (uint32_t *)(slot + kb());
    return b;
  }
  vx_status kernel(char *slot, uint64_t it, cudaStream_t s) override {
    const Job &j = jobs[it];
    if (j.sorted) return VX_OK;
    char *temp = slot + kb() + vb();
    if (first)
      VX_TRY(radix_prefix_sort_enqueue(bufs(j, slot), j.n, temp, s, ctx->num_sms, first, ctx->cfg.lookback_spin_limit));
    else
      VX_TRY(radix_sort_enqueue(bufs(j, slot), j.n, temp, s, ctx->num_sms, 8, ctx->cfg.lookback_spin_limit));
    launches += (first ? radix_prefix_launches(j.n, first) : radix_launches()) + 1;  // and publish
    return radix_publish_enqueue(temp, ctx->d_scalars + 64 + (it % S), s);
  }
  bool has_outputs() override { return true; }
  vx_status outputs(uint64_t it, char *slot, std::vector<CopyOp> &d2h) override {
    const Job &j = jobs[it];
    RadixBufs b = bufs(j, slot);
    int c = 0;
    for (bool again = !j.sorted; again;) {
      const uint64_t word = ((volatile uint64_t *)ctx->h_scalars)[64 + (it % S)];
      if (word >> 16 & 1) {
        set_error("radix sort of partition job %llu: a look-back wait gave up", (unsigned long long)it);
        return VX_E_TIMEOUT;
      }
      c = (int)(word & 0xFF);
      pass_pairs += j.n * ((word >> 8) & 0xFF);
      again = word >> 17 & 1;
      if (again) {  // a prefix that many keys share: sort the partition in full, from where it is
        if (c) {
          std::swap(b.keys[0], b.keys[1]);
          std::swap(b.vals[0], b.vals[1]);
        }
        char *temp = slot + kb() + vb();
        VX_TRY(radix_sort_enqueue(b, j.n, temp, ctx->s_compute, ctx->num_sms, 8, ctx->cfg.lookback_spin_limit));
        VX_TRY(radix_publish_enqueue(temp, ctx->d_scalars + 64 + (it % S), ctx->s_compute));
        launches += radix_launches() + 1;
        VX_CUDA_TRY(cudaStreamSynchronize(ctx->s_compute));
      }
    }
    d2h.push_back({b.keys[c], out_keys + j.at, 8 * j.n});
    d2h.push_back({b.vals[c], out_vals + j.at, 4 * j.n});
    return VX_OK;
  }
};

// partition p of spl's P = spl.size() + 1 holds one key value
bool single_key_partition(const std::vector<uint64_t> &spl, uint32_t p) {
  const uint64_t lo = p == 0 ? 0 : spl[p - 1];
  return p < spl.size() ? (spl[p] > lo && spl[p] - lo == 1) : lo == UINT64_MAX;
}

// Bytes of the arena that P regions (with their headroom, see resident_layout)
// leave to the slots; m sampled keys
uint64_t resident_left(uint64_t n, uint64_t m, uint32_t P, uint64_t avail) {
  const double pairs = 1.002 * (double)n +
                       P * (6.0 * std::sqrt((double)m / P + 1.0) * (double)n / (double)m + kRxTile + 128.0);
  const double left = (double)avail - 12.0 * pairs - (1 << 20);
  return left > 0 ? (uint64_t)left : 0;
}

// Partitions requested so that two slots of pass 2 fit what the regions leave,
// with room for uneven partitions; 0: they do not fit.
uint32_t resident_partitions(uint64_t n, uint64_t m, uint64_t avail, double headroom) {
  // at most 12M pairs a job as far as kMaxResident partitions go, so that the
  // stores start early (1e9 pairs under 16 GiB: 122 ms with 64 resident
  // partitions, 162 through host memory)
  constexpr double kMaxResident = 64.0;
  double P = std::min(kMaxResident, std::max(4.0, std::ceil((double)n / 12e6)));
  for (int i = 0; i < 8 && P <= kMaxResident; ++i) {
    const double jcap = (double)resident_left(n, m, (uint32_t)P, avail) / (2 * 12.6);
    if (jcap < 1) return 0;
    if (headroom * (double)n / jcap <= P) return (uint32_t)P;
    P = std::ceil(headroom * (double)n / jcap);
  }
  return 0;
}

// Pass 1's ring: chunks of n / 16 pairs (smaller if S slots of them do not fit),
// as many slots as fit and are of use.  False: no room.
bool resident_ring(vx_ctx *ctx, uint64_t n, uint64_t left, int S, ResidentPlan *rp) {
  auto slot = [](uint64_t R) { return (ResidentPartitionPass::bytes(R) + 255) & ~255ull; };
  for (rp->R = std::min<uint64_t>(std::max<uint64_t>(n / 16, 1 << 20), kPipelineRows) / kRxTile * kRxTile;
       rp->R >= (1 << 18); rp->R = rp->R / 2 / kRxTile * kRxTile)
    if ((uint64_t)S * slot(rp->R) <= left) break;
  if (rp->R < (1 << 18)) return false;
  rp->S1 = (int)std::max<uint64_t>(S, std::min<uint64_t>({left / slot(rp->R), (n + rp->R - 1) / rp->R, 12}));
  rp->ctx = ctx;
  rp->ring.arena = &ctx->arena;
  rp->ring.bytes = std::max<uint64_t>(rp->S1 * slot(rp->R), std::min<uint64_t>(left, 2 * 13 * 13000000ull));
  rp->ring.p = ctx->arena.alloc(rp->ring.bytes);
  return rp->ring.p != nullptr;
}

// Loads the first chunks into the ring on the host-to-device stream, behind the
// work that the compute stream has now.
vx_status resident_prefetch(const uint64_t *keys, const uint32_t *vals, uint64_t n, ResidentPlan *rp) {
  vx_ctx *ctx = rp->ctx;
  cudaEvent_t e;
  VX_CUDA_TRY(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  struct Free {
    cudaEvent_t e;
    ~Free() { cudaEventDestroy(e); }
  } fr{e};
  VX_CUDA_TRY(cudaEventRecord(e, ctx->s_compute));
  VX_CUDA_TRY(cudaStreamWaitEvent(ctx->s_h2d, e, 0));
  ResidentPartitionPass pp;
  pp.keys = keys;
  pp.vals = vals;
  pp.n = n;
  pp.R = rp->R;
  std::vector<CopyOp> ops;
  rp->drain = true;
  const uint64_t slot = (pp.slot_bytes() + 255) & ~255ull, k = std::min<uint64_t>(pp.size(), rp->S1);
  for (uint64_t it = 0; it < k; ++it) {
    ops.clear();
    pp.inputs(it, rp->ring.as<char>() + it * slot, ops);
    VX_TRY(issue_copies(ops, cudaMemcpyHostToDevice, ctx->s_h2d, &rp->bytes_loaded, h2d_sm_blocks(ctx)));
    cudaEvent_t done;
    VX_CUDA_TRY(cudaEventCreateWithFlags(&done, cudaEventDisableTiming));
    rp->loaded.push_back(done);
    VX_CUDA_TRY(cudaEventRecord(done, ctx->s_h2d));
  }
  return VX_OK;
}

// Regions from the sample's count in each partition: the estimate plus 0.2 %
// and six standard deviations (a region that is too small all the same ends the
// attempt).  False if the regions do not fit `rest` bytes or two slots of pass
// 2 the ring's.
bool resident_layout(uint64_t n, uint64_t m, const std::vector<uint64_t> &spl, const std::vector<uint64_t> &srank,
                     uint64_t rest, ResidentPlan *rp) {
  const uint32_t P = (uint32_t)spl.size() + 1;
  rp->off.resize(P);
  rp->cap.resize(P);
  rp->pairs = rp->jcap = 0;
  const double scale = (double)n / (double)m;
  for (uint32_t p = 0; p < P; ++p) {
    const double cnt = (double)((p + 1 < P ? srank[p] : m) - (p ? srank[p - 1] : 0));
    const double est = 1.002 * cnt * scale + 6.0 * std::sqrt(cnt + 1.0) * scale + kRxTile;
    rp->cap[p] = (std::min<uint64_t>(n, (uint64_t)std::ceil(est)) + 127) / 128 * 128;
    rp->off[p] = rp->pairs;
    rp->pairs += rp->cap[p];
    if (!single_key_partition(spl, p)) rp->jcap = std::max(rp->jcap, rp->cap[p]);
  }
  rp->jcap = std::max<uint64_t>(rp->jcap, kRxTile);
  rp->S2 = (int)std::min<uint64_t>(kMaxSortSlots, rp->ring.bytes / ((ResidentPartitionPass::bytes(rp->jcap) + 255) & ~255ull));
  return rp->S2 >= 2 && 12 * rp->pairs + sizeof(RxRegions) + 4096 <= rest;
}

// Both passes with resident partitions.  *done = false: a region was too small
// (nothing has been written to the output; the caller sorts the other way).
vx_status resident_sort(vx_ctx *ctx, const uint64_t *keys, const uint32_t *vals, uint64_t n, uint64_t *out_keys,
                        uint32_t *out_vals, const uint64_t *d_spl, const std::vector<uint64_t> &spl,
                        ResidentPlan &rp, int first, vx_sort_stats &ss, bool *done) {
  const uint32_t P = (uint32_t)spl.size() + 1;
  *done = false;
  DevBuf mem;
  mem.arena = &ctx->arena;
  const uint64_t kb = (8 * rp.pairs + 255) & ~255ull, vb = (4 * rp.pairs + 255) & ~255ull;
  mem.p = ctx->arena.alloc(kb + vb + sizeof(RxRegions));
  if (!mem.p) return VX_OK;
  uint64_t *res_keys = mem.as<uint64_t>();
  uint32_t *res_vals = (uint32_t *)(mem.as<char>() + kb);
  RxRegions *rg = (RxRegions *)(mem.as<char>() + kb + vb);
  cudaStream_t s = ctx->s_compute;
  double t0 = now_ms();
  auto h = std::make_unique<RxRegions>();
  memset(h.get(), 0, sizeof(RxRegions));
  for (uint32_t p = 0; p < P; ++p) {
    h->off[p] = rp.off[p];
    h->cap[p] = rp.cap[p];
  }
  VX_CUDA_TRY(cudaMemcpyAsync(rg, h.get(), sizeof(RxRegions), cudaMemcpyHostToDevice, s));
  {
    ResidentPartitionPass pp;
    pp.keys = keys;
    pp.vals = vals;
    pp.n = n;
    pp.R = rp.R;
    pp.S = rp.S1;
    pp.P = P;
    pp.d_spl = d_spl;
    pp.res_keys = res_keys;
    pp.res_vals = res_vals;
    pp.rg = rg;
    pp.base = rp.ring.as<char>();
    pp.loaded = &rp.loaded;
    ExecStats es;
    VX_TRY(run_pipeline(ctx, pp, &es));
    VX_CUDA_TRY(cudaMemcpyAsync(h.get(), rg, sizeof(RxRegions), cudaMemcpyDeviceToHost, s));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    ss.bytes_h2d += es.bytes_h2d;
    ss.kernel_launches += es.kernel_launches * 4;  // upsweep, row scan, placement, scatter
    rp.release();  // pass 2's slots take the ring's place
  }
  ss.ms_partition += now_ms() - t0;
  if (h->full) return VX_OK;
  t0 = now_ms();
  ResidentSortPass sp;
  sp.ctx = ctx;
  sp.cap = rp.jcap;
  sp.first = first;
  sp.out_keys = out_keys;
  sp.out_vals = out_vals;
  sp.S = rp.S2;
  uint64_t at = 0, mx = 0, mn = UINT64_MAX;
  for (uint32_t p = 0; p < P; ++p) {
    const uint64_t c = h->used[p];
    mx = std::max(mx, c);
    mn = std::min(mn, c);
    const bool one = single_key_partition(spl, p);
    if (c) {
      ss.passthrough_partitions += one;
      sp.jobs.push_back({res_keys + rp.off[p], res_vals + rp.off[p], c, at, one});
    }
    at += c;
  }
  ExecStats es;
  VX_TRY(run_pipeline(ctx, sp, &es));
  ss.bytes_h2d += es.bytes_h2d;
  ss.bytes_d2h += es.bytes_d2h;
  ss.kernel_launches += sp.launches;
  ss.ms_sort_kernel += es.ms_kernel;
  ss.radix_pass_pairs += sp.pass_pairs;
  ss.ms_sort += now_ms() - t0;
  ss.n_partitions = P;
  ss.max_partition = mx;
  ss.min_partition = mn;
  ss.imbalance = (double)mx / ((double)n / P);
  ss.contiguous_layout = 1;
  *done = true;
  return VX_OK;
}

}  // namespace

// sorts contiguous host pairs (keys/vals mapped or pinned) into out
static vx_status sort_pairs(vx_ctx *ctx, const uint64_t *keys, const uint32_t *vals, const uint64_t *dev_keys,
                            uint64_t n, uint64_t *out_keys, uint32_t *out_vals, const vx_sort_opts &o,
                            vx_sort_stats &ss, int depth, bool may_reside) {
  const int S = std::max(2, ctx->cfg.n_slots);
  const uint64_t avail = ctx->arena.largest_free();
  // pairs per slot: (2 x 12 B + histograms) per pair, S slots
  uint64_t cap = (uint64_t)((double)avail / (S * (24.0 + 256.0 * 8 / kRxTile)) * 0.97);
  cap = cap / kRxTile * kRxTile;
  if (o.max_slot_pairs) cap = std::min<uint64_t>(cap, o.max_slot_pairs / kRxTile * kRxTile);
  if (cap < kRxTile) {
    set_error("vx_sort: arena of %llu bytes too small", (unsigned long long)ctx->arena.capacity());
    return VX_E_NOMEM;
  }
  ss.slot_pairs = cap;
  if (n == 0) return VX_OK;
  double t0 = now_ms();
  // ---- P = 1: the input fits one slot
  if (n <= cap && o.n_partitions <= 1) {
    SortPass sp;
    sp.ctx = ctx;
    sp.cap = cap;
    sp.ext.push_back({{keys, vals, n}});
    sp.job_n.push_back(n);
    sp.job_off.push_back(0);
    sp.out_keys = out_keys;
    sp.out_vals = out_vals;
    sp.S = S;
    ExecStats es;
    VX_TRY(run_pipeline(ctx, sp, &es));
    ss.bytes_h2d += es.bytes_h2d;
    ss.bytes_d2h += es.bytes_d2h;
    ss.kernel_launches += es.kernel_launches * (radix_launches() + 1);  // and publish
    ss.ms_sort_kernel += es.ms_kernel;
    ss.radix_pass_pairs += sp.pass_pairs;
    ss.n_partitions = std::max<uint32_t>(ss.n_partitions, 1);
    ss.max_partition = std::max(ss.max_partition, n);
    ss.ms_sort += now_ms() - t0;
    return VX_OK;
  }
  // ---- splitters from a sample
  // requested partitions: 30% headroom at the top level, 2x inside a recursion
  const double over = depth == 0 ? 1.3 : 2.0;
  uint32_t P = o.n_partitions > 1 ? (uint32_t)o.n_partitions
                                  : (uint32_t)std::min<uint64_t>(kMaxRequestedPartitions,
                                                                 (uint64_t)std::ceil(over * (double)n / cap));
  if (P < 2) P = 2;
  // enough partitions that the sort pass pipelines (loads of partition p+1
  // and stores of p-1 overlap the sort of p) when the caller leaves P open
  if (depth == 0 && o.n_partitions <= 1 && n >= kPipelineRows * 4) P = std::max<uint32_t>(P, 16);
  if (P > kMaxRequestedPartitions) {
    set_error("vx_sort: at most %u partitions per pass", kMaxRequestedPartitions);
    return VX_E_UNSUPPORTED;
  }
  uint64_t m = std::min<uint64_t>(o.sample_size ? o.sample_size : (1ull << 20), n);
  DevBuf sbuf, splbuf;
  uint64_t *sorted = nullptr;
  double ts = now_ms();
  // the splitters outlive the sample: allocated first, they do not split the
  // arena's free space in two once the sample is released (the passes below
  // size their slots from the largest free block)
  splbuf.arena = &ctx->arena;
  splbuf.p = ctx->arena.alloc(kSplitterBufBytes);
  if (!splbuf.p) {
    set_error("vx_sort: no room for the splitters");
    return VX_E_NOMEM;
  }
  uint64_t *d_spl = splbuf.as<uint64_t>();
  // resident partitions, where the caller has not bounded the slots or the
  // regions (a smooth model's partitions are less even than the sample's): the
  // ring comes first in the arena, so that what is left is in one piece once the
  // sample is gone
  const uint32_t P_out = P;
  uint32_t P_in = 0;
  ResidentPlan rp;
  uint64_t rest = 0;
  if (may_reside && depth == 0 && !o.max_slot_pairs && !o.region_slack_pct) {
    const uint64_t avail = ctx->arena.largest_free();
    P_in = resident_partitions(n, m, avail, o.partitioner == VX_PART_LEARNED_MLP ? 1.4 : 1.1);
    if (P_in && o.n_partitions > 1) P_in = (uint32_t)o.n_partitions;
    if (P_in && !resident_ring(ctx, n, resident_left(n, m, P_in, avail), S, &rp)) P_in = 0;
    rest = ctx->arena.largest_free();
  }
  VX_TRY(sample_and_sort(ctx, dev_keys, n, m, o.seed + (uint64_t)depth * 7919, sbuf, &sorted, [&]() -> vx_status {
    return P_in ? resident_prefetch(keys, vals, n, &rp) : VX_OK;
  }));
  ss.bytes_h2d += rp.bytes_loaded;
  double ms_train = 0;
  uint32_t n_spl = 0;
  std::vector<uint64_t> spl, srank;
  DevBuf pbuf;  // sample_prefix_kernel's counts
  pbuf.arena = &ctx->arena;
  uint64_t prefix[4] = {0, 0, 0, 0};
  // splitters for `want` requested partitions and the sample's rank of each
  auto cut = [&](uint32_t want) -> vx_status {
    double ms = 0;
    VX_TRY(splitters_from_sample(ctx, o.partitioner, sorted, m, want, d_spl, o.mlp_steps, &ms, &n_spl));
    ms_train += ms;
    P = n_spl + 1;  // partitions after heavy-key isolation
    spl.resize(n_spl);
    srank.resize(n_spl);
    if (n_spl) {
      DevBuf rbuf;
      rbuf.arena = &ctx->arena;
      rbuf.p = ctx->arena.alloc(8 * n_spl);
      if (!rbuf.p) return VX_E_NOMEM;
      sample_ranks_kernel<<<1, 128, 0, ctx->s_compute>>>(sorted, m, d_spl, n_spl, rbuf.as<uint64_t>());
      VX_CUDA_TRY(cudaGetLastError());
      VX_CUDA_TRY(cudaMemcpyAsync(spl.data(), d_spl, 8 * n_spl, cudaMemcpyDeviceToHost, ctx->s_compute));
      VX_CUDA_TRY(cudaMemcpyAsync(srank.data(), rbuf.p, 8 * n_spl, cudaMemcpyDeviceToHost, ctx->s_compute));
    }
    if (pbuf.p)
      VX_CUDA_TRY(cudaMemcpyAsync(prefix, pbuf.p, sizeof prefix, cudaMemcpyDeviceToHost, ctx->s_compute));
    VX_CUDA_TRY(cudaStreamSynchronize(ctx->s_compute));
    return VX_OK;
  };
  int first = 0;  // key bytes that the partitions' sorts may leave to a repair
  bool reside = false;
  if (P_in) {
    pbuf.p = ctx->arena.alloc(sizeof prefix);
    if (pbuf.p) {
      VX_CUDA_TRY(cudaMemsetAsync(pbuf.p, 0, sizeof prefix, ctx->s_compute));
      sample_prefix_kernel<<<ctx->num_sms * 4, 256, 0, ctx->s_compute>>>(sorted, m, pbuf.as<unsigned long long>());
      VX_CUDA_TRY(cudaGetLastError());
    }
    VX_TRY(cut(P_in));
    reside = resident_layout(n, m, spl, srank, rest, &rp);
    if (pbuf.p) first = prefix_bytes(prefix, m, n, false);
    pbuf.release();
    if (!reside) rp.release();
  }
  if (!reside && P_in != P_out) VX_TRY(cut(P_out));
  sbuf.release();
  ss.ms_sample += now_ms() - ts - ms_train;
  ss.ms_train += ms_train;
  if (depth == 0 && o.splitters_out) memcpy(o.splitters_out, spl.data(), 8 * n_spl);
  if (reside) {
    bool done = false;
    VX_TRY(resident_sort(ctx, keys, vals, n, out_keys, out_vals, d_spl, spl, rp, first, ss, &done));
    if (done) return VX_OK;
    rp.release();
    splbuf.release();
    return sort_pairs(ctx, keys, vals, dev_keys, n, out_keys, out_vals, o, ss, depth, false);
  }

  // partition-pass chunks of kPipelineRows pairs: long enough for efficient
  // copies (576 MB), short enough that the pass pipelines over many chunks
  const uint64_t R = std::min<uint64_t>(cap, kPipelineRows);
  const uint64_t n_chunks = (n + R - 1) / R;

  // ---- host intermediate: one region per partition, sized from the sample's
  // count c in it (estimate n c / m) plus 1 % and four binomial standard
  // deviations, then an overflow area of what the intermediate has left (at
  // least n / 256 pairs); the sort stays exact whatever the estimates, only the
  // number of extents grows
  std::vector<uint64_t> reg_off(P), reg_cap(P);
  uint64_t regions = 0;
  for (uint32_t p = 0; p < P; ++p) {
    const uint64_t r1 = p < n_spl ? srank[p] : m, r0 = p ? srank[p - 1] : 0;
    const double cnt = (double)(r1 - r0), scale = (double)n / (double)m;
    const double slack = o.region_slack_pct ? o.region_slack_pct / 100.0 : 0.01;
    const double sigmas = o.region_slack_pct ? 0.0 : 4.0;
    const double est = (1.0 + slack) * cnt * scale + sigmas * std::sqrt(cnt + 1.0) * scale + kRxTile;
    // regions start on 128-pair boundaries (1 KB of keys, 512 B of values), so
    // the sort pass loads each from an aligned host address
    reg_cap[p] = (std::min<uint64_t>(n, (uint64_t)std::ceil(est)) + 127) / 128 * 128;
    reg_off[p] = regions;
    regions += reg_cap[p];
  }
  const uint64_t want = regions + n / 256 + kRxTile;
  uint64_t *mid_keys = nullptr;
  uint32_t *mid_vals = nullptr;
  uint64_t C = 0;  // pairs the intermediate holds
  bool contig = true;
  std::unique_ptr<char[]> own;
  HostReg reg_mid;
  std::deque<Spill> spills;
  if (depth == 0 && o.host_scratch && o.host_scratch_bytes >= 12 * n) {
    C = o.host_scratch_bytes / 12 / 128 * 128;  // the value array then starts 1 KB-aligned too
    contig = C >= want;  // else the blocked layout in the first 12 n bytes
    if (!contig) C = n;
    mid_keys = (uint64_t *)o.host_scratch;
    mid_vals = (uint32_t *)((char *)o.host_scratch + 8 * C);
    VX_TRY(reg_mid.add(o.host_scratch, 12 * C));
  } else {
    C = (regions + n / 64 + kRxTile + 127) / 128 * 128;
    own.reset(new (std::nothrow) char[12 * C + 4096]);
    if (!own) {
      set_error("vx_sort: no host memory for the %llu-pair intermediate", (unsigned long long)C);
      return VX_E_NOMEM;
    }
    char *base = (char *)(((uintptr_t)own.get() + 4095) & ~(uintptr_t)4095);  // page-aligned
    mid_keys = (uint64_t *)base;
    mid_vals = (uint32_t *)(base + 8 * C);
    VX_TRY(reg_mid.add(base, 12 * C));
  }

  // ---- pass 1: partition
  double tp = now_ms();
  PartitionPass pp;
  {
    uint64_t *h_bnd = nullptr;
    VX_CUDA_TRY(cudaHostAlloc((void **)&h_bnd, 8 * n_chunks * (P + 1), cudaHostAllocDefault));
    struct FreeHost {
      void *p;
      ~FreeHost() { cudaFreeHost(p); }
    } free_bnd{h_bnd};
    pp.ctx = ctx;
    pp.keys = keys;
    pp.vals = vals;
    pp.n = n;
    pp.R = R;
    pp.P = P;
    pp.d_spl = d_spl;
    pp.mid_keys = mid_keys;
    pp.mid_vals = mid_vals;
    pp.h_bnd = h_bnd;
    pp.contig = contig;
    pp.C = C;
    pp.reg_off = reg_off;
    pp.reg_cap = reg_cap;
    pp.used.assign(P, 0);
    pp.ovf = regions;
    pp.spills = &spills;
    pp.ext.resize(P);
    ExecStats es;
    VX_TRY(run_pipeline(ctx, pp, &es));
    VX_CUDA_TRY(cudaStreamSynchronize(ctx->s_compute));
    ss.bytes_h2d += es.bytes_h2d;
    ss.bytes_d2h += es.bytes_d2h;
    ss.kernel_launches += es.kernel_launches * 4;  // upsweep, row scan, totals, scatter
  }
  ss.ms_partition += now_ms() - tp;

  // ---- partition sizes and output offsets
  std::vector<uint64_t> psize(P, 0), poff(P, 0);
  for (uint32_t p = 0; p < P; ++p) {
    for (const Extent &e : pp.ext[p]) psize[p] += e.len;
    if (contig) ss.out_of_region_pairs += psize[p] - pp.used[p];
  }
  ss.spill_buffers += spills.size();
  if (depth == 0) ss.contiguous_layout = contig ? 1u : 0u;
  for (uint32_t p = 1; p < P; ++p) poff[p] = poff[p - 1] + psize[p - 1];
  auto extents = [&](uint32_t p) { return pp.ext[p]; };
  uint64_t mx = 0, mn = UINT64_MAX;
  for (uint32_t p = 0; p < P; ++p) {
    mx = std::max(mx, psize[p]);
    mn = std::min(mn, psize[p]);
  }
  if (depth == 0) {
    ss.n_partitions = P;
    ss.max_partition = mx;
    ss.min_partition = mn;
    ss.imbalance = (double)mx / ((double)n / P);
  }

  // ---- pass 2: sort the partitions that fit; copy through single-key ones;
  // recurse on the others
  double tq = now_ms();
  SortPass sp;
  sp.ctx = ctx;
  sp.cap = cap;
  sp.out_keys = out_keys;
  sp.out_vals = out_vals;
  sp.S = S;
  std::vector<uint32_t> big;
  for (uint32_t p = 0; p < P; ++p) {
    if (psize[p] == 0) continue;
    if (psize[p] <= cap) {
      sp.ext.push_back(extents(p));
      sp.job_n.push_back(psize[p]);
      sp.job_off.push_back(poff[p]);
    } else {
      big.push_back(p);
    }
  }
  {
    // Slots sized by the largest job, as many as fit (at most kMaxSortSlots):
    // a job's load, sort and store take about the same time, so with three
    // slots the next load waits for a store and every uneven partition leaves
    // the device idle; more slots let loads run ahead.  Never fewer than the
    // S slots of `cap` pairs the partition count was planned for.
    uint64_t jcap = 0;
    for (uint64_t x : sp.job_n) jcap = std::max(jcap, x);
    jcap = (jcap + kRxTile - 1) / kRxTile * kRxTile;
    if (jcap) {
      sp.cap = jcap;
      const uint64_t sb = (sp.slot_bytes() + 255) & ~255ull;
      sp.S = std::max<int>(S, (int)std::min<uint64_t>(kMaxSortSlots, ctx->arena.largest_free() / sb));
    }
    ExecStats es;
    VX_TRY(run_pipeline(ctx, sp, &es));
    ss.bytes_h2d += es.bytes_h2d;
    ss.bytes_d2h += es.bytes_d2h;
    ss.kernel_launches += es.kernel_launches * (radix_launches() + 1);  // and publish
    ss.ms_sort_kernel += es.ms_kernel;
    ss.radix_pass_pairs += sp.pass_pairs;
  }
  for (uint32_t p : big) {
    std::vector<Extent> ex = extents(p);
    if (single_key_partition(spl, p)) {  // already in input order: copy through
      uint64_t at = poff[p];
      for (const Extent &e : ex) {
        parallel_copy(out_keys + at, e.k, 8 * e.len);
        parallel_copy(out_vals + at, e.v, 4 * e.len);
        at += e.len;
      }
      ss.passthrough_partitions += 1;
      continue;
    }
    if (depth >= 3) {
      set_error("vx_sort: partition of %llu pairs still exceeds the slot after 3 levels",
                (unsigned long long)psize[p]);
      return VX_E_CAPACITY;
    }
    ss.overflow_retries += 1;
    // gather the partition contiguously (in input order) and sort it recursively
    std::vector<char> tmp(psize[p] * 12);
    uint64_t *tk = (uint64_t *)tmp.data();
    uint32_t *tv = (uint32_t *)(tmp.data() + 8 * psize[p]);
    uint64_t at = 0;
    for (const Extent &e : ex) {
      parallel_copy(tk + at, e.k, 8 * e.len);
      parallel_copy(tv + at, e.v, 4 * e.len);
      at += e.len;
    }
    HostReg rt;
    VX_TRY(rt.add(tmp.data(), tmp.size()));
    void *dk = nullptr;
    VX_CUDA_TRY(cudaHostGetDevicePointer(&dk, tk, 0));
    vx_sort_opts o2 = o;
    o2.n_partitions = 0;
    VX_TRY(sort_pairs(ctx, tk, tv, (const uint64_t *)dk, psize[p], out_keys + poff[p], out_vals + poff[p], o2, ss,
                      depth + 1, false));
  }
  ss.ms_sort += now_ms() - tq;
  return VX_OK;
}

vx_status sort_contiguous(vx_ctx *ctx, const uint64_t *keys, const uint32_t *vals, const uint64_t *dev_keys, uint64_t n,
                          uint64_t *out_keys, uint32_t *out_vals, const vx_sort_opts &o, vx_sort_stats &ss, int depth) {
  return sort_pairs(ctx, keys, vals, dev_keys, n, out_keys, out_vals, o, ss, depth, true);
}

}  // namespace vx

using namespace vx;

VX_API vx_status vx_sort(vx_ctx *ctx, int32_t key_col, int32_t rowid_col, uint64_t *out_keys, uint32_t *out_rowids,
                         const vx_sort_opts *opts, vx_sort_stats *stats) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  const Column *kc = get_col(ctx, key_col, VX_U64);
  const Column *vc = get_col(ctx, rowid_col, VX_U32);
  if (!kc || !vc) return VX_E_INVAL;
  if (kc->n_rows != vc->n_rows || ((!out_keys || !out_rowids) && kc->n_rows)) {
    set_error("vx_sort: columns differ in length or null output");
    return VX_E_INVAL;
  }
  vx_sort_opts o{};
  if (opts) o = *opts;
  if (o.partitioner < VX_PART_SAMPLE || o.partitioner > VX_PART_LEARNED_MLP || o.n_partitions < 0 ||
      o.n_partitions > 256 || (o.plan != VX_SORT_PARTITION && o.plan != VX_SORT_MERGE) || o.runs_mode < 0 ||
      o.runs_mode > 1) {
    set_error("vx_sort: bad options");
    return VX_E_INVAL;
  }
  const uint64_t n = kc->n_rows;
  HostReg r1, r2;
  VX_TRY(r1.add(out_keys, 8 * n));
  VX_TRY(r2.add(out_rowids, 4 * n));
  vx_sort_stats ss{};
  double t0 = now_ms();
  vx_status st = o.plan == VX_SORT_MERGE
                     ? merge_sort_plan(ctx, (const uint64_t *)kc->host, (const uint32_t *)vc->host,
                                       (const uint64_t *)kc->dev, n, out_keys, out_rowids, o, ss)
                     : sort_contiguous(ctx, (const uint64_t *)kc->host, (const uint32_t *)vc->host,
                                       (const uint64_t *)kc->dev, n, out_keys, out_rowids, o, ss, 0);
  ss.ms_total = now_ms() - t0;
  if (stats) *stats = ss;
  return st;
}

// Pairs from which vx_radix_sort_pairs asks a sample whether the low key bytes can
// be left to a repair.  The whole call with and without, uniform keys: 30K 157 and
// 155 us, 60K 153 and 162, 500K 215 and 248, 3M 633 and 762; when the answer is no
// the sample costs a few us of a small call (it is under the values' copy).
constexpr uint64_t kPairSampleMin = 1 << 15;

VX_API vx_status vx_radix_sort_pairs(vx_ctx *ctx, const uint64_t *keys, const uint32_t *vals, uint64_t n,
                                     uint64_t *out_keys, uint32_t *out_vals) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  if (n && (!keys || !vals || !out_keys || !out_vals)) {
    set_error("vx_radix_sort_pairs: null buffer");
    return VX_E_INVAL;
  }
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  if (n == 0) return VX_OK;
  DevBuf buf;
  buf.arena = &ctx->arena;
  const uint64_t kb = (8 * n + 255) & ~255ull, vb = (4 * n + 255) & ~255ull;
  buf.p = ctx->arena.alloc(2 * kb + 2 * vb + radix_temp_bytes(n));
  if (!buf.p) {
    set_error("vx_radix_sort_pairs: %llu pairs do not fit the arena", (unsigned long long)n);
    return VX_E_NOMEM;
  }
  char *p = buf.as<char>();
  RadixBufs b;
  b.keys[0] = (uint64_t *)p;
  b.keys[1] = (uint64_t *)(p + kb);
  b.vals[0] = (uint32_t *)(p + 2 * kb);
  b.vals[1] = (uint32_t *)(p + 2 * kb + vb);
  char *temp = p + 2 * kb + 2 * vb;
  cudaStream_t s = ctx->s_compute;
  const bool sample = n >= kPairSampleMin && n >> 32 == 0;
  // Where the keys are sampled, the values cross the link on the other stream
  // meanwhile: behind all that the compute stream was given before this call
  // (which may still use the arena), and waited for before the block goes back
  // to the arena, also when the call ends early.
  struct ValsIn {
    cudaStream_t other;
    cudaEvent_t e = nullptr;
    bool copying = false;
    ~ValsIn() {
      if (copying) cudaStreamSynchronize(other);
      if (e) cudaEventDestroy(e);
    }
  } vals_in{ctx->s_h2d};
  if (sample) {
    VX_CUDA_TRY(cudaEventCreateWithFlags(&vals_in.e, cudaEventDisableTiming));
    const cudaError_t idle = cudaStreamQuery(s);
    if (idle != cudaSuccess) {  // work left; where there is none, asking costs 2 us of a call and the wait up to 7
      if (idle != cudaErrorNotReady) VX_CUDA_TRY(idle);
      VX_CUDA_TRY(cudaEventRecord(vals_in.e, s));
      VX_CUDA_TRY(cudaStreamWaitEvent(ctx->s_h2d, vals_in.e, 0));
    }
  }
  VX_CUDA_TRY(cudaMemcpyAsync(b.keys[0], keys, 8 * n, cudaMemcpyHostToDevice, s));
  volatile uint64_t *word = ctx->h_scalars + 64;
  const uint32_t m = (uint32_t)std::min<uint64_t>(n, kPairSample);
  if (sample) {
    static OncePerDevice once;
    VX_TRY(raise_smem_limit(once, pair_prefix_kernel, sizeof(PairSampleSmem)));
    pair_prefix_kernel<<<1, 1024, sizeof(PairSampleSmem), s>>>(b.keys[0], n, m, ctx->d_scalars + 64);
    VX_CUDA_TRY(cudaGetLastError());
  }
  VX_CUDA_TRY(cudaMemcpyAsync(b.vals[0], vals, 4 * n, cudaMemcpyHostToDevice, sample ? ctx->s_h2d : s));
  int first = 0;
  if (sample) {
    vals_in.copying = true;
    VX_CUDA_TRY(cudaEventRecord(vals_in.e, ctx->s_h2d));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    const uint64_t c[4] = {word[0], word[1], word[2], word[3]};
    first = prefix_bytes(c, m, n, true);
  }
  const uint32_t limit = ctx->cfg.lookback_spin_limit;
  int cur = 0;
  bool redo = false;
  VX_TRY(first ? radix_prefix_sort_enqueue(b, n, temp, s, ctx->num_sms, first, limit, vals_in.e)
               : radix_sort_enqueue(b, n, temp, s, ctx->num_sms, 8, limit, false, vals_in.e));
  VX_TRY(radix_result(temp, s, &cur, first ? &redo : nullptr));
  vals_in.copying = false;  // s, which has waited for them, has been waited for
  if (redo) {  // a prefix that many keys share: sort in full, from where the pairs are
    if (cur) {
      std::swap(b.keys[0], b.keys[1]);
      std::swap(b.vals[0], b.vals[1]);
    }
    VX_TRY(radix_sort_enqueue(b, n, temp, s, ctx->num_sms, 8, limit));
    VX_TRY(radix_result(temp, s, &cur));
  }
  VX_CUDA_TRY(cudaMemcpyAsync(out_keys, b.keys[cur], 8 * n, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaMemcpyAsync(out_vals, b.vals[cur], 4 * n, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  return VX_OK;
}

VX_API vx_status vx_range_partition(vx_ctx *ctx, const uint64_t *keys, const uint32_t *vals, uint64_t n,
                                    const uint64_t *splitters, uint32_t n_partitions, uint64_t *out_keys,
                                    uint32_t *out_vals, uint64_t *boundary) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  if (n_partitions < 1 || n_partitions > 256 || (n_partitions > 1 && !splitters) || !boundary ||
      (n && (!keys || !vals || !out_keys || !out_vals))) {
    set_error("vx_range_partition: bad argument");
    return VX_E_INVAL;
  }
  for (uint32_t i = 1; i + 1 < n_partitions; ++i)
    if (splitters[i] < splitters[i - 1]) {
      set_error("vx_range_partition: splitters must be non-decreasing");
      return VX_E_INVAL;
    }
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  DevBuf buf;
  buf.arena = &ctx->arena;
  const uint64_t kb = (8 * std::max<uint64_t>(n, 1) + 255) & ~255ull, vb = (4 * std::max<uint64_t>(n, 1) + 255) & ~255ull;
  buf.p = ctx->arena.alloc(2 * kb + 2 * vb + radix_temp_bytes(std::max<uint64_t>(n, 1)) + 8 * 256);
  if (!buf.p) {
    set_error("vx_range_partition: %llu pairs do not fit the arena", (unsigned long long)n);
    return VX_E_NOMEM;
  }
  char *p = buf.as<char>();
  RadixBufs b;
  b.keys[0] = (uint64_t *)p;
  b.keys[1] = (uint64_t *)(p + kb);
  b.vals[0] = (uint32_t *)(p + 2 * kb);
  b.vals[1] = (uint32_t *)(p + 2 * kb + vb);
  char *temp = p + 2 * kb + 2 * vb;
  uint64_t *d_spl = (uint64_t *)(temp + radix_temp_bytes(std::max<uint64_t>(n, 1)));
  cudaStream_t s = ctx->s_compute;
  if (n_partitions > 1) VX_CUDA_TRY(cudaMemcpyAsync(d_spl, splitters, 8 * (n_partitions - 1), cudaMemcpyHostToDevice, s));
  if (n) {
    VX_CUDA_TRY(cudaMemcpyAsync(b.keys[0], keys, 8 * n, cudaMemcpyHostToDevice, s));
    VX_CUDA_TRY(cudaMemcpyAsync(b.vals[0], vals, 4 * n, cudaMemcpyHostToDevice, s));
  }
  VX_TRY(range_partition_enqueue(b, n, d_spl, n_partitions, temp, s));
  RadixState *st = radix_state_of(temp);
  VX_CUDA_TRY(cudaMemcpyAsync(boundary, st->base, 8ull * (n_partitions + 1), cudaMemcpyDeviceToHost, s));
  if (n) {
    VX_CUDA_TRY(cudaMemcpyAsync(out_keys, b.keys[1], 8 * n, cudaMemcpyDeviceToHost, s));
    VX_CUDA_TRY(cudaMemcpyAsync(out_vals, b.vals[1], 4 * n, cudaMemcpyDeviceToHost, s));
  }
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  boundary[n_partitions] = n;
  return VX_OK;
}

VX_API vx_status vx_sort_splitters(vx_ctx *ctx, int32_t key_col, int32_t partitioner, uint32_t n_partitions,
                                   uint64_t sample_size, uint64_t seed, uint64_t *splitters_out, uint32_t *n_out) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  const Column *kc = get_col(ctx, key_col, VX_U64);
  if (!kc) return VX_E_INVAL;
  if (n_partitions < 2 || n_partitions > kMaxRequestedPartitions || !splitters_out || !n_out || kc->n_rows == 0) {
    set_error("vx_sort_splitters: need 2..%u partitions, outputs, non-empty column", kMaxRequestedPartitions);
    return VX_E_INVAL;
  }
  uint64_t m = std::min<uint64_t>(sample_size ? sample_size : (1ull << 20), kc->n_rows);
  DevBuf sbuf, splbuf;
  uint64_t *sorted = nullptr;
  VX_TRY(sample_and_sort(ctx, (const uint64_t *)kc->dev, kc->n_rows, m, seed, sbuf, &sorted));
  splbuf.arena = &ctx->arena;
  splbuf.p = ctx->arena.alloc(kSplitterBufBytes);
  if (!splbuf.p) return VX_E_NOMEM;
  uint64_t *d_spl = splbuf.as<uint64_t>();
  double ms = 0;
  uint32_t k = 0;
  VX_TRY(splitters_from_sample(ctx, partitioner, sorted, m, n_partitions, d_spl, 0, &ms, &k));
  if (k) VX_CUDA_TRY(cudaMemcpyAsync(splitters_out, d_spl, 8ull * k, cudaMemcpyDeviceToHost, ctx->s_compute));
  VX_CUDA_TRY(cudaStreamSynchronize(ctx->s_compute));
  *n_out = k;
  return VX_OK;
}
