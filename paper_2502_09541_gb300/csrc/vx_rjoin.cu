// Radix-partitioned hash join (Section 6.2): the paper's RadixPartitionExKer
// and HashJoinExKer, for an equi-join of two tables larger than the budget.
//
// RadixPartitionExKer.  Each chunk of a table is clustered by the low b bits
// of the key (b = 24: 2^24 groups): a stable LSD radix sort over the low b/8
// key bytes of (key, chunk-local row) pairs, then find_boundary (Section
// 6.2.1, Fig. 9) — a boundary array of 2^b + 1 entries starts as
// placeholders, every position whose group differs from the previous
// position's records itself at its group's entry, the last entry is the
// chunk length, and each remaining placeholder takes the next valid entry to
// its right (a suffix minimum).  The clustered keys, the build side's
// payloads (gathered by the sorted local rows) or the probe side's local rows,
// and the boundary array go back to host memory.
//
// HashJoinExKer.  The data mapping cuts the 2^b groups into ranges whose
// tuples fit a staging slot, by binary search over the boundary arrays (the
// tuples of groups [g0, g1) in chunk c are [B_c[g0], B_c[g1]) of its
// clustered chunk).  A range's segments of every chunk of both tables and the
// slices B_c[g0 .. g1] of their boundary arrays are loaded; blocks join runs of
// consecutive groups in shared memory (rj_join_kernel).  Matches add to a
// count, a wrapping payload sum and the pair fingerprint
// mix64(probe_row ^ rotl(payload, 17)), probe_row = chunk * R + local row.
//
// When the clustered tables fit the arena beside the partition pass's slots,
// they stay there: nothing is stored to host memory or loaded again, and the
// boundary arrays hold only the ends of the block's runs of groups.
#include <algorithm>
#include <cmath>

#include "vx_internal.h"
#include "vx_sort.cuh"

namespace vx {

namespace {

constexpr uint32_t kRjNone = 0xFFFFFFFFu;  // boundary placeholder
constexpr int kRjSeg = 4096;               // boundary entries per block of the back-fill
constexpr int kRjThreads = 256;
constexpr uint32_t kRjTable = 2048;        // slots of a block's shared-memory table
constexpr uint32_t kRjPiece = kRjTable / 2;  // build tuples in it at once
constexpr uint32_t kRjRunBuild = 768;      // build tuples of a run of groups, on average at most
constexpr uint64_t kRjPart = 32768;        // probe tuples of one work item, at most
constexpr uint64_t kRjEmpty = ~0ull;       // empty slot key; a build key equal to it is kept aside

__device__ __forceinline__ uint64_t rj_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void rj_iota_kernel(uint32_t *v, uint64_t n) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    v[i] = (uint32_t)i;
}

// find_boundary, step 2: a position whose group differs from the previous
// position's records itself at its group's entry; the last entry is n
__global__ void rj_mark_kernel(const uint64_t *k0, const uint64_t *k1, const RadixState *st, int npass, uint64_t n,
                               uint64_t mask, uint32_t *bnd) {
  const uint64_t *k = st->cur[npass] ? k1 : k0;
  const uint64_t G = mask + 1;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t h = k[i] & mask;
    if (i == 0 || h != (k[i - 1] & mask)) bnd[h] = (uint32_t)i;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) bnd[G] = (uint32_t)n;
}

// find_boundary, step 3: each placeholder takes the next valid entry to its
// right.  Valid entries increase along the array, so that is the suffix
// minimum; per segment of kRjSeg entries first (its minimum to carry[seg]),
// then over the segments' carries, then applied.
__global__ void __launch_bounds__(256) rj_fill_local_kernel(uint32_t *bnd, uint64_t m, uint32_t *carry) {
  __shared__ uint32_t tmin[256];
  const uint64_t s0 = (uint64_t)blockIdx.x * kRjSeg;
  constexpr int kPer = kRjSeg / 256;
  const uint64_t a = s0 + (uint64_t)threadIdx.x * kPer;
  uint32_t v[kPer];
  uint32_t run = kRjNone;
#pragma unroll
  for (int j = kPer - 1; j >= 0; --j) {
    v[j] = a + j < m ? bnd[a + j] : kRjNone;
    run = v[j] < run ? v[j] : run;
    v[j] = run;
  }
  tmin[threadIdx.x] = run;
  __syncthreads();
  // minimum over the threads to the right (a suffix scan over 256 values)
  for (int off = 1; off < 256; off <<= 1) {
    const uint32_t y = threadIdx.x + off < 256 ? tmin[threadIdx.x + off] : kRjNone;
    __syncthreads();
    if (y < tmin[threadIdx.x]) tmin[threadIdx.x] = y;
    __syncthreads();
  }
  const uint32_t right = threadIdx.x + 1 < 256 ? tmin[threadIdx.x + 1] : kRjNone;
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (a + j < m) bnd[a + j] = v[j] < right ? v[j] : right;
  if (threadIdx.x == 0) carry[blockIdx.x] = tmin[0];
}

__global__ void __launch_bounds__(1024) rj_fill_carry_kernel(uint32_t *carry, uint32_t nseg) {
  // one block: carry[s] becomes the minimum over segments after s (exclusive suffix minimum)
  __shared__ uint32_t sm[1024];
  uint32_t run = kRjNone;
  const uint32_t per = (nseg + 1023) / 1024;
  const uint32_t a = threadIdx.x * per;
  for (uint32_t j = 0; j < per; ++j)
    if (a + j < nseg && carry[a + j] < run) run = carry[a + j];
  sm[threadIdx.x] = run;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const uint32_t y = threadIdx.x + off < 1024 ? sm[threadIdx.x + off] : kRjNone;
    __syncthreads();
    if (y < sm[threadIdx.x]) sm[threadIdx.x] = y;
    __syncthreads();
  }
  uint32_t after = threadIdx.x + 1 < 1024 ? sm[threadIdx.x + 1] : kRjNone;
  for (int j = (int)per - 1; j >= 0; --j) {
    if (a + j >= nseg) continue;
    const uint32_t own = carry[a + j];
    carry[a + j] = after;
    if (own < after) after = own;
  }
}

__global__ void rj_fill_apply_kernel(uint32_t *bnd, uint64_t m, const uint32_t *carry) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t c = carry[i / kRjSeg];
    if (c < bnd[i]) bnd[i] = c;
  }
}

// payload of the clustered build tuples: out[i] = in[sorted local row i]
__global__ void rj_gather_kernel(const uint32_t *v0, const uint32_t *v1, const RadixState *st, int npass, uint64_t n,
                                 const uint64_t *in, uint64_t *out) {
  const uint32_t *v = st->cur[npass] ? v1 : v0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = in[v[i]];
}

struct RjAcc {
  unsigned long long count, psum, fp;
  uint32_t err;
};

// resident mode, after a chunk's clustering: buffer `home` is the resident
// array, where the passes have left the keys (and the probe side's rows) unless
// an odd number of them was skipped.  The build side's payloads follow in
// clustered order.
__global__ void rj_keep_kernel(const RadixBufs b, int home, const RadixState *st, int npass, uint64_t n,
                               const uint64_t *pay, uint64_t *opay, RjAcc *acc) {
  const int c = st->cur[npass];
  const uint64_t *k = c ? b.keys[1] : b.keys[0];
  const uint32_t *v = c ? b.vals[1] : b.vals[0];
  bool moved = false;
  for (int q = 0; q < npass; ++q) moved = moved || !st->skip[q];
  if (st->err && blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&acc->err, ERR_WAIT);
  if (c == home && moved && !opay) return;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t row = moved ? v[i] : (uint32_t)i;
    if (c != home) b.keys[home][i] = k[i];
    if (opay) opay[i] = pay[row];
    else b.vals[home][i] = row;
  }
}

// resident mode: where the runs of 2^shift groups start in each clustered chunk
// of R tuples (chunk c: bnd[c * (n_runs + 1) + r] for r <= n_runs), by binary
// search: a run has hundreds of tuples, so this reads far less than the keys
__global__ void rj_cuts_kernel(const uint64_t *keys, uint64_t n, uint64_t R, uint64_t mask, int shift, uint32_t n_runs,
                               uint32_t *bnd) {
  const uint64_t r0 = blockIdx.y * R;
  const uint64_t *k = keys + r0;
  const uint32_t m = (uint32_t)(n - r0 < R ? n - r0 : R);
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r <= n_runs; r += gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = m;
    while (lo < hi) {
      const uint32_t mid = lo + (hi - lo) / 2;
      if ((k[mid] & mask) >> shift < r) lo = mid + 1; else hi = mid;
    }
    bnd[blockIdx.y * (n_runs + 1ull) + r] = lo;
  }
}

// one range of groups, all chunks of both tables in device memory
struct RjJoinParams {
  const uint64_t *akeys, *apay;  // build tuples of the range, chunk after chunk
  const uint64_t *bkeys;         // probe tuples of the range, chunk after chunk
  const uint32_t *brows;         // their chunk-local rows
  const uint32_t *abnd, *bbnd;   // per chunk, boundary slice B_c[g0 .. g1] (ng + 1 entries)
  const uint64_t *abase, *bbase; // per chunk, first tuple of the chunk's segment
  uint32_t na, nb, ng;           // build chunks, probe chunks, groups of the range
  uint32_t step, n_runs;         // groups per run, runs of the range
  uint64_t probe_chunk_rows;     // R of the probe side's partition pass
  RjAcc *acc;
  uint2 *items;                  // work items (run, part of its probe tuples)
  unsigned int *n_items, *next;  // how many there are; the next one to take
};

__device__ __forceinline__ uint64_t rj_run_tuples(const uint32_t *bnd, uint32_t nchunks, uint64_t ng1, uint32_t ga,
                                                  uint32_t gb) {
  uint64_t t = 0;
  for (uint32_t c = 0; c < nchunks; ++c) t += bnd[c * ng1 + gb] - bnd[c * ng1 + ga];
  return t;
}

// one thread per run of groups: a run is joined by as many work items as its
// probe tuples need (a skewed run is spread over many blocks), none when it has
// no build tuple (or one, which cannot repeat, and no probe tuple)
__global__ void rj_items_kernel(const RjJoinParams p) {
  if (p.acc->err) return;  // a clustering pass gave up a wait: its boundaries mean nothing
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < p.n_runs; r += gridDim.x * blockDim.x) {
    const uint32_t ga = r * p.step, gb = ga + p.step < p.ng ? ga + p.step : p.ng;
    const uint64_t a = rj_run_tuples(p.abnd, p.na, (uint64_t)p.ng + 1, ga, gb);
    if (a == 0) continue;
    const uint64_t b = rj_run_tuples(p.bbnd, p.nb, (uint64_t)p.ng + 1, ga, gb);
    if (b == 0 && a == 1) continue;
    const uint32_t parts = (uint32_t)((b + kRjPart - 1) / kRjPart) + (b == 0 ? 1u : 0u);
    const unsigned int at = atomicAdd(p.n_items, parts);
    for (uint32_t q = 0; q < parts; ++q) p.items[at + q] = make_uint2(r, q);
  }
}

// A run's tuples of one side, chunk after chunk: thread t of the block reads
// the boundaries of chunk c0 + t, a block scan gives where its tuples start.
struct RjSegs {
  uint64_t start[kRjThreads + 1];  // ordinal of the chunk's first tuple among the batch's
  uint64_t at[kRjThreads];         // its index in the side's arrays
  uint64_t wsum[kRjThreads / 32];
};
__device__ __forceinline__ void rj_segs(RjSegs &s, const uint32_t *bnd, const uint64_t *base, uint32_t nchunks,
                                        uint32_t c0, uint64_t ng1, uint32_t ga, uint32_t gb) {
  const uint32_t c = c0 + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t m = 0;
  if (c < nchunks) {
    const uint32_t *bd = bnd + c * ng1;
    const uint32_t lo = bd[ga];
    m = bd[gb] - lo;
    s.at[threadIdx.x] = base[c] + (lo - bd[0]);
  }
  uint64_t x = m;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= (uint32_t)o) x += y;
  }
  if (lane == 31) s.wsum[w] = x;
  __syncthreads();
  for (uint32_t q = 0; q < w; ++q) x += s.wsum[q];
  s.start[threadIdx.x + 1] = x;
  if (threadIdx.x == 0) s.start[0] = 0;
  __syncthreads();
}

// Calls f(chunk, index) for the run's tuples of one side with ordinals
// [o0, o1), the block's threads on consecutive ones, kU of them at a time:
// f gets kU chunks and indices (index ~0: none).  Every thread must call it.
template <int kU, class F>
__device__ __forceinline__ void rj_for_tuples(RjSegs &s, const uint32_t *bnd, const uint64_t *base, uint32_t nchunks,
                                              uint64_t ng1, uint32_t ga, uint32_t gb, uint64_t o0, uint64_t o1, F &&f) {
  uint64_t done = 0;
  for (uint32_t c0 = 0; c0 < nchunks && done < o1; c0 += kRjThreads) {
    rj_segs(s, bnd, base, nchunks, c0, ng1, ga, gb);
    const uint32_t m = nchunks - c0 < (uint32_t)kRjThreads ? nchunks - c0 : (uint32_t)kRjThreads;
    const uint64_t total = s.start[m];
    const uint64_t lo = o0 > done ? o0 - done : 0, hi = o1 - done < total ? o1 - done : total;
    uint32_t a = 0;  // the chunk of the thread's latest tuple: its ordinals only grow
    for (uint64_t i0 = lo; i0 < hi; i0 += kU * kRjThreads) {
      uint32_t ch[kU];
      uint64_t ix[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const uint64_t i = i0 + (uint64_t)u * kRjThreads + threadIdx.x;
        ix[u] = ~0ull;
        ch[u] = 0;
        if (i < hi) {
          // the last chunk that starts at or before i: mostly the same or the next
          if (i >= s.start[a + 1] && i >= s.start[++a + 1]) {
            uint32_t b = m - 1;
            for (++a; a < b;) {
              const uint32_t mid = (a + b + 1) / 2;
              if (s.start[mid] <= i) a = mid; else b = mid - 1;
            }
          }
          ch[u] = c0 + a;
          ix[u] = s.at[a] + (i - s.start[a]);
        }
      }
      f(ch, ix);
    }
    done += total;
    __syncthreads();  // the segments are read no more
  }
}

// HashJoinExKer: a block takes (run of groups, part of its probe tuples) items,
// puts the run's build tuples into an open-addressing table in shared memory
// and probes it with the part's probe tuples.  The clustered layout makes both
// contiguous within each chunk, so the loads coalesce and a run costs two
// boundary reads per chunk and side.  A run with more build tuples than the
// table takes is joined piece by piece (a probe key matches in one piece at
// most). 
__global__ void __launch_bounds__(kRjThreads) rj_join_kernel(const RjJoinParams p) {
  __shared__ unsigned long long tkey[kRjTable], tpay[kRjTable];
  __shared__ RjSegs segs;
  __shared__ unsigned long long sent[2];  // a build key equal to kRjEmpty: present flag, payload
  __shared__ unsigned int s_item;
  const unsigned int n_items = *p.n_items;
  const uint64_t ng1 = (uint64_t)p.ng + 1;
  unsigned long long cnt = 0, psum = 0, fp = 0;
  for (;;) {
    if (threadIdx.x == 0) s_item = atomicAdd(p.next, 1u);
    __syncthreads();
    const unsigned int it = s_item;
    if (it >= n_items) break;
    const uint2 item = p.items[it];
    const uint32_t ga = item.x * p.step, gb = ga + p.step < p.ng ? ga + p.step : p.ng;
    const uint64_t nbuild = rj_run_tuples(p.abnd, p.na, ng1, ga, gb);
    for (uint64_t piece = 0; piece < nbuild; piece += kRjPiece) {
      const uint64_t pend = piece + kRjPiece < nbuild ? piece + kRjPiece : nbuild;
      uint32_t cap = 64;
      while (cap < 2 * (uint32_t)(pend - piece)) cap <<= 1;
      for (uint32_t i = threadIdx.x; i < cap; i += kRjThreads) tkey[i] = kRjEmpty;
      if (threadIdx.x == 0 && piece == 0) sent[0] = 0;
      __syncthreads();
      // the slot of key k, or of the empty slot that ends its walk (the table
      // is at most half full)
      auto find = [&](uint64_t k) {
        uint32_t h = (uint32_t)rj_mix(k) & (cap - 1);
        while (tkey[h] != k && tkey[h] != kRjEmpty) h = (h + 1) & (cap - 1);
        return h;
      };
      rj_for_tuples<1>(segs, p.abnd, p.abase, p.na, ng1, ga, gb, piece, pend, [&](const uint32_t *, const uint64_t *ix) {
        if (ix[0] == ~0ull) return;
        const uint64_t k = p.akeys[ix[0]], pay = p.apay[ix[0]];
        if (k == kRjEmpty) {
          if (atomicExch(&sent[0], 1ull)) atomicOr(&p.acc->err, ERR_DUPKEY);
          sent[1] = pay;
          return;
        }
        uint32_t h = (uint32_t)rj_mix(k) & (cap - 1);
        for (;;) {  // the table is at most half full: an empty slot ends every walk
          const unsigned long long old = atomicCAS(&tkey[h], kRjEmpty, k);
          if (old == kRjEmpty) {
            tpay[h] = pay;
            break;
          }
          if (old == k) {
            atomicOr(&p.acc->err, ERR_DUPKEY);
            break;
          }
          h = (h + 1) & (cap - 1);
        }
      });
      __syncthreads();
      if (pend < nbuild && item.y == 0)  // keys of later pieces must not repeat one of this piece
        rj_for_tuples<1>(segs, p.abnd, p.abase, p.na, ng1, ga, gb, pend, nbuild,
                         [&](const uint32_t *, const uint64_t *ix) {
                           if (ix[0] == ~0ull) return;
                           const uint64_t k = p.akeys[ix[0]];
                           if (k != kRjEmpty && tkey[find(k)] == k) atomicOr(&p.acc->err, ERR_DUPKEY);
                         });
      const bool last = pend == nbuild;  // the key equal to the empty marker is known by then
      rj_for_tuples<4>(segs, p.bbnd, p.bbase, p.nb, ng1, ga, gb, item.y * kRjPart, (item.y + 1ull) * kRjPart,
                       [&](const uint32_t *ch, const uint64_t *ix) {
                         uint64_t k[4];
                         uint32_t r[4];
#pragma unroll
                         for (int u = 0; u < 4; ++u) {
                           k[u] = ix[u] == ~0ull ? kRjEmpty : p.bkeys[ix[u]];
                           r[u] = ix[u] == ~0ull ? 0u : p.brows[ix[u]];  // in flight with the keys
                         }
#pragma unroll
                         for (int u = 0; u < 4; ++u) {
                           if (ix[u] == ~0ull) continue;
                           uint64_t pay;
                           if (k[u] == kRjEmpty) {
                             if (!last || !sent[0]) continue;
                             pay = sent[1];
                           } else {
                             const uint32_t h = find(k[u]);
                             if (tkey[h] != k[u]) continue;
                             pay = tpay[h];
                           }
                           const uint64_t row = (uint64_t)ch[u] * p.probe_chunk_rows + r[u];
                           cnt += 1;
                           psum += pay;
                           fp += rj_mix(row ^ ((pay << 17) | (pay >> 47)));
                         }
                       });
      __syncthreads();  // the table is read no more
    }
    __syncthreads();  // s_item is read no more
  }
  for (int off = 16; off > 0; off >>= 1) {
    cnt += __shfl_down_sync(0xffffffffu, cnt, off);
    psum += __shfl_down_sync(0xffffffffu, psum, off);
    fp += __shfl_down_sync(0xffffffffu, fp, off);
  }
  if ((threadIdx.x & 31) == 0 && cnt) {
    atomicAdd(&p.acc->count, cnt);
    atomicAdd(&p.acc->psum, psum);
    atomicAdd(&p.acc->fp, fp);
  }
}

int grid_for(vx_ctx *ctx, uint64_t items, int threads, int per_sm) {
  const uint64_t g = (items + threads - 1) / threads;
  return (int)std::max<uint64_t>(1, std::min<uint64_t>(g, (uint64_t)ctx->num_sms * per_sm));
}

// enqueues find_boundary of a clustered chunk (bnd: 2^bits + 1 entries)
vx_status find_boundary_enqueue(vx_ctx *ctx, RadixBufs b, const RadixState *st, int npass, uint64_t n, int bits,
                                uint32_t *bnd, uint32_t *carry, cudaStream_t s) {
  const uint64_t G = 1ull << bits, m = G + 1;
  VX_CUDA_TRY(cudaMemsetAsync(bnd, 0xFF, 4 * m, s));
  rj_mark_kernel<<<grid_for(ctx, n, 256, 8), 256, 0, s>>>(b.keys[0], b.keys[1], st, npass, n, G - 1, bnd);
  const uint32_t nseg = (uint32_t)((m + kRjSeg - 1) / kRjSeg);
  rj_fill_local_kernel<<<nseg, 256, 0, s>>>(bnd, m, carry);
  rj_fill_carry_kernel<<<1, 1024, 0, s>>>(carry, nseg);
  rj_fill_apply_kernel<<<grid_for(ctx, m, 256, 8), 256, 0, s>>>(bnd, m, carry);
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

// RadixPartitionExKer of one table: chunks of R tuples clustered into the host
// intermediate (keys, then payloads or local rows) plus a boundary array per chunk
struct RjPartitionPass : ExKernel {
  vx_ctx *ctx;
  const uint64_t *keys, *payload;  // payload null: the probe side (local rows are kept instead)
  uint64_t n, R;
  int bits, npass, S;
  int first = 0;  // resident: the lowest key byte that the clustering orders by
  uint64_t *mid_keys;
  uint64_t *mid_pay;    // build side
  uint32_t *mid_rows;   // probe side
  uint32_t *mid_bnd;    // chunk c at c * (2^bits + 1)
  // resident: mid_keys, mid_pay and mid_rows are device memory, which the
  // clustering writes; the slot holds the other buffer
  bool resident = false;
  RjAcc *acc = nullptr;
  uint64_t size() override { return (n + R - 1) / R; }
  int n_slots() override { return S; }
  int max_in_flight() override { return S; }
  uint64_t rows(uint64_t it) const { return std::min(R, n - it * R); }
  uint64_t G1() const { return (1ull << bits) + 1; }
  uint64_t kb() const { return (8 * R + 255) & ~255ull; }
  uint64_t vb() const { return (4 * R + 255) & ~255ull; }
  uint64_t bb() const { return (4 * G1() + 255) & ~255ull; }
  uint64_t cb() const { return (4 * ((G1() + kRjSeg - 1) / kRjSeg) + 255) & ~255ull; }
  uint64_t slot_bytes() override {
    if (resident) return kb() + 2 * vb() + radix_temp_bytes(R) + (payload ? kb() : 0);
    return 2 * kb() + 2 * vb() + radix_temp_bytes(R) + bb() + cb() + (payload ? 2 * kb() : 0);
  }
  RadixBufs bufs(char *slot) const {
    RadixBufs b;
    b.keys[0] = (uint64_t *)slot;
    b.keys[1] = (uint64_t *)(slot + kb());
    b.vals[0] = (uint32_t *)(slot + 2 * kb());
    b.vals[1] = (uint32_t *)(slot + 2 * kb() + vb());
    return b;
  }
  // resident: [keys | rows | rows (build side) | temp | payloads].  The passes
  // end in the resident arrays: an odd number starts from the slot, an even one
  // from the arrays themselves, into which the chunk is then loaded
  int home() const { return (npass - first) & 1; }
  RadixBufs resident_bufs(char *slot, uint64_t it) const {
    const int h = home();
    RadixBufs b;
    b.keys[1 - h] = (uint64_t *)slot;
    b.keys[h] = mid_keys + it * R;
    b.vals[1 - h] = (uint32_t *)(slot + kb());
    b.vals[h] = payload ? (uint32_t *)(slot + kb() + vb()) : mid_rows + it * R;
    return b;
  }
  char *temp(char *slot) const { return slot + (resident ? 1 : 2) * kb() + 2 * vb(); }
  uint32_t *bnd(char *slot) const { return (uint32_t *)(temp(slot) + radix_temp_bytes(R)); }
  uint32_t *carry(char *slot) const { return (uint32_t *)((char *)bnd(slot) + bb()); }
  uint64_t *pay_in(char *slot) const {
    return (uint64_t *)(resident ? temp(slot) + radix_temp_bytes(R) : (char *)carry(slot) + cb());
  }
  uint64_t *pay_out(char *slot) const { return (uint64_t *)((char *)pay_in(slot) + kb()); }
  void inputs(uint64_t it, char *slot, std::vector<CopyOp> &h2d) override {
    h2d.push_back({keys + it * R, (resident ? resident_bufs(slot, it) : bufs(slot)).keys[0], 8 * rows(it)});
    if (payload) h2d.push_back({payload + it * R, pay_in(slot), 8 * rows(it)});
  }
  vx_status kernel(char *slot, uint64_t it, cudaStream_t s) override {
    const uint64_t m = rows(it);
    if (resident) {
      const RadixBufs rb = resident_bufs(slot, it);
      VX_TRY(radix_sort_enqueue(rb, m, temp(slot), s, ctx->num_sms, npass, ctx->cfg.lookback_spin_limit, true,
                                nullptr, first));
      rj_keep_kernel<<<grid_for(ctx, m, 256, 8), 256, 0, s>>>(rb, home(), radix_state_of(temp(slot)), npass, m,
                                                              payload ? pay_in(slot) : nullptr,
                                                              payload ? mid_pay + it * R : nullptr, acc);
      VX_CUDA_TRY(cudaGetLastError());
      return VX_OK;
    }
    RadixBufs b = bufs(slot);
    rj_iota_kernel<<<grid_for(ctx, m, 256, 8), 256, 0, s>>>(b.vals[0], m);
    VX_TRY(radix_sort_enqueue(b, m, temp(slot), s, ctx->num_sms, npass, ctx->cfg.lookback_spin_limit));
    const RadixState *st = radix_state_of(temp(slot));
    VX_TRY(find_boundary_enqueue(ctx, b, st, npass, m, bits, bnd(slot), carry(slot), s));
    if (payload)
      rj_gather_kernel<<<grid_for(ctx, m, 256, 8), 256, 0, s>>>(b.vals[0], b.vals[1], st, npass, m, pay_in(slot),
                                                                pay_out(slot));
    VX_CUDA_TRY(cudaGetLastError());
    return radix_publish_enqueue(temp(slot), ctx->d_scalars + 64 + (it % S), s, npass);
  }
  bool has_outputs() override { return !resident; }
  vx_status outputs(uint64_t it, char *slot, std::vector<CopyOp> &d2h) override {
    RadixBufs b = bufs(slot);
    const uint64_t word = ((volatile uint64_t *)ctx->h_scalars)[64 + (it % S)];
    if (word >> 16 & 1) {
      set_error("radix join: the clustering sort of chunk %llu gave up a look-back wait", (unsigned long long)it);
      return VX_E_TIMEOUT;
    }
    const int c = (int)(word & 0xFF);
    const uint64_t m = rows(it);
    d2h.push_back({b.keys[c], mid_keys + it * R, 8 * m});
    if (payload) d2h.push_back({pay_out(slot), mid_pay + it * R, 8 * m});
    else d2h.push_back({b.vals[c], mid_rows + it * R, 4 * m});
    d2h.push_back({bnd(slot), mid_bnd + it * G1(), 4 * G1()});
    return VX_OK;
  }
};

// work items of a join over n_runs runs of groups and nb probe tuples: the
// counters, then the items
uint64_t rj_items_bytes(uint64_t n_runs, uint64_t nb) { return 256 + ((8 * (n_runs + nb / kRjPart + 1) + 255) & ~255ull); }

vx_status rj_join_enqueue(vx_ctx *ctx, RjJoinParams p, char *items, cudaStream_t s) {
  p.n_items = (unsigned int *)items;
  p.next = p.n_items + 1;
  p.items = (uint2 *)(items + 256);
  VX_CUDA_TRY(cudaMemsetAsync(items, 0, 8, s));
  rj_items_kernel<<<grid_for(ctx, p.n_runs, 256, 8), 256, 0, s>>>(p);
  rj_join_kernel<<<(unsigned)ctx->num_sms * 5, kRjThreads, 0, s>>>(p);
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

// one range of groups and where its pieces sit in a slot
struct RjRange {
  uint64_t g0, g1;
  uint64_t akeys, apay, bkeys, brows, abnd, bbnd, abase, bbase, items, bytes;  // byte offsets in the slot
  uint64_t na_tuples, nb_tuples;
};

// HashJoinExKer: ranges of groups, each joined in shared memory
struct RjJoinPass : ExKernel {
  vx_ctx *ctx;
  uint64_t slot_b;
  int S;
  uint32_t NA, NB;
  uint64_t G1, RA, RB;
  const uint64_t *akeys, *apay, *bkeys;
  const uint32_t *brows, *abnd_h, *bbnd_h;
  std::vector<RjRange> ranges;
  const uint64_t *base_h = nullptr;  // page-locked; per range NA + NB words: abase, then bbase
  uint32_t step;  // groups per run
  RjAcc *acc;
  std::vector<cudaEvent_t> ev0, ev1;
  double ms_join = 0;
  ~RjJoinPass() override {
    for (auto e : ev0) cudaEventDestroy(e);
    for (auto e : ev1) cudaEventDestroy(e);
  }
  uint64_t size() override { return ranges.size(); }
  int n_slots() override { return S; }
  int max_in_flight() override { return S; }
  uint64_t slot_bytes() override { return slot_b; }
  void inputs(uint64_t it, char *slot, std::vector<CopyOp> &h2d) override {
    const RjRange &r = ranges[it];
    const uint64_t ng1 = r.g1 - r.g0 + 1;
    for (uint32_t c = 0; c < NA; ++c) {
      const uint32_t *bd = abnd_h + c * G1;
      const uint64_t lo = bd[r.g0], hi = bd[r.g1], at = base_h[it * (NA + NB) + c];
      if (hi > lo) {
        h2d.push_back({akeys + c * RA + lo, slot + r.akeys + 8 * at, 8 * (hi - lo)});
        h2d.push_back({apay + c * RA + lo, slot + r.apay + 8 * at, 8 * (hi - lo)});
      }
      h2d.push_back({bd + r.g0, slot + r.abnd + 4 * c * ng1, 4 * ng1});
    }
    for (uint32_t c = 0; c < NB; ++c) {
      const uint32_t *bd = bbnd_h + c * G1;
      const uint64_t lo = bd[r.g0], hi = bd[r.g1], at = base_h[it * (NA + NB) + NA + c];
      if (hi > lo) {
        h2d.push_back({bkeys + c * RB + lo, slot + r.bkeys + 8 * at, 8 * (hi - lo)});
        h2d.push_back({brows + c * RB + lo, slot + r.brows + 4 * at, 4 * (hi - lo)});
      }
      h2d.push_back({bd + r.g0, slot + r.bbnd + 4 * c * ng1, 4 * ng1});
    }
    h2d.push_back({base_h + it * (NA + NB), slot + r.abase, 8ull * (NA + NB)});
  }
  vx_status kernel(char *slot, uint64_t it, cudaStream_t s) override {
    const RjRange &r = ranges[it];
    RjJoinParams p{};
    p.akeys = (const uint64_t *)(slot + r.akeys);
    p.apay = (const uint64_t *)(slot + r.apay);
    p.bkeys = (const uint64_t *)(slot + r.bkeys);
    p.brows = (const uint32_t *)(slot + r.brows);
    p.abnd = (const uint32_t *)(slot + r.abnd);
    p.bbnd = (const uint32_t *)(slot + r.bbnd);
    p.abase = (const uint64_t *)(slot + r.abase);
    p.bbase = p.abase + NA;
    p.na = NA;
    p.nb = NB;
    p.ng = (uint32_t)(r.g1 - r.g0);
    p.step = step;
    p.n_runs = (p.ng + step - 1) / step;
    p.probe_chunk_rows = RB;
    p.acc = acc;
    const size_t e = it % S;
    if (!ev0.empty()) VX_CUDA_TRY(cudaEventRecord(ev0[e], s));
    VX_TRY(rj_join_enqueue(ctx, p, slot + r.items, s));
    if (!ev1.empty()) VX_CUDA_TRY(cudaEventRecord(ev1[e], s));
    return VX_OK;
  }
  void on_retire(uint64_t it) override {
    if (ev0.empty()) return;
    float ms = 0;
    if (cudaEventElapsedTime(&ms, ev0[it % S], ev1[it % S]) == cudaSuccess) ms_join += ms;
    cudaGetLastError();
  }
};

struct HostBuf {
  std::unique_ptr<char[]> mem;
  HostReg reg;
  char *p = nullptr;
  vx_status alloc(uint64_t bytes) {
    mem.reset(new (std::nothrow) char[bytes + 4096]);
    if (!mem) {
      set_error("radix join: no host memory for a %llu-byte intermediate", (unsigned long long)bytes);
      return VX_E_NOMEM;
    }
    p = (char *)(((uintptr_t)mem.get() + 4095) & ~(uintptr_t)4095);
    return reg.add(p, bytes);
  }
};

// smallest partition-pass chunk of the resident mode
constexpr uint64_t kRjMinResidentRows = 1 << 18;

// byte offsets of the resident tables in their arena block
struct RjResident {
  uint32_t NA, NB;
  uint64_t akeys, apay, bkeys, brows, abnd, bbnd, base, items, bytes;
  uint64_t layout(uint64_t nb, uint64_t np, uint64_t R, uint64_t n_runs) {
    auto al = [](uint64_t x) { return (x + 255) & ~255ull; };
    NA = (uint32_t)((nb + R - 1) / R);
    NB = (uint32_t)((np + R - 1) / R);
    akeys = 0;
    apay = akeys + al(8 * nb);
    bkeys = apay + al(8 * nb);
    brows = bkeys + al(8 * np);
    abnd = brows + al(4 * np);
    bbnd = abnd + al(4 * (n_runs + 1) * NA);
    base = bbnd + al(4 * (n_runs + 1) * NB);
    items = base + al(8ull * (NA + NB));
    bytes = items + rj_items_bytes(n_runs, np);
    return bytes;
  }
  static uint64_t slot_bytes(uint64_t R) { return 2 * (8 * R + 255) + 2 * (4 * R + 255) + radix_temp_bytes(R); }
};

// The join with both clustered tables kept in device memory.  Against host
// intermediates this saves their allocation and page-locking in every call,
// the stores and reloads of 12 to 16 bytes a tuple and the boundary arrays
// (64 MiB a chunk at 24 bits): 3M build and 30M probe rows took 41 ms, 22 of
// them for page-locking, and take 2.0.
vx_status radix_join_resident(vx_ctx *ctx, const Column *bk, const Column *bp, const Column *pk, int bits, int run_shift,
                              uint64_t R, const RjResident &rs, RjAcc *acc, vx_join_result &res) {
  const uint64_t nb = bk->n_rows, np = pk->n_rows;
  const uint32_t n_runs = 1u << (bits - run_shift);
  cudaStream_t s = ctx->s_compute;
  DevBuf mem;
  mem.arena = &ctx->arena;
  mem.p = ctx->arena.alloc(rs.bytes);
  if (!mem.p) {
    set_error("vx_join: the clustered tables do not fit the arena");
    return VX_E_NOMEM;
  }
  char *m = mem.as<char>();
  const double tp = now_ms();
  // first tuple of each chunk: build chunks, then probe chunks
  std::vector<uint64_t> base(rs.NA + rs.NB);
  for (uint32_t c = 0; c < rs.NA; ++c) base[c] = (uint64_t)c * R;
  for (uint32_t c = 0; c < rs.NB; ++c) base[rs.NA + c] = (uint64_t)c * R;
  if (!base.empty())
    VX_CUDA_TRY(cudaMemcpyAsync(m + rs.base, base.data(), 8 * base.size(), cudaMemcpyHostToDevice, s));
  for (int side = 0; side < 2; ++side) {
    const uint64_t n = side ? np : nb;
    if (!n) continue;
    RjPartitionPass pp;
    pp.ctx = ctx;
    pp.keys = (const uint64_t *)(side ? pk->host : bk->host);
    pp.payload = side ? nullptr : (const uint64_t *)bp->host;
    pp.n = n;
    pp.R = R;
    pp.bits = bits;
    pp.npass = bits / 8;
    // the join takes whole runs: bytes below a run's first bit need no order
    // (3M x 30M, runs of 4,096 groups: the call 2.27 -> 2.00 ms)
    pp.first = std::min(run_shift / 8, pp.npass - 1);
    pp.S = std::max(2, ctx->cfg.n_slots);
    pp.mid_bnd = nullptr;
    pp.mid_keys = (uint64_t *)(m + (side ? rs.bkeys : rs.akeys));
    pp.mid_pay = (uint64_t *)(m + rs.apay);
    pp.mid_rows = (uint32_t *)(m + rs.brows);
    pp.resident = true;
    pp.acc = acc;
    ExecStats es;
    VX_TRY(run_pipeline(ctx, pp, &es));
    const uint32_t chunks = side ? rs.NB : rs.NA;
    rj_cuts_kernel<<<dim3((unsigned)grid_for(ctx, n_runs + 1, 256, 8), chunks), 256, 0, s>>>(
        pp.mid_keys, n, R, (1ull << bits) - 1, run_shift, n_runs, (uint32_t *)(m + (side ? rs.bbnd : rs.abnd)));
    VX_CUDA_TRY(cudaGetLastError());
    res.bytes_h2d += es.bytes_h2d;
    res.kernel_launches += es.kernel_launches * (radix_launches(pp.npass, pp.first) + 1) + 1;  // keep; cuts
    res.ms_kernel += es.ms_kernel;
  }
  res.ms_partition = res.ms_build = now_ms() - tp;
  const double tj = now_ms();
  if (nb && np) {
    RjJoinParams p{};
    p.akeys = (const uint64_t *)(m + rs.akeys);
    p.apay = (const uint64_t *)(m + rs.apay);
    p.bkeys = (const uint64_t *)(m + rs.bkeys);
    p.brows = (const uint32_t *)(m + rs.brows);
    p.abnd = (const uint32_t *)(m + rs.abnd);
    p.bbnd = (const uint32_t *)(m + rs.bbnd);
    p.abase = (const uint64_t *)(m + rs.base);
    p.bbase = p.abase + rs.NA;
    p.na = rs.NA;
    p.nb = rs.NB;
    p.ng = n_runs;
    p.step = 1;
    p.n_runs = n_runs;
    p.probe_chunk_rows = R;
    p.acc = acc;
    cudaEvent_t e0, e1;
    VX_CUDA_TRY(cudaEventCreate(&e0));
    VX_CUDA_TRY(cudaEventCreate(&e1));
    struct Free {
      cudaEvent_t a, b;
      ~Free() {
        cudaEventDestroy(a);
        cudaEventDestroy(b);
      }
    } fr{e0, e1};
    VX_CUDA_TRY(cudaEventRecord(e0, s));
    VX_TRY(rj_join_enqueue(ctx, p, m + rs.items, s));
    VX_CUDA_TRY(cudaEventRecord(e1, s));
    VX_CUDA_TRY(cudaStreamSynchronize(s));
    float ms = 0;
    VX_CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
    res.kernel_launches += 2;
    res.ms_probe_kernel = ms;
    res.ms_kernel += ms;
    res.ranges = n_runs;
  }
  RjAcc h{};
  VX_CUDA_TRY(cudaMemcpyAsync(&h, acc, sizeof h, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  res.ms_probe = now_ms() - tj;
  if (h.err & ERR_WAIT) {
    set_error("radix join: the clustering sort of a chunk gave up a look-back wait");
    return VX_E_TIMEOUT;
  }
  if (h.err & ERR_DUPKEY) {
    set_error("vx_join: duplicate build key");
    return VX_E_DUPKEY;
  }
  res.count = h.count;
  res.payload_sum = h.psum;
  res.pair_fp = h.fp;
  res.n_partitions = 1u << bits;
  res.max_partition = 0;
  return VX_OK;
}

}  // namespace

vx_status radix_join(vx_ctx *ctx, const Column *bk, const Column *bp, const Column *pk, const vx_join_opts &o,
                     vx_join_result *out) {
  const double t0 = now_ms();
  const int bits = o.radix_bits ? o.radix_bits : 24;
  if (bits != 8 && bits != 16 && bits != 24) {
    set_error("vx_join: radix_bits must be 8, 16 or 24");
    return VX_E_INVAL;
  }
  const int npass = bits / 8;
  const uint64_t G = 1ull << bits, G1 = G + 1;
  const uint64_t nb = bk->n_rows, np = pk->n_rows;
  vx_join_result res{};
  res.algorithm = VX_JOIN_RADIX;
  const int S = std::max(2, ctx->cfg.n_slots);
  cudaStream_t s = ctx->s_compute;
  DevBuf accb;
  accb.arena = &ctx->arena;
  accb.p = ctx->arena.alloc(256);
  if (!accb.p) {
    set_error("vx_join: arena exhausted");
    return VX_E_NOMEM;
  }
  RjAcc *acc = accb.as<RjAcc>();
  VX_CUDA_TRY(cudaMemsetAsync(acc, 0, sizeof(RjAcc), s));

  // ---- partition pass chunk size: R tuples per slot (both tables), and
  // chunk-local rows must fit 32 bits
  const uint64_t avail = ctx->arena.largest_free();
  const uint64_t fixed = 4 * G1 + 4 * ((G1 + kRjSeg - 1) / kRjSeg) + 8192;
  if (avail < S * (fixed + (1 << 20))) {
    set_error("vx_join: budget too small for the radix join's staging slots");
    return VX_E_NOMEM;
  }
  uint64_t R = (uint64_t)((double)(avail / S - fixed) / (40.0 + 256.0 * 8 / kRxTile) * 0.9);
  R = std::min<uint64_t>(R / kRxTile * kRxTile, kPipelineRows);
  if (R < kRxTile) {
    set_error("vx_join: budget too small for the radix join");
    return VX_E_NOMEM;
  }
  const uint32_t NA = (uint32_t)((nb + R - 1) / R), NB = (uint32_t)((np + R - 1) / R);

  // runs of groups that a block joins at once: about kRjRunBuild build tuples
  int run_bits = 0;
  while (run_bits < bits && run_bits < 20 && (nb >> run_bits) > kRjRunBuild) ++run_bits;
  const int run_shift = bits - run_bits;
  uint32_t step = 1u << run_shift;

  // ---- both clustered tables in the arena, if they fit beside the slots of
  // the partition pass (chunks small enough to pipeline)
  uint64_t RR = std::min<uint64_t>(std::max<uint64_t>(std::max(nb, np) / 8, 1 << 20), kPipelineRows);
  RjResident rs;
  for (RR = RR / kRxTile * kRxTile; RR >= kRjMinResidentRows; RR = RR / 2 / kRxTile * kRxTile)
    if (rs.layout(nb, np, RR, 1u << run_bits) + S * (rs.slot_bytes(RR) + 256) + 4096 <= avail) break;
  if (RR >= kRjMinResidentRows) {
    VX_TRY(radix_join_resident(ctx, bk, bp, pk, bits, run_shift, RR, rs, acc, res));
    res.ms_total = now_ms() - t0;
    *out = res;
    return VX_OK;
  }

  // ---- host intermediates
  HostBuf ha_keys, ha_pay, hb_keys, hb_rows, ha_bnd, hb_bnd;
  VX_TRY(ha_keys.alloc(8 * std::max<uint64_t>(nb, 1)));
  VX_TRY(ha_pay.alloc(8 * std::max<uint64_t>(nb, 1)));
  VX_TRY(hb_keys.alloc(8 * std::max<uint64_t>(np, 1)));
  VX_TRY(hb_rows.alloc(4 * std::max<uint64_t>(np, 1)));
  VX_TRY(ha_bnd.alloc(4 * G1 * std::max<uint32_t>(NA, 1)));
  VX_TRY(hb_bnd.alloc(4 * G1 * std::max<uint32_t>(NB, 1)));

  // ---- RadixPartitionExKer over both tables
  const double tp = now_ms();
  for (int side = 0; side < 2; ++side) {
    const uint64_t n = side ? np : nb;
    if (!n) continue;
    RjPartitionPass pp;
    pp.ctx = ctx;
    pp.keys = (const uint64_t *)(side ? pk->host : bk->host);
    pp.payload = side ? nullptr : (const uint64_t *)bp->host;
    pp.n = n;
    pp.R = R;
    pp.bits = bits;
    pp.npass = npass;
    pp.S = S;
    pp.mid_keys = (uint64_t *)(side ? hb_keys.p : ha_keys.p);
    pp.mid_pay = (uint64_t *)ha_pay.p;
    pp.mid_rows = (uint32_t *)hb_rows.p;
    pp.mid_bnd = (uint32_t *)(side ? hb_bnd.p : ha_bnd.p);
    ExecStats es;
    VX_TRY(run_pipeline(ctx, pp, &es));
    res.bytes_h2d += es.bytes_h2d;
    res.bytes_d2h += es.bytes_d2h;
    // rows, the sort, boundaries (4), publish, and the build side's payloads
    res.kernel_launches += es.kernel_launches * (radix_launches(npass) + 6 + (pp.payload ? 1 : 0));
    res.ms_kernel += es.ms_kernel;
  }
  res.ms_partition = now_ms() - tp;
  res.ms_build = res.ms_partition;

  // ---- HashJoinExKer data mapping: group ranges whose tuples and boundary
  // slices fit a slot, by binary search over the boundary arrays
  const double tj = now_ms();
  const uint32_t *abnd = (const uint32_t *)ha_bnd.p, *bbnd = (const uint32_t *)hb_bnd.p;
  auto tuples_below = [&](const uint32_t *bnd, uint32_t N, uint64_t g) {
    uint64_t t = 0;
    for (uint32_t c = 0; c < N; ++c) t += bnd[c * G1 + g];
    return t;
  };
  // Build keys may crowd into a small part of the groups (dense small keys do),
  // and runs of more tuples than a table takes read their probe tuples once per
  // table: shorter runs, as long as they make the run that a build tuple is in
  // smaller.  200M probes of 200,000 dense keys: join kernel 20.7 -> 1.1 ms; of
  // 700,000 13.0 -> 1.2.  Uniform keys keep their runs.
  auto run_size = [&](uint32_t groups) {
    double squares = 0;
    uint64_t below = 0;
    for (uint64_t g = groups; g <= G && nb; g += groups) {
      const uint64_t t = tuples_below(abnd, NA, g);
      squares += (double)(t - below) * (double)(t - below);
      below = t;
    }
    return nb ? squares / (double)nb : 0.0;
  };
  for (double size = run_size(step); step > 1 && size > kRjPiece;) {
    const double half = run_size(step / 2);
    if (half > 0.75 * size) break;  // one group's tuples
    step /= 2;
    size = half;
  }
  const uint64_t slot_b = (uint64_t)((double)ctx->arena.largest_free() / S * 0.95) / 256 * 256;
  auto layout = [&](RjRange &r) {
    const uint64_t ng1 = r.g1 - r.g0 + 1;
    r.na_tuples = tuples_below(abnd, NA, r.g1) - tuples_below(abnd, NA, r.g0);
    r.nb_tuples = tuples_below(bbnd, NB, r.g1) - tuples_below(bbnd, NB, r.g0);
    auto al = [](uint64_t x) { return (x + 255) & ~255ull; };
    r.akeys = 0;
    r.apay = r.akeys + al(8 * r.na_tuples);
    r.bkeys = r.apay + al(8 * r.na_tuples);
    r.brows = r.bkeys + al(8 * r.nb_tuples);
    r.abnd = r.brows + al(4 * r.nb_tuples);
    r.bbnd = r.abnd + al(4 * NA * ng1);
    r.abase = r.bbnd + al(4 * NB * ng1);
    r.bbase = r.abase + 8 * NA;
    r.items = r.abase + al(8 * (NA + NB));
    r.bytes = r.items + rj_items_bytes((r.g1 - r.g0 + step - 1) / step, r.nb_tuples);
  };
  RjJoinPass jp;
  jp.ctx = ctx;
  jp.S = S;
  jp.NA = NA;
  jp.NB = NB;
  jp.G1 = G1;
  jp.RA = R;
  jp.RB = R;
  jp.akeys = (const uint64_t *)ha_keys.p;
  jp.apay = (const uint64_t *)ha_pay.p;
  jp.bkeys = (const uint64_t *)hb_keys.p;
  jp.brows = (const uint32_t *)hb_rows.p;
  jp.abnd_h = abnd;
  jp.bbnd_h = bbnd;
  jp.step = step;
  jp.acc = acc;
  jp.slot_b = slot_b;
  if (nb && np) {
    for (uint64_t g0 = 0; g0 < G;) {
      RjRange r{};
      r.g0 = g0;
      uint64_t lo = g0 + 1, hi = G;  // largest g1 in [g0 + 1, G] whose range fits
      r.g1 = lo;
      layout(r);
      if (r.bytes > slot_b) {
        set_error("vx_join: radix group %llu alone (%llu build, %llu probe tuples) exceeds a staging slot",
                  (unsigned long long)g0, (unsigned long long)r.na_tuples, (unsigned long long)r.nb_tuples);
        return VX_E_NOMEM;
      }
      while (lo < hi) {
        const uint64_t mid = lo + (hi - lo + 1) / 2;
        RjRange t = r;
        t.g1 = mid;
        layout(t);
        if (t.bytes <= slot_b) lo = mid; else hi = mid - 1;
      }
      r.g1 = lo;
      layout(r);
      jp.ranges.push_back(r);
      g0 = r.g1;
    }
  }
  res.ranges = (uint32_t)jp.ranges.size();
  HostBuf hbase;
  if (!jp.ranges.empty()) {
    // per range and chunk: where the chunk's segment starts in the range's slot
    VX_TRY(hbase.alloc(8ull * jp.ranges.size() * (NA + NB)));
    uint64_t *base = (uint64_t *)hbase.p;
    for (size_t q = 0; q < jp.ranges.size(); ++q) {
      const RjRange &r = jp.ranges[q];
      uint64_t *b = base + q * (NA + NB);
      uint64_t at = 0;
      for (uint32_t c = 0; c < NA; ++c) {
        b[c] = at;
        at += abnd[c * G1 + r.g1] - abnd[c * G1 + r.g0];
      }
      at = 0;
      for (uint32_t c = 0; c < NB; ++c) {
        b[NA + c] = at;
        at += bbnd[c * G1 + r.g1] - bbnd[c * G1 + r.g0];
      }
    }
    jp.base_h = base;
    if (ctx->cfg.sched == VX_SCHED_IMMEDIATE) {
      jp.ev0.resize(S);
      jp.ev1.resize(S);
      for (int i = 0; i < S; ++i) {
        VX_CUDA_TRY(cudaEventCreate(&jp.ev0[i]));
        VX_CUDA_TRY(cudaEventCreate(&jp.ev1[i]));
      }
    }
    ExecStats es;
    VX_TRY(run_pipeline(ctx, jp, &es));
    res.bytes_h2d += es.bytes_h2d;
    res.kernel_launches += es.kernel_launches * 2;  // work items and join
    res.ms_kernel += jp.ms_join;
    res.ms_probe_kernel = jp.ms_join;
  }
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  res.ms_probe = now_ms() - tj;
  RjAcc h{};
  VX_CUDA_TRY(cudaMemcpy(&h, acc, sizeof h, cudaMemcpyDeviceToHost));
  if (h.err & ERR_DUPKEY) {
    set_error("vx_join: duplicate build key");
    return VX_E_DUPKEY;
  }
  res.count = h.count;
  res.payload_sum = h.psum;
  res.pair_fp = h.fp;
  res.n_partitions = (uint32_t)G;
  res.max_partition = 0;
  res.ms_total = now_ms() - t0;
  *out = res;
  return VX_OK;
}

}  // namespace vx

using namespace vx;

VX_API vx_status vx_radix_cluster(vx_ctx *ctx, const uint64_t *keys, uint64_t n, int32_t bits, uint64_t *out_keys,
                                  uint32_t *out_rows, uint32_t *out_boundary) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  if ((bits != 8 && bits != 16 && bits != 24) || n >= (1ull << 32) || (n && (!keys || !out_keys || !out_rows)) ||
      !out_boundary) {
    set_error("vx_radix_cluster: bad argument (bits 8, 16 or 24; n < 2^32)");
    return VX_E_INVAL;
  }
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  const uint64_t G1 = (1ull << bits) + 1, m = std::max<uint64_t>(n, 1);
  const uint64_t kb = (8 * m + 255) & ~255ull, vb = (4 * m + 255) & ~255ull, bb = (4 * G1 + 255) & ~255ull;
  const uint64_t cb = (4 * ((G1 + kRjSeg - 1) / kRjSeg) + 255) & ~255ull;
  DevBuf buf;
  buf.arena = &ctx->arena;
  buf.p = ctx->arena.alloc(2 * kb + 2 * vb + radix_temp_bytes(m) + bb + cb);
  if (!buf.p) {
    set_error("vx_radix_cluster: %llu keys do not fit the arena", (unsigned long long)n);
    return VX_E_NOMEM;
  }
  char *p = buf.as<char>();
  RadixBufs b;
  b.keys[0] = (uint64_t *)p;
  b.keys[1] = (uint64_t *)(p + kb);
  b.vals[0] = (uint32_t *)(p + 2 * kb);
  b.vals[1] = (uint32_t *)(p + 2 * kb + vb);
  char *temp = p + 2 * kb + 2 * vb;
  uint32_t *bnd = (uint32_t *)(temp + radix_temp_bytes(m));
  uint32_t *carry = (uint32_t *)((char *)bnd + bb);
  cudaStream_t s = ctx->s_compute;
  const int npass = bits / 8;
  if (n) VX_CUDA_TRY(cudaMemcpyAsync(b.keys[0], keys, 8 * n, cudaMemcpyHostToDevice, s));
  rj_iota_kernel<<<grid_for(ctx, m, 256, 8), 256, 0, s>>>(b.vals[0], n);
  VX_TRY(radix_sort_enqueue(b, n, temp, s, ctx->num_sms, npass, ctx->cfg.lookback_spin_limit));
  const RadixState *st = radix_state_of(temp);
  VX_TRY(find_boundary_enqueue(ctx, b, st, npass, n, bits, bnd, carry, s));
  RadixState h;
  VX_CUDA_TRY(cudaMemcpyAsync(&h, st, offsetof(RadixState, totals), cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  if (h.err) {
    set_error("vx_radix_cluster: a look-back wait gave up");
    return VX_E_TIMEOUT;
  }
  const int c = n ? h.cur[npass] : 0;
  if (n) {
    VX_CUDA_TRY(cudaMemcpyAsync(out_keys, b.keys[c], 8 * n, cudaMemcpyDeviceToHost, s));
    VX_CUDA_TRY(cudaMemcpyAsync(out_rows, b.vals[c], 4 * n, cudaMemcpyDeviceToHost, s));
  }
  VX_CUDA_TRY(cudaMemcpyAsync(out_boundary, bnd, 4 * G1, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  return VX_OK;
}
