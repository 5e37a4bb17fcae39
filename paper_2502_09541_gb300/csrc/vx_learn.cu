// Learned range partitioner: a monotone CDF MLP (1 -> H -> 1, fp32) trained on
// the device by a kernel that runs all Adam steps of a call (forward, backward
// and update, a grid-wide barrier per step), then inverted by bisection to give
// integer splitters.  The model only decides where partitions are cut; every
// cut gives the same sorted output.
//
//   y(x) = gamma + sum_j softplus(alpha_j) * sigmoid(softplus(omega_j) x + beta_j)
//
// Both weight layers pass through softplus, so y is non-decreasing in x and
// its inverse is well defined for bisection.
#include <algorithm>
#include <cmath>

#include "vx_internal.h"
#include "vx_math.cuh"
#include "vx_sort.cuh"

namespace vx {

__device__ __forceinline__ float softplusf(float v) { return v > 20.f ? v : log1pf(expf(v)); }
__device__ __forceinline__ float sigmoidf(float v) { return 1.f / (1.f + expf(-v)); }

constexpr int kMlpMaxH = 64;
constexpr int kMlpThreads = 256;

// dL/dtheta and L over m points; grad/loss are accumulated with atomics
// (caller zeroes them).  theta = [omega(H), beta(H), alpha(H), gamma].  Lane
// j of a warp owns hidden unit j (H <= 32): a warp evaluates one point at a
// time, every lane its unit, a butterfly sum gives y, and each lane keeps its
// unit's three partial derivatives in registers.
template <int H>
__global__ void __launch_bounds__(kMlpThreads, 2) mlp_fwd_bwd_kernel(const float *__restrict__ theta,
                                                                   const float *__restrict__ x,
                                                                   const float *__restrict__ t, uint64_t m,
                                                                   float *grad, float *loss) {
  static_assert(H >= 1 && H <= 32, "one hidden unit per lane");
  __shared__ float sg[3 * H + 2];
  for (int k = threadIdx.x; k < 3 * H + 2; k += blockDim.x) sg[k] = 0.f;
  __syncthreads();
  const unsigned lane = threadIdx.x & 31;
  const bool on = lane < (unsigned)H;
  const float w = on ? softplusf(theta[lane]) : 0.f, dw = on ? sigmoidf(theta[lane]) : 0.f;
  const float b = on ? theta[H + lane] : 0.f;
  const float a = on ? softplusf(theta[2 * H + lane]) : 0.f, da = on ? sigmoidf(theta[2 * H + lane]) : 0.f;
  const float gamma = theta[3 * H];
  const float inv_m = 1.f / (float)m;
  float g_om = 0.f, g_be = 0.f, g_al = 0.f, g_ga = 0.f, l = 0.f;
  // a warp takes 32 consecutive points at a time: one coalesced load of x and
  // t, then the points one by one, broadcast from the lane that loaded them
  const uint64_t n_warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t base = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < m;
       base += n_warps * 32) {
    const uint64_t mine = base + lane;
    const float xl = mine < m ? x[mine] : 0.f, tl = mine < m ? t[mine] : 0.f;
    const int cnt = m - base < 32 ? (int)(m - base) : 32;
    for (int k = 0; k < cnt; ++k) {
      const float xi = __shfl_sync(0xffffffffu, xl, k), ti = __shfl_sync(0xffffffffu, tl, k);
      const float si = on ? sigmoidf(w * xi + b) : 0.f;
      float v = a * si;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
      const float r = gamma + v - ti;
      const float dy = 2.f * r * inv_m;
      l += r * r;  // the same in every lane; lane 0's copy is kept
      g_ga += dy;
      const float q = dy * a * si * (1.f - si);
      g_be += q;
      g_om += q * xi * dw;
      g_al += dy * da * si;
    }
  }
  if (on) {
    atomicAdd(&sg[lane], g_om);
    atomicAdd(&sg[H + lane], g_be);
    atomicAdd(&sg[2 * H + lane], g_al);
  }
  if (lane == 0) {
    atomicAdd(&sg[3 * H], g_ga);
    atomicAdd(&sg[3 * H + 1], l);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < 3 * H + 1; k += blockDim.x) atomicAdd(&grad[k], sg[k]);
  if (threadIdx.x == 0) atomicAdd(loss, sg[3 * H + 1] * inv_m);
}

// All `steps` full-batch Adam steps (Kingma & Ba 2015) of one training call.
// A step is little work (65,536 points x 32 units: about 1.5 us of the chip's
// issue) behind a serial chain, so the blocks stay resident (cooperative
// launch) and meet at one barrier per step instead of a launch: each warp takes
// 32 points, lane j of it hidden unit j; the 32 outputs are summed over the
// units by a transposing butterfly (31 shuffles, and lane k ends with point
// k's), each lane adds up its unit's three partial derivatives over the points,
// the block its warps', and writes its 97 sums as one row; behind the barrier
// every block adds up all blocks' rows in the same order and applies the same
// update to its own copy of the parameters and moments.  The rows' buffers
// alternate, so a block can run at most one barrier ahead of the slowest reader.
// 300 steps on 65,536 points: 5.2 ms as a launch per step in captured graphs (a
// warp walked its points one by one, 98 global atomics per block, the update in
// the last block); 1.84 ms for the whole call with the sums written parameter by
// parameter and a fence in every thread; 1.70 ms now.  Of a step's 11,200 cycles
// the outputs take about 3,300 (two special-function instructions a point and unit:
// 2,050), the gradient sums 950 and the block's 1,300, the barrier with the read
// of the rows 4,200 and the update 800.  Sums that carry their step's number and are
// polled for, added up parameter by parameter in one block each, took 2.2 ms.
struct TrainArgs {
  float *theta;
  const float *x, *t;
  uint64_t m;
  uint32_t steps;
  float lr, b1, b2, eps;
  float *part;         // 2 x blocks x train_row(H)
  unsigned int *bar;   // [0] arrivals, [1] nonzero: a barrier wait gave up
};

// sigmoid of the training steps: the argument of exp stops at 80 (the result,
// 2e-35, is far below what any sum keeps; a NaN stays one), so that 1 + exp(-v)
// stays in the reciprocal's range
__device__ __forceinline__ float sigmoid_step(float v) { return reciprocal(1.f + expf(v < -80.f ? 80.f : -v)); }

// floats of a block's sums: whole 16-byte words, so that the blocks' rows are
// written and read in few wide accesses
constexpr int train_row(int H) { return (3 * H + 1 + 3) / 4 * 4; }
constexpr int kTrainWarps = 14;  // x 147 blocks: a warp per 32 of the 65,536 points
constexpr uint32_t kTrainPolls = 1u << 22;

template <int H>
__global__ void __launch_bounds__(32 * kTrainWarps, 1) mlp_train_kernel(const TrainArgs p) {
  static_assert(H >= 1 && H <= 32, "one hidden unit per lane");
  constexpr int kParams = 3 * H + 1, kRow = train_row(H), kCols = kRow / 4;
  constexpr int kGroups = 32 * kTrainWarps / kCols < 17 ? 32 * kTrainWarps / kCols : 17;
  __shared__ __align__(16) float s_x[kTrainWarps][32], s_dy[kTrainWarps][32];
  __shared__ float s_part[kTrainWarps][3 * 32 + 1];
  __shared__ __align__(16) float s_sum[kGroups][kRow];
  __shared__ float s_unit[6][32];  // softplus(omega), its derivative, beta, softplus(alpha), its derivative, gamma
  __shared__ int s_stop;
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const bool on = lane < (uint32_t)H;
  const uint32_t k = threadIdx.x, own = k - 32;  // warp 0 waits at the barrier; the next threads own a parameter each
  float theta = 0.f, m1 = 0.f, m2 = 0.f;
  auto unit = [&] {  // what the steps use of it
    if (own < (uint32_t)H || (own >= 2u * H && own < 3u * H)) {
      const uint32_t row = own < (uint32_t)H ? 0 : 3;
      s_unit[row][own % H] = softplusf(theta);
      s_unit[row + 1][own % H] = sigmoidf(theta);
    } else {
      s_unit[own < 3u * H ? 2 : 5][own % H] = theta;
    }
  };
  for (uint32_t i = k; i < 6 * 32; i += 32 * kTrainWarps) (&s_unit[0][0])[i] = 0.f;  // lanes without a unit
  __syncthreads();
  if (own < (uint32_t)kParams) {
    theta = p.theta[own];
    unit();
  }
  const uint64_t n_warps = (uint64_t)gridDim.x * kTrainWarps, first = ((uint64_t)blockIdx.x * kTrainWarps + w) * 32;
  const float x0 = first + lane < p.m ? p.x[first + lane] : 0.f, t0 = first + lane < p.m ? p.t[first + lane] : 0.f;
  const float inv_m = 1.f / (float)p.m;
  for (uint32_t step = 1; step <= p.steps; ++step) {
    __syncthreads();  // the parameters are there
    const float uw = s_unit[0][lane], ub = s_unit[2][lane], ua = s_unit[3][lane], gamma = s_unit[5][0];
    float g_om = 0.f, g_be = 0.f, g_al = 0.f, g_ga = 0.f;
    for (uint64_t base = first; base < p.m; base += n_warps * 32) {
      const bool real = base + lane < p.m;
      const float xl = base == first ? x0 : real ? p.x[base + lane] : 0.f;
      const float tl = base == first ? t0 : real ? p.t[base + lane] : 0.f;
      s_x[w][lane] = xl;
      __syncwarp();
      float sg[32], v[32];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 x4 = reinterpret_cast<const float4 *>(s_x[w])[q];
        const float xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          sg[4 * q + e] = on ? sigmoid_step(uw * xs[e] + ub) : 0.f;
          v[4 * q + e] = ua * sg[4 * q + e];
        }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int j = 0; j < off; ++j) {
          const float keep = up ? v[j + off] : v[j], send = up ? v[j] : v[j + off];
          v[j] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      }
      const float dy = real ? 2.f * (gamma + v[0] - tl) * inv_m : 0.f;  // of the lane's own point
      g_ga += dy;
      s_dy[w][lane] = dy;
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 d4 = reinterpret_cast<const float4 *>(s_dy[w])[q], x4 = reinterpret_cast<const float4 *>(s_x[w])[q];
        const float ds[4] = {d4.x, d4.y, d4.z, d4.w}, xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float si = sg[4 * q + e], u = ds[e] * si;
          const float r = u * ua * (1.f - si);
          g_be += r;
          g_om += r * xs[e];
          g_al += u;
        }
      }
      __syncwarp();  // s_x, s_dy are read no more
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) g_ga += __shfl_xor_sync(0xffffffffu, g_ga, off);
    s_part[w][lane] = g_om * s_unit[1][lane];
    s_part[w][32 + lane] = g_be;
    s_part[w][64 + lane] = g_al * s_unit[4][lane];
    if (lane == 0) s_part[w][96] = g_ga;
    __syncthreads();
    float *part = p.part + (size_t)(step & 1) * kRow * gridDim.x;
    if (k < kRow) {
      const int at = k >= 3 * H ? 96 : (int)(k / H) * 32 + (int)(k % H);
      float sum = 0.f;
      if (k < kParams) {
#pragma unroll
        for (int q = 0; q < kTrainWarps; ++q) sum += s_part[q][at];
      }
      __stcg(&part[(size_t)blockIdx.x * kRow + k], sum);
    }
    __syncthreads();
    if (k == 0) {  // barrier: arrivals only grow, step s ends at s x blocks
      __threadfence();  // the block's sums, which the barrier above has ordered before it
      atomicAdd(&p.bar[0], 1u);
      const uint32_t want = step * gridDim.x;
      int stop = 0;
      for (uint32_t polls = 0; *(volatile unsigned int *)&p.bar[0] < want; ++polls)
        if (polls > kTrainPolls || (polls % 64 == 63 && *(volatile unsigned int *)&p.bar[1])) {
          p.bar[1] = 1;
          stop = 1;
          break;
        }
      __threadfence();
      s_stop = stop;
    }
    float to_m = 0.f, to_v = 0.f;
    if (own < (uint32_t)kParams) {  // while warp 0 waits
      to_m = p.lr / (1.f - powf(p.b1, (float)step));
      to_v = 1.f / (1.f - powf(p.b2, (float)step));
    }
    __syncthreads();
    if (s_stop) return;
    // a thread per four parameters and kGroups-th block: all its loads in flight
    if (k < kCols * kGroups) {
      constexpr int kR = 9;
      const uint32_t g = k / kCols, c = k % kCols;
      float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
      for (uint32_t b0 = g; b0 < gridDim.x; b0 += kGroups * kR) {
        float4 v[kR];
#pragma unroll
        for (int j = 0; j < kR; ++j)
          v[j] = b0 + j * kGroups < gridDim.x
                     ? __ldcg(reinterpret_cast<const float4 *>(part + (size_t)(b0 + j * kGroups) * kRow) + c)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          sum.x += v[j].x;
          sum.y += v[j].y;
          sum.z += v[j].z;
          sum.w += v[j].w;
        }
      }
      reinterpret_cast<float4 *>(s_sum[g])[c] = sum;
    }
    __syncthreads();
    if (own < (uint32_t)kParams) {
      float g = 0.f;
#pragma unroll
      for (int q = 0; q < kGroups; ++q) g += s_sum[q][own];
      m1 = p.b1 * m1 + (1.f - p.b1) * g;
      m2 = p.b2 * m2 + (1.f - p.b2) * g * g;
      theta -= to_m * m1 / (sqrtf(m2 * to_v) + p.eps);
      unit();
    }
  }
  if (blockIdx.x == 0 && own < (uint32_t)kParams) p.theta[own] = theta;
}

// data-driven initial parameters from the (sorted) training points: unit j is
// a sigmoid step of height 1/H centred at the (j + 0.5)/H quantile of x, with a
// slope inverse to the width of its quantile bin, so the untrained network is
// already a smoothed H-segment quantile model that training then refines
__global__ void mlp_init_from_points_kernel(const float *x, uint32_t M, float *theta, int H) {
  for (int j = threadIdx.x; j < H; j += blockDim.x) {
    const uint32_t a = (uint32_t)((uint64_t)j * M / H), b = (uint32_t)((uint64_t)(j + 1) * M / H);
    const uint32_t c = (uint32_t)(((uint64_t)2 * j + 1) * M / (2 * H));
    const float lo = x[a < M ? a : M - 1], hi = x[b < M ? b : M - 1], mid = x[c < M ? c : M - 1];
    const float width = fmaxf(hi - lo, 1e-7f);
    const float slope = fminf(4.f / width, 1e7f);
    theta[j] = slope > 20.f ? slope : logf(expm1f(slope));  // softplus^-1(slope)
    theta[H + j] = -slope * mid;
    theta[2 * H + j] = logf(expm1f(1.f / H));  // softplus^-1(1/H)
  }
  if (threadIdx.x == 0) theta[3 * H] = 0.f;
}

// training points from the sorted sample: M evenly spaced order statistics,
// x = (key - kmin) / (kmax - kmin), target = empirical CDF (idx + 0.5) / m
__global__ void mlp_points_kernel(const uint64_t *sorted, uint64_t m, uint32_t M, float *x, float *t) {
  const uint64_t kmin = sorted[0], kmax = sorted[m - 1];
  const double span = kmax > kmin ? (double)(kmax - kmin) : 1.0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < M; i += gridDim.x * blockDim.x) {
    const uint64_t idx = M > 1 ? (uint64_t)i * (m - 1) / (M - 1) : 0;
    x[i] = (float)((double)(sorted[idx] - kmin) / span);
    t[i] = (float)(((double)idx + 0.5) / (double)m);
  }
}

// splitter p: bisection of y(x) = p/P on [0, 1], mapped back to the key
// domain and snapped to the first sample key >= it (so that a heavy key, a
// vertical step of the CDF, yields repeated splitters that isolate it).  A warp
// per splitter, lane j evaluating unit j (one thread per splitter walked the 40
// x 32 units in series: 229 us for four splitters).
template <int H>
__global__ void __launch_bounds__(256) mlp_splitters_kernel(const float *theta, const uint64_t *sorted, uint64_t m,
                                                            uint32_t P, uint64_t *spl) {
  const uint64_t kmin = sorted[0], kmax = sorted[m - 1];
  const double span = (double)(kmax - kmin);
  const uint32_t lane = threadIdx.x & 31;
  const bool on = lane < (uint32_t)H;
  const float w = on ? softplusf(theta[lane]) : 0.f, b = on ? theta[H + lane] : 0.f;
  const float a = on ? softplusf(theta[2 * H + lane]) : 0.f, gamma = theta[3 * H];
  const uint32_t warps = gridDim.x * blockDim.x / 32;
  for (uint32_t p = 1 + (blockIdx.x * blockDim.x + threadIdx.x) / 32; p < P; p += warps) {
    const float q = (float)p / (float)P;
    float lo = 0.f, hi = 1.f;
    for (int it = 0; it < 40; ++it) {
      const float mid = 0.5f * (lo + hi);
      float y = a * sigmoidf(w * mid + b);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) y += __shfl_xor_sync(0xffffffffu, y, off);
      if (gamma + y < q) lo = mid;
      else hi = mid;
    }
    if (lane) continue;
    double kf = (double)kmin + (double)hi * span;
    uint64_t key = kf >= (double)kmax ? kmax : (kf <= (double)kmin ? kmin : (uint64_t)kf);
    uint64_t a0 = 0, b0 = m;  // first index with sorted[i] >= key
    while (a0 < b0) {
      const uint64_t mid = (a0 + b0) >> 1;
      if (sorted[mid] < key) a0 = mid + 1;
      else b0 = mid;
    }
    spl[p - 1] = sorted[a0 < m ? a0 : m - 1];
  }
}

// ------------------------------------------------------------------ host

struct MlpWork {
  DevBuf buf;
  float *theta, *grad, *loss, *x, *t;
  unsigned int *bar;  // training: barrier arrivals, error
  float *part;        // training: kFewBlocks blocks' partial sums
};

constexpr uint32_t kFewBlocks = 2;

static vx_status mlp_alloc(vx_ctx *ctx, uint64_t M, MlpWork &w) {
  const uint64_t bytes = 4096 + 2 * ((4 * M + 255) & ~255ull) + 1024;
  w.buf.arena = &ctx->arena;
  w.buf.p = ctx->arena.alloc(bytes);
  if (!w.buf.p) {
    set_error("MLP work area of %llu bytes does not fit the arena", (unsigned long long)bytes);
    return VX_E_NOMEM;
  }
  char *p = w.buf.as<char>();
  w.theta = (float *)p;
  w.grad = (float *)(p + 1024);
  w.loss = (float *)(p + 2048);
  w.bar = (unsigned int *)(p + 2048 + 64);
  w.part = (float *)(p + 2048 + 256);
  static_assert(2 * train_row(32) * kFewBlocks * 4 <= 4096 - 2048 - 256, "partial sums of kFewBlocks blocks");
  char *q = p + 4096;
  w.x = (float *)q;
  w.t = (float *)(q + ((4 * M + 255) & ~255ull));
  return VX_OK;
}

// blocks of the forward/backward kernel: 32 points per warp, at most two
// blocks per SM (each block adds 3H + 2 atomics to the global gradient)
static int mlp_grid(const vx_ctx *ctx, uint64_t m) {
  const uint64_t per_block = 32 * (kMlpThreads / 32);
  return (int)std::max<uint64_t>(1, std::min<uint64_t>((m + per_block - 1) / per_block, 2ull * ctx->num_sms));
}

static vx_status launch_fwd_bwd(int H, const float *theta, const float *x, const float *t, uint64_t m, float *grad,
                                float *loss, int grid, cudaStream_t s) {
  if (H == 32)
    mlp_fwd_bwd_kernel<32><<<grid, kMlpThreads, 0, s>>>(theta, x, t, m, grad, loss);
  else if (H == 16)
    mlp_fwd_bwd_kernel<16><<<grid, kMlpThreads, 0, s>>>(theta, x, t, m, grad, loss);
  else if (H == 8)
    mlp_fwd_bwd_kernel<8><<<grid, kMlpThreads, 0, s>>>(theta, x, t, m, grad, loss);
  else if (H == 1)
    mlp_fwd_bwd_kernel<1><<<grid, kMlpThreads, 0, s>>>(theta, x, t, m, grad, loss);
  else {
    set_error("MLP width %d not built (1, 8, 16, 32)", H);
    return VX_E_UNSUPPORTED;
  }
  VX_CUDA_TRY(cudaGetLastError());
  return VX_OK;
}

// Enqueues `steps` Adam steps on w.theta: one cooperative launch, a block per
// 14 x 32 points as far as blocks fit the device at once (and their partial sums
// the arena).  w.bar[1] tells afterwards whether a barrier wait gave up.
static vx_status train(vx_ctx *ctx, int H, MlpWork &w, uint64_t m, uint32_t steps, float lr, DevBuf &part) {
  cudaStream_t s = ctx->s_compute;
  VX_CUDA_TRY(cudaMemsetAsync(w.bar, 0, 8, s));
  if (steps == 0) return VX_OK;
  const void *kernel = H == 32   ? (const void *)mlp_train_kernel<32>
                       : H == 16 ? (const void *)mlp_train_kernel<16>
                       : H == 8  ? (const void *)mlp_train_kernel<8>
                       : H == 1  ? (const void *)mlp_train_kernel<1>
                                 : nullptr;
  if (!kernel) {
    set_error("MLP width %d not built (1, 8, 16, 32)", H);
    return VX_E_UNSUPPORTED;
  }
  int per_sm = 0;
  VX_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32 * kTrainWarps, 0));
  const uint64_t want = (m + 32 * kTrainWarps - 1) / (32 * kTrainWarps);
  uint32_t grid = (uint32_t)std::min<uint64_t>(want, (uint64_t)std::max(per_sm, 1) * ctx->num_sms);
  // arrivals are counted in 32 bits: steps x blocks stays below 2^32
  grid = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(grid, 0xFFFFFFFFull / steps));
  TrainArgs a{w.theta, w.x, w.t, m, steps, lr, 0.9f, 0.999f, 1e-8f, w.part, w.bar};
  if (grid > kFewBlocks) {
    part.arena = &ctx->arena;
    part.p = ctx->arena.alloc(2ull * train_row(H) * grid * 4);
    if (part.p) a.part = part.as<float>();
    else grid = kFewBlocks;
  }
  void *args[] = {&a};
  VX_CUDA_TRY(cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(32 * kTrainWarps), args, 0, s));
  return VX_OK;
}

// after the stream has been waited for
static vx_status train_status(const unsigned int *bar) {
  if (!bar[1]) return VX_OK;
  set_error("MLP training: a barrier wait gave up");
  return VX_E_TIMEOUT;
}

vx_status mlp_splitters(vx_ctx *ctx, const uint64_t *sorted, uint64_t m, uint32_t P, uint32_t steps, uint64_t *d_spl,
                        double *ms_train) {
  const uint32_t M = (uint32_t)std::min<uint64_t>(m, 65536);
  MlpWork w;
  VX_TRY(mlp_alloc(ctx, M, w));
  cudaStream_t s = ctx->s_compute;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0, s);
  mlp_points_kernel<<<(M + 255) / 256, 256, 0, s>>>(sorted, m, M, w.x, w.t);
  mlp_init_from_points_kernel<<<1, 64, 0, s>>>(w.x, M, w.theta, kMlpHidden);
  VX_CUDA_TRY(cudaGetLastError());
  DevBuf part;
  unsigned int bar[2] = {0, 0};
  VX_TRY(train(ctx, kMlpHidden, w, M, steps ? steps : 300, 1e-2f, part));
  mlp_splitters_kernel<kMlpHidden><<<(P + 7) / 8, 256, 0, s>>>(w.theta, sorted, m, P, d_spl);
  VX_CUDA_TRY(cudaGetLastError());
  cudaEventRecord(e1, s);
  VX_CUDA_TRY(cudaMemcpyAsync(bar, w.bar, sizeof bar, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  float ms = 0;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (ms_train) *ms_train = ms;
  return train_status(bar);
}

}  // namespace vx

using namespace vx;

static vx_status mlp_host_setup(vx_ctx *ctx, int32_t H, const float *x, const float *t, uint64_t m, MlpWork &w) {
  if (H < 1 || H > kMlpMaxH || m == 0 || !x || !t) {
    set_error("MLP: need 1 <= H <= %d, m > 0 and points", kMlpMaxH);
    return VX_E_INVAL;
  }
  VX_TRY(mlp_alloc(ctx, m, w));
  cudaStream_t s = ctx->s_compute;
  VX_CUDA_TRY(cudaMemcpyAsync(w.x, x, 4 * m, cudaMemcpyHostToDevice, s));
  VX_CUDA_TRY(cudaMemcpyAsync(w.t, t, 4 * m, cudaMemcpyHostToDevice, s));
  return VX_OK;
}

VX_API vx_status vx_mlp_loss_grad(vx_ctx *ctx, const float *theta, int32_t H, const float *x, const float *t,
                                  uint64_t m, float *grad_out, float *loss_out) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  if (!theta || !grad_out || !loss_out) return VX_E_INVAL;
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  MlpWork w;
  VX_TRY(mlp_host_setup(ctx, H, x, t, m, w));
  cudaStream_t s = ctx->s_compute;
  VX_CUDA_TRY(cudaMemcpyAsync(w.theta, theta, 4 * (3 * H + 1), cudaMemcpyHostToDevice, s));
  VX_CUDA_TRY(cudaMemsetAsync(w.grad, 0, 2048, s));
  const int grid = mlp_grid(ctx, m);
  VX_TRY(launch_fwd_bwd(H, w.theta, w.x, w.t, m, w.grad, w.loss, grid, s));
  VX_CUDA_TRY(cudaMemcpyAsync(grad_out, w.grad, 4 * (3 * H + 1), cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaMemcpyAsync(loss_out, w.loss, 4, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  return VX_OK;
}

VX_API vx_status vx_mlp_train(vx_ctx *ctx, float *theta, int32_t H, const float *x, const float *t, uint64_t m,
                              uint32_t steps, float lr, float *loss_out) {
  clear_error();
  VX_TRY(check_ctx(ctx));
  if (!theta || !loss_out || !(lr > 0.f)) return VX_E_INVAL;
  std::lock_guard<std::recursive_mutex> g(ctx->mu);
  MlpWork w;
  VX_TRY(mlp_host_setup(ctx, H, x, t, m, w));
  cudaStream_t s = ctx->s_compute;
  VX_CUDA_TRY(cudaMemcpyAsync(w.theta, theta, 4 * (3 * H + 1), cudaMemcpyHostToDevice, s));
  DevBuf part;
  unsigned int bar[2] = {0, 0};
  VX_TRY(train(ctx, H, w, m, steps, lr, part));
  VX_CUDA_TRY(cudaMemcpyAsync(bar, w.bar, sizeof bar, cudaMemcpyDeviceToHost, s));
  // loss of the final parameters
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  VX_TRY(train_status(bar));
  VX_CUDA_TRY(cudaMemsetAsync(w.grad, 0, 2048, s));
  const int grid = mlp_grid(ctx, m);
  VX_TRY(launch_fwd_bwd(H, w.theta, w.x, w.t, m, w.grad, w.loss, grid, s));
  VX_CUDA_TRY(cudaMemcpyAsync(theta, w.theta, 4 * (3 * H + 1), cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaMemcpyAsync(loss_out, w.loss, 4, cudaMemcpyDeviceToHost, s));
  VX_CUDA_TRY(cudaStreamSynchronize(s));
  return VX_OK;
}
