// A kernel that holds SMs for a bounded time, for tests of what runs beside it:
// one block per SM with all of the SM's shared memory, so that no block of
// another kernel that needs any finds room there.
#include <cuda_runtime.h>

#include <chrono>
#include <cstdint>

static __device__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__global__ void hold(unsigned long long ns, unsigned int *started) {
  const unsigned long long t0 = now_ns();
  atomicAdd_system(started, 1u);
  for (unsigned long long i = 0; i < ns / 1000 && now_ns() - t0 < ns; ++i) __nanosleep(10000);
}

static cudaStream_t g_stream;
static unsigned int *g_started;

// holds all SMs but `leave` for ms milliseconds; returns the SMs held once all
// of them are (0: an error)
extern "C" int hog_start(int leave, int ms) {
  int dev = 0, sms = 0, smem = 0;
  if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) ||
      cudaDeviceGetAttribute(&smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) ||
      cudaFuncSetAttribute(hold, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) ||
      cudaStreamCreateWithFlags(&g_stream, cudaStreamNonBlocking) ||
      cudaHostAlloc((void **)&g_started, sizeof *g_started, cudaHostAllocMapped))
    return 0;
  *g_started = 0;
  hold<<<sms - leave, 32, smem, g_stream>>>((unsigned long long)ms * 1000000ull, g_started);
  if (cudaGetLastError()) return 0;
  const auto t0 = std::chrono::steady_clock::now();
  while (*(volatile unsigned int *)g_started < (unsigned)(sms - leave))
    if (std::chrono::steady_clock::now() - t0 > std::chrono::milliseconds(ms)) return 0;
  return sms - leave;
}

extern "C" int hog_running() { return cudaStreamQuery(g_stream) == cudaErrorNotReady; }

extern "C" int hog_wait() {
  const cudaError_t e = cudaStreamSynchronize(g_stream);
  cudaStreamDestroy(g_stream);
  cudaFreeHost(g_started);
  return (int)e;
}
