// reciprocal() (csrc/vx_math.cuh) against CUDA's division for every float from 1 to
// 6e34: how many results differ, and by how many units in the last place at most.
#include <cuda_runtime.h>

#include "vx_math.cuh"

__global__ void compare(unsigned first, unsigned last, unsigned long long *differ, unsigned *most) {
  unsigned long long n = 0;
  unsigned worst = 0;
  for (unsigned long long i = first + (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i <= last;
       i += (unsigned long long)gridDim.x * blockDim.x) {
    const float d = __uint_as_float((unsigned)i);
    const unsigned a = __float_as_uint(vx::reciprocal(d)), b = __float_as_uint(1.f / d);
    const unsigned off = a > b ? a - b : b - a;
    n += off != 0;
    worst = off > worst ? off : worst;
  }
  atomicAdd(differ, n);
  atomicMax(most, worst);
}

__global__ void of_nan(unsigned *out) { *out = isnan(vx::reciprocal(__uint_as_float(0x7FC00000u))); }

// values compared, results that differ, the largest difference, whether a NaN stays one; 0: done
extern "C" int reciprocal_check(unsigned long long *values, unsigned long long *differ, unsigned *most, unsigned *nan) {
  unsigned long long *d_n = nullptr;
  if (cudaMalloc((void **)&d_n, 32) || cudaMemset(d_n, 0, 32)) return 1;
  unsigned first, last;
  const float lo = 1.f, hi = 6e34f;
  __builtin_memcpy(&first, &lo, 4);
  __builtin_memcpy(&last, &hi, 4);
  compare<<<1216, 256>>>(first, last, d_n, (unsigned *)(d_n + 1));
  of_nan<<<1, 1>>>((unsigned *)(d_n + 2));
  unsigned long long h[3];
  if (cudaGetLastError() || cudaMemcpy(h, d_n, sizeof h, cudaMemcpyDeviceToHost)) return 1;
  cudaFree(d_n);
  *values = (unsigned long long)last - first + 1;
  *differ = h[0];
  *most = (unsigned)h[1];
  *nan = (unsigned)h[2];
  return 0;
}
