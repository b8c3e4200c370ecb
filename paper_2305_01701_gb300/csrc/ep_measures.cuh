// ep_measures.cuh -- what the stage kernels of ep_sweep2d.cu and ep_sweep64.cu share: the
// stopping measures, reduced per block, and the end of a solve.
#pragma once

#include <cuda_runtime.h>

#include "ep_internal.cuh"

namespace ep {

__device__ __forceinline__ double maxn(double a, double b) { return (a > b || a != a) ? a : b; }
// |a - b|, formed in FP64
__device__ __forceinline__ double gap(double a, double b) { return fabs(a - b); }

// block-wide max of |v| as IEEE bits (a NaN sorts above infinity), one atomic per
// block; blocks are (32, rows), up to 8 rows
__device__ __forceinline__ void block_max(double v, unsigned long long *slot) {
  __shared__ unsigned long long sm[8];
  unsigned long long b = (unsigned long long)__double_as_longlong(fabs(v));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, b, o);
    b = b > w ? b : w;
  }
  __syncthreads();
  if (threadIdx.x == 0) sm[threadIdx.y] = b;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    for (int q = 1; q < (int)blockDim.y; ++q) b = b > sm[q] ? b : sm[q];
    if (b) atomicMax(slot, b);
  }
}

__device__ __forceinline__ bool skip(const DevInfo *di) { return di != nullptr && *(volatile const int *)&di->done != 0; }

}  // namespace ep
