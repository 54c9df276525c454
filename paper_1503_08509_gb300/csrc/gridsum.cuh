// Deterministic sum over a grid of 256-thread blocks, finished by its last block.
#pragma once
#include <cuda_runtime.h>

namespace fep3m {

__device__ __forceinline__ double block_sum256(double a, double* sh /* 8 */) {   // in thread 0
  for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int k = 0; k < 8; ++k) s += sh[k];
  return s;
}

// acc: the thread's value; partial: one double per block; counter: zero before,
// and zero again after.  True in thread 0 of the last block to finish, with
// the total (the partials added in a fixed order).
__device__ __forceinline__ bool grid_sum256(double acc, unsigned nblocks, unsigned bid, double* partial,
                                            unsigned int* counter, double& total) {
  __shared__ double sh[8];
  __shared__ bool last;
  const double s = block_sum256(acc, sh);
  if (threadIdx.x == 0) {
    partial[bid] = s;
    __threadfence();
    last = atomicAdd(counter, 1u) == nblocks - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double a = 0.0;
  for (unsigned k = threadIdx.x; k < nblocks; k += 256) a += ((volatile double*)partial)[k];
  total = block_sum256(a, sh);
  if (threadIdx.x != 0) return false;
  *counter = 0u;
  return true;
}

// The power of two 2^-k with 2^k near the RMS sqrt(sum / n), and its inverse,
// into scale[0], scale[1]: what a residual is scaled by into FP32
__device__ __forceinline__ void rms_scale(double sum, double n, float* scale) {
  const double rms = sqrt(sum / n);
  int k = rms > 0.0 && isfinite(rms) ? ilogb(rms) : 0;
  k = max(-100, min(100, k));
  scale[0] = (float)ldexp(1.0, -k);
  scale[1] = (float)ldexp(1.0, k);
}

}  // namespace fep3m
