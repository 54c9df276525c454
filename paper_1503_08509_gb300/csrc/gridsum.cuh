// Deterministic sum over a grid of 256-thread blocks, finished by its last block.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

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
// into the state: what a residual is scaled by into FP32, and the sum of
// squares of a scaled residual of rtol times the first one's norm
__device__ __forceinline__ void refine_begin(double sum, double n, double rtol, RefineState* st) {
  const double rms = sqrt(sum / n);
  int k = rms > 0.0 && isfinite(rms) ? ilogb(rms) : 0;
  k = max(-100, min(100, k));
  st->scale = (float)ldexp(1.0, -k);
  st->inv = (float)ldexp(1.0, k);
  const double f = rtol * ldexp(1.0, -k);
  st->limit = f * f * sum;
}

}  // namespace fep3m
