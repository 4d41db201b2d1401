// su3_reduce.cuh -- per-block reductions of the half-sweep kernels: acceptance
// counts and the partial sums of the fused plaquette.
#pragma once

#include "su3_update.cuh"

namespace su3dev {

// Adds the warp's counts (every lane of the warp calls).
template <bool STATS>
__device__ __forceinline__ void count_stats(UpdateCount c, unsigned long long* stats) {
  if (STATS) {
    const int acc = __reduce_add_sync(0xffffffffu, c.accepted);
    const int prop = __reduce_add_sync(0xffffffffu, c.proposed);
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&stats[0], (unsigned long long)acc);
      atomicAdd(&stats[1], (unsigned long long)prop);
    }
  }
}

// Block sum of one value per thread into out[blockIdx.x] (fixed order).
__device__ __forceinline__ void block_partial(double v, double* out) {
  __shared__ double red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double w = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if (threadIdx.x == 0) out[blockIdx.x] = w;
  }
}

}  // namespace su3dev
