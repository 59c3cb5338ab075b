// Route progress and block sums shared by the observation kernels of both forms of the state.
#pragma once
#include "gbt_internal.cuh"

namespace gbt {

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int ln = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (ln == 0) sh[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = ln < (int)(blockDim.x >> 5) ? sh[ln] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;
}

__device__ __forceinline__ double prefix_len(const Dev& d, int vid, int upto) {
  const int off = d.roff[vid];
  double p = 0.0;
  for (int k = 0; k < upto; k++) p += (double)d.links[d.routes[off + k]].len;
  return p;
}

}  // namespace gbt
