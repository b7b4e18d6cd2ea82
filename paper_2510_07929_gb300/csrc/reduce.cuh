// Sums over a grid whose last CTA adds the CTAs' partial sums.
#pragma once
#include <cuda_runtime.h>

namespace kqr {

// Block sums of NS values per thread (256 threads) into part[blockIdx.x * NS ..]; returns true in the
// CTA that finishes last, where thread s (s < NS) then holds the total of value s in *total.  That
// CTA's warps add the partials of one value each, lanes striding over the CTAs: 65-cycle FP64
// additions make a serial walk over 300 partials cost 10 us.  Fixed order.  Resets the counter.
template <int NS>
__device__ __forceinline__ bool grid_sums(double (&v)[NS], double* __restrict__ part,
                                          unsigned int* __restrict__ counter, double* total) {
  __shared__ double gs_ws[8][NS];
  __shared__ double gs_tot[NS];
  __shared__ bool gs_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    double x = v[s];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) gs_ws[warp][s] = x;
  }
  __syncthreads();
  if (threadIdx.x < NS) {
    const int s = threadIdx.x;
    part[blockIdx.x * NS + s] = ((gs_ws[0][s] + gs_ws[1][s]) + (gs_ws[2][s] + gs_ws[3][s])) +
                                ((gs_ws[4][s] + gs_ws[5][s]) + (gs_ws[6][s] + gs_ws[7][s]));
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) gs_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!gs_last) return false;
  __threadfence();
  for (int s = warp; s < NS; s += 8) {
    double x = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) x += __ldcg(part + b * NS + s);
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) gs_tot[s] = x;
  }
  __syncthreads();
  if (threadIdx.x < NS) *total = gs_tot[threadIdx.x];
  if (threadIdx.x == 0) *counter = 0u;
  return true;
}

}  // namespace kqr
