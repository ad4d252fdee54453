// ucp_scan.cuh -- block-wide prefix sums shared by the build's kernels.
#pragma once

#include "ucp_internal.cuh"

namespace ucp {

__device__ __forceinline__ int warp_incl_scan(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Exclusive scan of one value per thread over a block.
__device__ __forceinline__ int block_excl_scan(int v, int* total)
{
    __shared__ int warp_sums[32];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int inc = warp_incl_scan(v, lane);
    if (lane == 31) warp_sums[w] = inc;
    __syncthreads();
    if (w == 0) {
        int nw = blockDim.x >> 5;
        int s = lane < nw ? warp_sums[lane] : 0;
        int si = warp_incl_scan(s, lane);
        if (lane < nw) warp_sums[lane] = si - s;
        if (lane == 31) *total = si;
    }
    __syncthreads();
    int r = warp_sums[w] + inc - v;
    __syncthreads();
    return r;
}

}  // namespace ucp
