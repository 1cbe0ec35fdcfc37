// Prefix sums within a warp and within a block.
#pragma once

#include "common.cuh"

namespace e2egrec {

template <typename AccT>
__device__ inline AccT warp_inclusive_scan(AccT v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        AccT t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// Exclusive scan across the block of one value per thread; returns the exclusive prefix,
// `total` receives the block sum.  smem must hold THREADS/32 values.
template <int THREADS, typename AccT>
__device__ inline AccT block_exclusive_scan(AccT v, AccT &total, AccT *smem)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    AccT inc = warp_inclusive_scan(v);
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        AccT w = lane < THREADS / 32 ? smem[lane] : AccT(0);
        AccT wi = warp_inclusive_scan(w);
        if (lane < THREADS / 32) smem[lane] = wi - w;
        if (lane == THREADS / 32 - 1) smem[THREADS / 32] = wi;
    }
    __syncthreads();
    AccT res = smem[warp] + inc - v;
    total = smem[THREADS / 32];
    __syncthreads();
    return res;
}

}  // namespace e2egrec
