// Block-wide prefix sum.
#pragma once

#include <stdint.h>

namespace disco {

// Inclusive prefix sum over the threads of a block (blockDim.x a multiple of 32, at most 1024): shuffles inside
// the warps, one pass over the warp totals, two barriers.  `wtot` is shared scratch of 32 entries; every thread
// of the block must call.  Returns this thread's inclusive sum; *total receives the block's sum.
template <class T>
__device__ __forceinline__ T block_inclusive_scan(T v, T* wtot, T* total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const T up = __shfl_up_sync(0xFFFFFFFFu, v, off);
        if (lane >= off) v += up;
    }
    if (lane == 31) wtot[w] = v;
    __syncthreads();
    if (w == 0) {
        T t = lane < nw ? wtot[lane] : T(0);
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const T up = __shfl_up_sync(0xFFFFFFFFu, t, off);
            if (lane >= off) t += up;
        }
        wtot[lane] = t;                                   // inclusive over the warps
    }
    __syncthreads();
    if (total) *total = wtot[nw - 1];
    return w ? v + wtot[w - 1] : v;
}

}  // namespace disco
