// Appending to a device list whose length lives in one counter, from every
// thread of a block at once (stream compaction without a separate scan).
#pragma once

#include <cstdint>

namespace cc {

// The slot of this thread's item among the block's items, reserved with ONE
// atomicAdd per block on `count` (rather than one per warp): a list that
// grows by a million items per launch through a single counter otherwise
// queues tens of thousands of atomics on that one word. The warps' counts are
// scanned by the first warp, which takes the block's range.
// Every thread of the block must call it (it contains barriers); threads with
// has == false get a slot they must not use. A warp reads and writes only its
// own count, the next call's write coming after that call's warp-wide ballot
// (which all lanes reach only after their reads), and the scan and the base
// are rewritten only after the next call's first barrier, so consecutive
// calls need no barrier between them.
__device__ __forceinline__ unsigned block_slot(bool has, unsigned* __restrict__ count) {
    __shared__ unsigned warp_base[32];
    __shared__ unsigned block_base;
    const unsigned mask = __ballot_sync(0xffffffffu, has);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) warp_base[w] = __popc(mask);
    __syncthreads();
    if (w == 0) {  // exclusive scan of the warps' counts; one lane takes the block's range
        const int warps = (blockDim.x + 31) >> 5;
        const unsigned own = lane < warps ? warp_base[lane] : 0u;
        unsigned incl = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += y;
        }
        if (lane < warps) warp_base[lane] = incl - own;
        if (lane == 31) block_base = incl ? atomicAdd(count, incl) : 0u;
    }
    __syncthreads();
    return block_base + warp_base[w] + __popc(mask & ((1u << lane) - 1));
}

__device__ __forceinline__ void append1_block(bool has, int v, int* __restrict__ out,
                                              unsigned* __restrict__ count) {
    const unsigned slot = block_slot(has, count);
    if (has) out[slot] = v;
}

__device__ __forceinline__ void append2_block(bool has, int a, int b, int* __restrict__ out,
                                              unsigned* __restrict__ count) {
    const unsigned slot = block_slot(has, count);
    if (has) {
        out[2 * (size_t)slot] = a;
        out[2 * (size_t)slot + 1] = b;
    }
}

}  // namespace cc
