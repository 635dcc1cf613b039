// leaf_tasks.cuh -- the leaves of a range of planes, and their tiles, handed to
// warps (decode.cu, diff.cu).
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace aqmp {

// The first leaf with plane >= `plane`; leaves in canonical order (planes
// ascending).  One warp, 32 probes a round.
__device__ __forceinline__ unsigned long long first_of_plane(const LeafRec *leaves, unsigned long long n,
                                                             uint32_t plane) {
    const unsigned lane = threadIdx.x & 31u;
    unsigned long long lo = 0, hi = n;                 // the answer lies in [lo, hi]
    while (lo < hi) {
        const unsigned long long step = (hi - lo + 31) / 32;
        const unsigned long long at = lo + lane * step;
        const bool before = at < hi && leaves[at].plane < plane;     // the answer is past `at`
        const unsigned cnt = (unsigned)__popc(__ballot_sync(0xffffffffu, before));
        if (cnt == 0) {
            hi = lo;
        } else {
            const unsigned long long next = lo + cnt * step;         // first probe not before, or past hi
            lo += (unsigned long long)(cnt - 1) * step + 1;
            if (next < hi) hi = next;
        }
    }
    return lo;
}

// Calls body(leaf record, leaf index, tile) for warp g of W: task f is tile
// f / leaves of leaf f mod leaves, for as many tiles as the largest side has;
// the warp takes tasks g, g + W, ... and looks 32 of them over at a time for
// those that exist (count_of(side) tiles).  Neighbouring tiles of one leaf are
// thus W-scattered, which balances leaves of very different step counts
// without a counter.  Warp-uniform; body must leave the warp converged.
template <class Count, class Body>
__device__ __forceinline__ void for_tiles(const LeafRec *leaves, unsigned long long lo, unsigned count, unsigned tiles,
                                          unsigned g, unsigned W, Count count_of, Body body) {
    const unsigned lane = threadIdx.x & 31u;
    const unsigned long long tasks = (unsigned long long)count * tiles;
    for (unsigned long long f0 = g; f0 < tasks; f0 += 32ull * W) {
        const unsigned long long f = f0 + (unsigned long long)lane * W;
        unsigned leaf = 0, tile = 0;
        bool there = false;
        if (f < tasks) {
            tile = (unsigned)(f / count);
            leaf = (unsigned)(f - (unsigned long long)tile * count);
            there = (int)tile < count_of((int)leaves[lo + leaf].b);
        }
        for (unsigned left = __ballot_sync(0xffffffffu, there); left; left &= left - 1u) {
            const int src = __ffs((int)left) - 1;
            const unsigned long long li = lo + __shfl_sync(0xffffffffu, leaf, src);
            body(leaves[li], li, (int)__shfl_sync(0xffffffffu, tile, src));
        }
    }
}

}  // namespace aqmp
