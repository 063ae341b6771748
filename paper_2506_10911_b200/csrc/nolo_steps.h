// Inner steps and their Philox blocks of four, for any count H >= 1 that an int holds: no sum here leaves int, nor
// does a block's number advanced past the last one by a warp's width.  And how the threads of the straggler
// simulation are laid over a slab's items.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define NOLO_STEPS_BOTH __host__ __device__ __forceinline__
#else
#define NOLO_STEPS_BOTH inline
#endif

namespace nolo {

NOLO_STEPS_BOTH int step_blocks(int H) { return (H - 1) / 4 + 1; }

// Of block k < step_blocks(H): 4, or what is left in the last one.
NOLO_STEPS_BOTH int steps_in_block(int H, int k) {
    const int left = H - 4 * k;
    return left < 4 ? left : 4;
}

// Units of `threads` items (iteration, worker) of a slab.  Units of one trial each while the items of a trial fill them to
// seven eighths, for their threads share the round keys of Philox; else units over the whole slab, of which
// only the last may be part-filled.
struct WorkUnits {
    bool across;               // over trials
    int64_t items, chunks;     // of a trial, or of the slab where across
    int64_t count;             // of the slab
    static inline WorkUnits of(int W, int iterations, int64_t trials, int threads) {
        WorkUnits u;
        u.items = (int64_t)iterations * W;
        u.chunks = (u.items + threads - 1) / threads;
        u.across = 8 * u.items < 7 * u.chunks * threads;
        u.count = u.chunks * trials;
        if (u.across) {
            u.items *= trials;
            u.count = u.chunks = (u.items + threads - 1) / threads;
        }
        return u;
    }
};

}  // namespace nolo
