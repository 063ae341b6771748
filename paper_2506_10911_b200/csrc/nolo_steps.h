// Inner steps and their Philox blocks of four, for any count H >= 1 that an int holds: no sum here leaves int, nor
// does a block's number advanced past the last one by a warp's width.
#pragma once

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

}  // namespace nolo
