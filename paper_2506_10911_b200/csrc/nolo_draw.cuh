// Ranking of random keys by one CTA, for permutation draws in device code.
#pragma once

#include <stdint.h>

#include "nolo_philox.cuh"

namespace nolo {

// The whole draw of N <= 32 elements by one warp: the rank of this lane's element (N and above for
// lanes without one).  About 0.3 us, most of it the ten dependent rounds of the key: what a kernel with
// few CTAs saves over reading a table is a launch in front of it.
__device__ __forceinline__ int rank_by_warp(int N, uint64_t boundary, uint64_t slot, uint64_t domain, uint64_t seed,
                                            uint64_t step) {
    const int lane = threadIdx.x & 31;
    const uint64_t key = draw_key((uint64_t)lane, boundary, slot, domain, seed, step);
    int rank = 0;
    for (int j = 0; j < N; ++j) {
        const uint64_t kj = __shfl_sync(0xffffffffu, key, j);
        rank += (kj < key) || (kj == key && j < lane);
    }
    return lane < N ? rank : lane;
}

constexpr int kDrawPerThread = 4;   // elements of a draw per thread, at most

// Shared memory of a draw of N elements by a CTA of `threads`: keys, bucket starts, bucket contents.
__host__ __device__ constexpr size_t draw_scratch_bytes(int N, int threads) {
    return (size_t)N * (sizeof(uint64_t) + sizeof(uint16_t)) + ((size_t)threads + 1) * sizeof(uint32_t) + 2;
}

// Position of every element in ascending (key, index) order: rank[m] is that of element
// threadIdx.x + m * THREADS, where there is one.  key(i) gives the 64-bit key of element i.  Called by the
// whole CTA of THREADS (a power of two) threads; N <= kDrawPerThread * THREADS; raw: draw_scratch_bytes
// of 8-byte aligned shared memory.
//
// The keys are uniform 64-bit numbers, so their leading bits spread them evenly over one bucket per
// thread: a counting pass, a scan of the counts and a comparison with the few other elements of the
// same bucket give the rank in O(N) work.  (Any keys give the right ranks; only the time depends on
// their being spread.)  Counting the smaller keys directly is O(N^2); an outer step of N workers that
// is all draw (1000 parameters) measured, counting -> buckets: 11.4 -> 8.4 us at N = 256, 69.8 -> 12.5
// at 1024, 246 -> 18.5 at 2048, 945 -> 29.3 at 4096 (8.3 us, two launches, at N = 64 either way).
template <int THREADS, typename Key>
__device__ __forceinline__ void rank_by_buckets(unsigned char* raw, int N, Key key, int (&rank)[kDrawPerThread]) {
    static_assert(THREADS >= 32 && (THREADS & (THREADS - 1)) == 0, "whole warps, a power of two");
    constexpr int kMost = kDrawPerThread;
    constexpr int kShift = 64 - (THREADS == 32 ? 5 : THREADS == 128 ? 7 : THREADS == 256 ? 8 : THREADS == 512 ? 9 : 10);
    static_assert((1ull << (64 - kShift)) == THREADS, "one bucket per thread");
    __shared__ uint32_t warp_total[THREADS / 32];
    uint64_t* keys = reinterpret_cast<uint64_t*>(raw);            // [N]
    uint32_t* start = reinterpret_cast<uint32_t*>(keys + N);      // [THREADS + 1]
    uint16_t* member = reinterpret_cast<uint16_t*>(start + THREADS + 1);   // [N]
    const int tid = threadIdx.x;
    start[tid] = 0;
    __syncthreads();
    uint64_t k[kMost];
    uint32_t at[kMost];                           // position within the bucket, in order of arrival
#pragma unroll
    for (int m = 0; m < kMost; ++m) {
        const int i = tid + m * THREADS;
        if (i < N) {
            k[m] = key(i);
            keys[i] = k[m];
            at[m] = atomicAdd(&start[k[m] >> kShift], 1u);
        }
    }
    __syncthreads();
    // exclusive scan of the counts, in place
    const uint32_t count = start[tid];
    uint32_t incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
        if ((tid & 31) >= o) incl += up;
    }
    if ((tid & 31) == 31) warp_total[tid >> 5] = incl;
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < (tid >> 5); ++w) before += warp_total[w];
    start[tid] = before + incl - count;
    if (tid == THREADS - 1) start[THREADS] = before + incl;
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kMost; ++m) {
        const int i = tid + m * THREADS;
        if (i < N) member[start[k[m] >> kShift] + at[m]] = (uint16_t)i;
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < kMost; ++m) {
        const int i = tid + m * THREADS;
        if (i < N) {
            const uint32_t lo = start[k[m] >> kShift], hi = start[(k[m] >> kShift) + 1];
            rank[m] = (int)lo;
            for (uint32_t p = lo; p < hi; ++p) {
                const int j = member[p];
                const uint64_t kj = keys[j];
                rank[m] += (kj < k[m]) || (kj == k[m] && j < i);
            }
        }
    }
}

}  // namespace nolo
