// Device side of kernels that are launched while their predecessor in the stream still runs.
#pragma once

#include <stdint.h>

namespace nolo {

// Returns when everything before this kernel in the stream is complete and visible.  Nothing that an
// earlier kernel writes may be read, and nothing that it reads or writes may be written, before this.
__device__ __forceinline__ void wait_for_predecessors() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Reads, after the wait, of what an earlier kernel wrote.  Not __ldg (ld.global.nc) and not through const __restrict__
// pointers: both promise that nothing writes the memory as long as the kernel runs, and the kernel is running
// while its predecessor still writes.  volatile keeps them behind the wait.
__device__ __forceinline__ int32_t load_written(const int32_t* p) {
    int32_t v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 load_written(const double2* p) {
    double2 v;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// Lets the next kernel of the stream be set up once every CTA of this one has got here or has ended.
// The next kernel's own wait is for the whole of this one; every kernel here waits for its predecessors
// before it ends, so that is a wait for all that went before.
//
// The next kernel may be a caller's, and what such kernels read ahead of their wait is what the kernel before them is
// not expected to write: weights.  So the kernels that write the state never call this (their successor starts when all
// their CTAs are done, as after any kernel that does not), and the others that can end a call do so behind their own
// wait, if at all.  Only a draw, which the same call follows with a kernel that waits, calls it earlier.
__device__ __forceinline__ void let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Asks for memory to be brought to L2: the 128-byte line that holds *p, or a range (16-byte aligned, a multiple of
// 16 bytes) by one instruction of one thread.  It changes nothing that any kernel reads, so it may stand before
// the wait, also for memory that an earlier kernel still writes: what is written meanwhile is written in L2.
__device__ __forceinline__ void prefetch_to_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void prefetch_to_l2(const void* p, int64_t bytes) {
    if (bytes > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"((uint32_t)bytes) : "memory");
}

}  // namespace nolo
