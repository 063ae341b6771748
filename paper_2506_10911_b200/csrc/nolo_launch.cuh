// Device side of kernels that are launched while their predecessor in the stream still runs.
#pragma once

namespace nolo {

// Returns when everything before this kernel in the stream is complete and visible.  Nothing that an
// earlier kernel writes may be read, and nothing that it reads or writes may be written, before this.
__device__ __forceinline__ void wait_for_predecessors() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Lets the next kernel of the stream be set up once every CTA of this one has got here or has ended.
// The next kernel's own wait is for the whole of this one; every kernel here waits for its predecessors
// before it ends, so that is a wait for all that went before.
__device__ __forceinline__ void let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Asks for memory to be brought to L2: the 128-byte line that holds *p, or a range (16-byte aligned, a multiple of
// 16 bytes) by one instruction of one thread.  It changes nothing that any kernel reads, so it may stand before
// the wait, also for memory that an earlier kernel still writes: what is written meanwhile is written in L2.
__device__ __forceinline__ void prefetch_to_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void prefetch_to_l2(const void* p, int64_t bytes) {
    if (bytes > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"((uint32_t)bytes) : "memory");
}

}  // namespace nolo
