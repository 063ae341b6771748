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

}  // namespace nolo
