// Random permutations for subgroup draws (Section 3.2) and pipeline routes (Section 3.1).
//
// The paper only asks for random subgroups / random permutations from a seed.  Here element i
// of a draw gets a 64-bit key from the Philox-4x64-10 counter-based generator (Salmon, Moraes,
// Dror, Shaw: "Parallel random numbers: as easy as 1, 2, 3", SC'11) with
// counter = (i, boundary, slot, domain) and key = (seed, step); the permutation lists the
// indices in ascending (key, index) order.  Integer arithmetic only, so the tables are
// reproducible bit for bit on any machine.
#include "nolo_draw.cuh"
#include "nolo_internal.h"
#include "nolo_launch.cuh"
#include "nolo_philox.cuh"

namespace nolo {

namespace {

// One CTA per permutation, one thread per element up to N = 1024 and four above.  Bound by latency:
// the ten dependent rounds of a key (about 0.4 us), then five barriers.  All of that needs nothing from
// earlier kernels and is done while they still run; only the table is written after them.
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
draw_perm_kernel(uint64_t seed, uint64_t step, uint64_t domain, int N, int first_boundary, int slots_drawn,
                 int slots_total, int32_t* __restrict__ table) {
    extern __shared__ uint64_t raw[];
    const int b = first_boundary + blockIdx.x / slots_drawn;
    const int s = blockIdx.x % slots_drawn;
    const int k_lo = (slots_drawn == slots_total) ? s : 0;
    const int k_hi = (slots_drawn == slots_total) ? s + 1 : slots_total;
    let_successor_start();          // it waits for this kernel, and this kernel for all before it
    int rank[kDrawPerThread];
    rank_by_buckets<THREADS>(
        reinterpret_cast<unsigned char*>(raw), N,
        [&](int i) { return draw_key((uint64_t)i, (uint64_t)b, (uint64_t)s, domain, seed, step); }, rank);
    wait_for_predecessors();
#pragma unroll
    for (int m = 0; m < kDrawPerThread; ++m) {
        const int i = threadIdx.x + m * THREADS;
        if (i < N)
            for (int k = k_lo; k < k_hi; ++k) table[((int64_t)b * slots_total + k) * N + rank[m]] = i;
    }
}

}  // namespace

cudaError_t launch_draw_range(uint64_t seed, uint64_t step, int domain, int N, int first_boundary,
                              int boundaries, int slots_drawn, int slots_total, int32_t* table,
                              cudaStream_t stream) {
    const int blocks = boundaries * slots_drawn;
    if (blocks <= 0 || N <= 0) return cudaSuccess;
    auto launch = [&](auto kernel, int threads) {
        return launch_overlapped(kernel, dim3((unsigned)blocks), threads, draw_scratch_bytes(N, threads), stream, seed, step,
                                 (uint64_t)domain, N, first_boundary, slots_drawn, slots_total, table);
    };
    if (N <= 32) return launch(draw_perm_kernel<32>, 32);
    if (N <= 128) return launch(draw_perm_kernel<128>, 128);
    if (N <= 512) return launch(draw_perm_kernel<512>, 512);
    return launch(draw_perm_kernel<1024>, 1024);
}

cudaError_t launch_draw(uint64_t seed, uint64_t step, int domain, int N, int boundaries,
                        int slots_drawn, int slots_total, int32_t* table, cudaStream_t stream) {
    return launch_draw_range(seed, step, domain, N, 0, boundaries, slots_drawn, slots_total, table, stream);
}

}  // namespace nolo
