// Internal launch interfaces between the C ABI layer and the kernels.
// Nothing here is exported.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nolo {

constexpr int kDomainGroups = 1;  // counter word 3 for subgroup draws
constexpr int kDomainRoute = 2;   // counter word 3 for routing draws

// Draw `blocks` permutations of 0..N-1 into `table`.
// Permutation p (0 <= p < boundaries*slots_drawn) has boundary b = p / slots_drawn and
// slot s = p % slots_drawn, and is written to table[(b*slots_total + k)*N ..] for k = s when
// slots_drawn == slots_total, or for every k in [0, slots_total) when slots_drawn == 1.
cudaError_t launch_draw(uint64_t seed, uint64_t step, int domain, int N, int boundaries,
                        int slots_drawn, int slots_total, int32_t* table, cudaStream_t stream);

// The same for boundaries first_boundary .. first_boundary + boundaries - 1 only (table indexed by the
// absolute boundary).
cudaError_t launch_draw_range(uint64_t seed, uint64_t step, int domain, int N, int first_boundary,
                              int boundaries, int slots_drawn, int slots_total, int32_t* table,
                              cudaStream_t stream);

// Launch of a kernel that calls wait_for_predecessors() (nolo_launch.cuh): its CTAs may be set up
// while the kernel before it in the stream is still running (programmatic dependent launch).
template <typename... Params, typename... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream,
                              Args... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

struct OuterArgs {
    float* phi;          // [W][stride]
    void* theta;         // [W][stride] float or bf16
    float* delta;        // [W][stride]
    int32_t* perm;       // [W]; subgroup g = perm[g*n .. g*n+n-1]
    bool draw = false;   // the kernel draws perm itself from (seed, step) and writes it: see outer_draws
    uint64_t seed = 0, step = 0;
    int64_t stride;      // elements between rows
    int64_t P;           // columns to process, starting at the pointers given
    int W, n;
    int theta_bf16;
    float alpha, beta, gamma;
    // Subgroup means of phi prepared in advance (float64, [W/n][mean_stride], row g for subgroup g of
    // `perm`); NULL = the kernel forms the means itself.
    const double* mean_phi = nullptr;
    int64_t mean_stride = 0;
};

// Whether launch_outer can draw the partition itself (a.draw) at these sizes; otherwise perm has to be
// drawn by launch_draw first.
bool outer_draws(const OuterArgs& a);

// Fused Eq. 1-3 + theta reset over columns [0, P) of the rows (pointers may be pre-offset by
// a multiple of 8 columns).  One launch.
cudaError_t launch_outer(const OuterArgs& a, cudaStream_t stream);

// mean[g][0..P) = float64 mean of phi over subgroup g of `perm` (the part of Eq. 2 that depends on
// the slow weights only).  One launch.
cudaError_t launch_group_mean(const float* phi, const int32_t* perm, int W, int n, int64_t stride, int64_t P,
                              double* mean, int64_t mean_stride, cudaStream_t stream);

struct RouteArgs {
    const void* in;        // [B][R][K][E]
    void* out;             // [B][R][K][E]
    int32_t* table;        // [B][K][R]
    int B, R, K;
    int64_t E;
    int elem_size;         // bytes
    int backward;          // 0: out[b][r][k] = in[b][table[b][k][r]][k]; 1: the inverse
    bool draw = false;     // the kernel draws the table itself and writes it: see route_draws
    uint64_t seed = 0, step = 0;
    int first_boundary = 0, per_microbatch = 0;
    int64_t first_element = 0, elements = 0;   // the part of every block to copy; 0 elements = all of it
};

// Whether launch_route can draw the table itself (a.draw) at these sizes; otherwise it has to be drawn by
// launch_draw first.
bool route_draws(const RouteArgs& a);

cudaError_t launch_route(const RouteArgs& a, cudaStream_t stream);

// Plain copy of `bytes` (a multiple of 16): one-shot grid, 128-bit streaming loads and stores.
cudaError_t launch_copy_probe(const void* in, void* out, int64_t bytes, cudaStream_t stream);

// Replica divergence of phi (Fig. 3b): out2[0] = mean over parameters of the across-worker
// population standard deviation, out2[1] = sqrt(mean over parameters of the across-worker variance).
// `partials` is device scratch of divergence_partials(W, P) * 16 bytes, `arrived` a device counter that is zero
// before and after; out2 is device or mapped host memory.  *launches receives the number of kernels, one or two.
int64_t divergence_partials(int W, int64_t P);
cudaError_t launch_divergence(const float* phi, int W, int64_t stride, int64_t P, void* partials, unsigned* arrived,
                              double* out2, cudaStream_t stream, int* launches);

// Latency simulations (Section 4.3).  per_trial: device [trials] resp. [trials][2];
// stats: device or mapped host memory, the column means followed by their standard errors; copy: of per_trial, in mapped host memory, or NULL.
// scratch: device, tree_scratch() bytes.
size_t tree_scratch();
cudaError_t launch_tree_allreduce(int W, double mu, double sigma, int64_t trials, uint64_t seed,
                                  double* per_trial, double* stats, double* copy, void* scratch, cudaStream_t stream);
// scratch: device, straggler_scratch() bytes (at most about 50 MB).
size_t straggler_scratch(int W, int T, int64_t trials);
cudaError_t launch_straggler(int W, int n, int H, int T, double mu, double sigma, int64_t trials, uint64_t seed,
                             double* per_trial, double* stats, double* copy, void* scratch, cudaStream_t stream);

}  // namespace nolo
