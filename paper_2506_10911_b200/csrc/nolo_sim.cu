// Monte-Carlo latency simulations of Section 4.3 and the latency-analysis appendix.
//
//  * tree all-reduce vs pair exchange: message times t ~ LogNormal(mu, sigma^2), i.i.d.; a parent of
//    the binary tree is ready when both children's messages have arrived, the result then descends
//    the same tree; the completion time is the last leaf's arrival.  (Constant t_c gives the paper's
//    2 t_c log2 W; W = 2 is the pair exchange max(t1,t2) + max(t3,t4).)
//  * straggler effect: inner-step times LogNormal(mu, sigma^2); DiLoCo waits at a global barrier
//    after every H inner steps, NoLoCo only for the members of its random subgroup of n.
//
// The random times and their stream are those of nolo_lognormal.cuh: four per Philox block, sample j of a
// stream in position j % 4 of block j / 4.  float64 throughout.
#include "nolo.h"
#include "nolo_draw.cuh"
#include "nolo_internal.h"
#include "nolo_launch.cuh"
#include "nolo_lognormal.cuh"
#include "nolo_philox.cuh"
#include "nolo_steps.h"

#include <cmath>

namespace nolo {

namespace {

constexpr int kSimThreads = 256;
constexpr uint64_t kDomainTree = 3;
constexpr uint64_t kDomainStraggler = 4;

// ---- tree all-reduce ---------------------------------------------------------------------------
//
// A group of threads per trial: `group` = W/2 of them (one Philox block of each direction each) up to 256;
// a CTA holds several trials at a time and strides over the trials.  The times of all edges of one
// direction are made first, by all threads at once, into shared memory, indexed like a binary heap (root 1,
// children of p are 2p and 2p+1, leaves W .. 2W-1; block q holds those above the nodes 4q .. 4q+3); then the
// levels are swept, the upper ones (nodes below 128) by one warp, which alone makes and reads those nodes'
// times: between the last wide level up and the first wide level down no barrier is needed, and the other warps
// make the times of the way down meanwhile.  (Subtrees per warp need fewer barriers still, but more
// instructions on part-filled warps, and measured slower.)  What Philox makes of a block's number is the same
// for all trials, what it makes of a trial's for all blocks: both are kept (LEAD).  Bound by the log-normal times
// and the barriers (0.505 -> 0.492 ms without those around the root, W = 1024).  Whole call, (W, trials): one CTA
// per trial that drew the times level by level, two threads for a block -> all times first, a barrier per level ->
// now, ms: (1024, 20 000) 2.0 -> 0.54 -> 0.49, (256, 100 000) 3.3 -> 0.79 -> 0.73, (16, 400 000) 3.8 -> 0.30 -> 0.21
// (0.65 of the first was an allocation).

constexpr int kTreeThreads = 512;
// Trials of a CTA whose part of Philox is made at a time: a multiple of those that it has at once.
__host__ __device__ constexpr int trials_ahead(int per_cta) { return per_cta > 32 ? per_cta : 32; }
constexpr int kLeadMaxW = 1024;      // 32 KB of shared memory; above, one trial per CTA and no LEAD

// Barrier of the threads of one trial.  Trials of more than a warp share the CTA's barrier: all trials of a CTA
// take the same steps.  (Named barriers, one per trial, cost CTAs per SM: all 16 of a CTA are set aside.)
__device__ __forceinline__ void sync_group(int group) {
    if (group <= 32) __syncwarp();
    else __syncthreads();
}

template <bool TAME, bool LEAD>
__global__ void __launch_bounds__(LEAD ? kTreeThreads : 256, LEAD ? 2 : 5)
tree_allreduce_kernel(int W, int group, int64_t trials, LogNormal q, uint64_t seed, double* __restrict__ out) {
    extern __shared__ double2 dynamic[];
    __shared__ LogNormalTables tables;
    __shared__ double part[kTreeThreads / 32];
    const int blocks = W / 2 > 1 ? W / 2 : 1;         // of four times each, the first two of block 0 above no node
    const int per_cta = blockDim.x / group, mine = threadIdx.x / group, lane = threadIdx.x % group;
    const int keep = trials_ahead(per_cta);
    // [direction][block] a, b and c, d; [trial][direction]; then the nodes of each trial of the CTA
    ulonglong2* lead_ab = reinterpret_cast<ulonglong2*>(dynamic);
    ulonglong2* lead_cd = lead_ab + (LEAD ? 2 * blocks : 0);
    PhiloxOfC1* of_trials = reinterpret_cast<PhiloxOfC1*>(lead_cd + (LEAD ? 2 * blocks : 0));
    fill_tables(tables, q);
    if constexpr (LEAD) {
        for (int i = threadIdx.x; i < 2 * blocks; i += blockDim.x) {
            const PhiloxOfC0 l = philox_of_c0(i % blocks, i / blocks, kDomainTree, seed, 0);
            lead_ab[i] = make_ulonglong2(l.a, l.b);
            lead_cd[i] = make_ulonglong2(l.c, l.d);
        }
    }
    __syncthreads();
    double* node = reinterpret_cast<double*>(of_trials + (LEAD ? 2 * keep : 0)) + (size_t)mine * 2 * W;
    const int wide = group > 32 ? 32 : group;         // threads of the warp, or of the part of one, that a trial has
    int turn = 0;                                     // of the CTA; its trials' part of Philox is made `keep` at a time
    for (int64_t first_trial = (int64_t)blockIdx.x * per_cta; first_trial < trials;
         first_trial += (int64_t)gridDim.x * per_cta, ++turn) {
        const int64_t trial = first_trial + mine;
        const int ahead = turn * per_cta & (keep - 1);
        if constexpr (LEAD) {
            if (ahead == 0) {
                __syncthreads();
                for (int i = threadIdx.x; i < 2 * keep; i += blockDim.x) {
                    const int later = i / 2 / per_cta, which = i / 2 % per_cta;
                    of_trials[i] = philox_of_c1(first_trial + (int64_t)later * gridDim.x * per_cta + which, i & 1, seed);
                }
                __syncthreads();
            }
        }
        const bool live = trial < trials;             // the threads of other trials only keep the barriers company
        auto draw = [&](int direction) {
            if (!live) return;
            PhiloxOfC1 of_trial;
            if constexpr (LEAD) of_trial = of_trials[2 * (ahead + mine) + direction];
            for (int b = lane; b < blocks; b += group) {
                Philox4 x;
                if constexpr (LEAD) {
                    const ulonglong2 ab = lead_ab[direction * blocks + b], cd = lead_cd[direction * blocks + b];
                    x = philox_join({ab.x, ab.y, cd.x, cd.y}, of_trial, seed, 0);
                } else {
                    x = philox4x64_10(b, trial, direction, kDomainTree, seed, 0);
                }
                double t[4];
                lognormal4<TAME>(tables, x, q, t);
                double2* to = reinterpret_cast<double2*>(node + 4 * b);
                to[0] = make_double2(t[0], t[1]);
                if (4 * b + 2 < 2 * W) to[1] = make_double2(t[2], t[3]);
            }
        };
        // up: node[c] = time at which c's message has reached its parent.  The parents of one level are first ..
        // 2 * first - 1.
        auto up = [&](int first, int threads) {
            for (int i = lane; i < first; i += threads) {
                const double2 c = reinterpret_cast<const double2*>(node)[first + i];
                node[first + i] += fmax(c.x, c.y);
            }
        };
        draw(0);
        sync_group(group);
        int first = W >> 1;
        for (; first > 32; first >>= 1) {
            up(first, group);
            sync_group(group);
        }
        if (lane < wide) {
            for (; first >= 2; first >>= 1) {
                up(first, wide);
                __syncwarp();
            }
        }
        const double root = lane < wide ? fmax(node[2], node[3]) : 0.0;
        __syncwarp();
        // down: node[c] = time at which the result has reached c.  Children in sibling pairs, those of the
        // parents pairs .. 2 * pairs - 1.
        auto down = [&](int pairs, int threads) {
            for (int i = lane; i < pairs; i += threads) {
                double2* c = reinterpret_cast<double2*>(node) + pairs + i;
                const double parent = node[pairs + i];
                *c = make_double2(parent + c->x, parent + c->y);
            }
        };
        draw(1);
        __syncwarp();
        if (lane < wide) {
            if (lane == 0) {
                node[2] += root;
                node[3] += root;
            }
            __syncwarp();
            for (int pairs = 2; pairs < W && pairs <= 32; pairs <<= 1) {
                down(pairs, wide);
                __syncwarp();
            }
        }
        sync_group(group);
        for (int pairs = 64; pairs < W; pairs <<= 1) {
            down(pairs, group);
            sync_group(group);
        }
        double m = 0.0;
        for (int leaf = W + lane; leaf < 2 * W; leaf += group) m = fmax(m, node[leaf]);
        for (int o = wide / 2; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (group > 32) {
            if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
            sync_group(group);
            if (lane == 0)
                for (int w = 1; w < group / 32; ++w) m = fmax(m, part[(threadIdx.x >> 5) + w]);
        }
        if (live && lane == 0) out[trial] = m;
        sync_group(group);                      // node[] and part[] are used again
    }
}

// ---- straggler simulation --------------------------------------------------------------------------
//
// Only the clocks depend on the iteration before: the work of every worker in every iteration and the
// partitions do not.  So a slab of iterations is done by three kernels: the work sums (all of the random
// times; bound by issue slots, any number of trials fills the chip), the partitions with the longest
// work of each iteration (one CTA or warp each), and the clocks (one CTA per trial, a few exchanges
// through shared memory per iteration).  One CTA per trial for everything used as many SMs as there were
// trials, ranked the keys by O(W^2) comparisons in each iteration, and waited for itself.  Whole call, before ->
// now, (W, n, H, T, trials): (1024, 2, 100, 250, 148) 39.0 -> 16.1 ms, (1024, 512, 100, 500, 8) 91.7 -> 3.1,
// (100, 100, 100, 500, 50) 16.9 -> 1.54, (4, 2, 100, 500, 592) 15.7 -> 0.94, (64, 2, 50, 100, 8) 2.3 -> 0.13.
struct Slab {
    int W, n, H;
    int iterations;            // of this slab, from t0 on
    int64_t t0, trial0, trials;
    uint64_t seed;
    double* work;              // [trials][iterations][W]
    uint16_t* order;           // [trials][iterations][W]: the worker in each position of the partition
    double* longest;           // [trials][iterations]
    double* clock;             // [trials][W], from slab to slab
    double* out;               // [trials][2]: barrier and subgroup time so far
};

// The times of one block.
template <bool TAME>
__device__ __forceinline__ double block_work(const LogNormalTables& tables, const Philox4& x, const LogNormal& q) {
    double step[4];
    lognormal4<TAME>(tables, x, q, step);
    return (step[0] + step[1]) + (step[2] + step[3]);
}
// The first `steps` of them, fewer than four: the end of an item.
template <bool TAME>
__device__ __forceinline__ double part_work(const LogNormalTables& tables, const Philox4& x, const LogNormal& q, int steps) {
    double a, b;
    lognormal2<TAME>(tables, x.w0, x.w1, q, a, b);
    double work = steps > 1 ? a + b : a;
    if (steps > 2) {
        lognormal2<TAME>(tables, x.w2, x.w3, q, a, b);
        work += a;
    }
    return work;
}

// A thread per item (iteration, worker) of a trial, for W >= kSharedRowsW.  A CTA's kSimThreads items lie in few rows
// (iterations), so the part of the Philox rounds that depends on the row and the block only is made once for
// the CTA, kSharedBlocks blocks at a time; they are of one trial, so the round keys are the same for the CTA.
// Bound as nolo_lognormal.cuh says: 323 thread-instructions per four times, 0.60 of the issue slots.  The tables are filled
// once for several units of 256 items.  (1024, 2, 100, 250, 148) 16.1 -> 14.7 ms; 3 CTAs per SM 14.8, 5 14.8, 2 of 512 threads 14.6.
constexpr int kSharedRowsW = 64;
constexpr int kSharedRows = (kSimThreads - 2) / kSharedRowsW + 2;
constexpr int kSharedBlocks = 32;

template <bool TAME>
__global__ void __launch_bounds__(kSimThreads, 4)
straggler_work_kernel(const Slab s, const LogNormal q) {
    __shared__ LogNormalTables tables;
    __shared__ PhiloxOfC0 lead[kSharedRows][kSharedBlocks];
    fill_tables(tables, q);
    const int items = s.iterations * s.W;                            // of a trial
    const int chunks = (items + kSimThreads - 1) / kSimThreads;
    const int blocks = step_blocks(s.H);
    for (int64_t unit = blockIdx.x; unit < s.trials * chunks; unit += gridDim.x) {
        const int64_t trial = unit / chunks;
        const int base = (int)(unit - trial * chunks) * kSimThreads, item = base + threadIdx.x;
        const int row0 = base / s.W, rows = (min(base + kSimThreads, items) - 1) / s.W - row0 + 1;
        const int row = item / s.W, mine = item < items ? row - row0 : 0;
        const PhiloxOfC1 of_worker = philox_of_c1(item - row * s.W, s.t0 + row, s.seed);
        const uint64_t key1 = s.trial0 + trial;
        double work = 0.0;
        for (int b0 = 0; b0 < blocks; b0 += kSharedBlocks) {
            __syncthreads();
            for (int i = threadIdx.x; i < rows * kSharedBlocks; i += kSimThreads)
                lead[i / kSharedBlocks][i % kSharedBlocks] =
                    philox_of_c0(b0 + i % kSharedBlocks, s.t0 + row0 + i / kSharedBlocks, kDomainStraggler, s.seed, key1);
            __syncthreads();
            const int here = blocks - b0 < kSharedBlocks ? blocks - b0 : kSharedBlocks;
            const int last = steps_in_block(s.H, b0 + here - 1), full = last < 4 ? here - 1 : here;
            for (int k = 0; k < full; ++k)                           // inner steps 4 (b0 + k) .. + 3 share a block
                work += block_work<TAME>(tables, philox_join(lead[mine][k], of_worker, s.seed, key1), q);
            if (full < here) work += part_work<TAME>(tables, philox_join(lead[mine][full], of_worker, s.seed, key1), q, last);
        }
        if (item < items) s.work[trial * items + item] = work;
    }
}

// The same for any W: `lanes` (a power of two, at most 32) threads share the blocks of an item, so that few
// items fill the chip too.
template <bool TAME>
__global__ void __launch_bounds__(kSimThreads, 4)
straggler_split_work_kernel(const Slab s, const LogNormal q, int lanes, int64_t items) {
    __shared__ LogNormalTables tables;
    fill_tables(tables, q);
    __syncthreads();
    const int lane = threadIdx.x % lanes;
    const int blocks = step_blocks(s.H);
    for (int64_t first = (int64_t)blockIdx.x * kSimThreads; first < items * lanes; first += (int64_t)gridDim.x * kSimThreads) {
        const int64_t item = (first + threadIdx.x) / lanes;
        double work = 0.0;
        if (item < items) {
            const int64_t row = item / s.W;
            const int w = (int)(item - row * s.W);
            const int64_t trial = row / s.iterations, t = row - trial * s.iterations;
            for (int k = lane; k < blocks; k += lanes) {
                const Philox4 x = philox4x64_10(k, w, s.t0 + t, kDomainStraggler, s.seed, s.trial0 + trial);
                const int steps = steps_in_block(s.H, k);
                work += steps == 4 ? block_work<TAME>(tables, x, q) : part_work<TAME>(tables, x, q, steps);
            }
        }
        for (int o = lanes / 2; o > 0; o >>= 1) work += __shfl_xor_sync(0xffffffffu, work, o);
        if (item < items && lane == 0) s.work[item] = work;
    }
}

// One row (trial, iteration) per CTA of THREADS; with 32 threads and W <= 32, one per warp of a larger CTA.
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
straggler_order_kernel(const Slab s) {
    extern __shared__ uint64_t raw[];
    __shared__ double part[THREADS / 32];
    let_successor_start();          // it waits for this kernel, and this kernel for all before it
    const int64_t row = blockIdx.x;
    const int64_t trial = row / s.iterations, t = row - trial * s.iterations;
    int rank[kDrawPerThread];
    rank_by_buckets<THREADS>(
        reinterpret_cast<unsigned char*>(raw), s.W,
        [&](int i) { return draw_key(i, s.trial0 + trial, 0, kDomainGroups, s.seed, s.t0 + t); }, rank);
    wait_for_predecessors();
    double m = 0.0;
#pragma unroll
    for (int k = 0; k < kDrawPerThread; ++k) {
        const int w = threadIdx.x + k * THREADS;
        if (w < s.W) {
            s.order[row * s.W + rank[k]] = (uint16_t)w;
            m = fmax(m, s.work[row * s.W + w]);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < THREADS / 32; ++w) m = fmax(m, part[w]);
        s.longest[row] = m;
    }
}

__global__ void __launch_bounds__(kSimThreads)
straggler_order_warp_kernel(const Slab s, int64_t rows) {
    const int64_t row = ((int64_t)blockIdx.x * kSimThreads + threadIdx.x) >> 5;
    wait_for_predecessors();
    let_successor_start();
    if (row >= rows) return;
    const int lane = threadIdx.x & 31;
    const int64_t trial = row / s.iterations, t = row - trial * s.iterations;
    const int rank = rank_by_warp(s.W, s.trial0 + trial, 0, kDomainGroups, s.seed, s.t0 + t);
    double m = 0.0;
    if (lane < s.W) {
        s.order[row * s.W + rank] = (uint16_t)lane;
        m = s.work[row * s.W + lane];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) s.longest[row] = m;
}

// The clocks of one trial per CTA.  `lanes` (a power of two, at most 32 and n) threads share a subgroup.  The
// work and the partition of an iteration are read AHEAD iterations ahead: an iteration is two short exchanges
// through shared memory, a read from L2 several times that.
template <int MOST, int AHEAD>
__global__ void __launch_bounds__(1024)
straggler_clock_kernel(const Slab s, int lanes) {
    extern __shared__ uint64_t raw[];
    double* clock = reinterpret_cast<double*>(raw);           // [W] when each worker is done with its work
    uint16_t* order = reinterpret_cast<uint16_t*>(clock + s.W);   // [W]
    const int64_t trial = blockIdx.x;
    const int lane = threadIdx.x % lanes, groups = s.W / s.n;
    let_successor_start();
    for (int w = threadIdx.x; w < s.W; w += blockDim.x) clock[w] = s.t0 ? s.clock[trial * s.W + w] : 0.0;
    double barrier = s.t0 ? s.out[2 * trial] : 0.0;
    double work[AHEAD][MOST], longest[AHEAD];
    uint16_t position[AHEAD][MOST];
    auto read = [&](int slot, int i) {
        if (i >= s.iterations) return;
        const int64_t row = trial * s.iterations + i;
#pragma unroll
        for (int k = 0; k < MOST; ++k) {
            const int w = threadIdx.x + k * blockDim.x;
            if (w < s.W) {
                work[slot][k] = s.work[row * s.W + w];
                position[slot][k] = s.order[row * s.W + w];
            }
        }
        longest[slot] = s.longest[row];
    };
#pragma unroll
    for (int u = 0; u < AHEAD; ++u) read(u, u);
    __syncthreads();
    for (int i0 = 0; i0 < s.iterations; i0 += AHEAD) {
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            if (i0 + u >= s.iterations) break;
#pragma unroll
            for (int k = 0; k < MOST; ++k) {
                const int w = threadIdx.x + k * blockDim.x;
                if (w < s.W) {
                    clock[w] += work[u][k];
                    order[w] = position[u][k];
                }
            }
            barrier += longest[u];
            read(u, i0 + u + AHEAD);
            __syncthreads();
            for (int g0 = 0; g0 < groups; g0 += blockDim.x / lanes) {     // every lane of a subgroup takes the same turns
                const int g = g0 + threadIdx.x / lanes;
                const uint16_t* member = order + (g < groups ? g : 0) * s.n;
                double m = 0.0;
                if (g < groups)
                    for (int j = lane; j < s.n; j += lanes) m = fmax(m, clock[member[j]]);
                for (int o = lanes / 2; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (g < groups)
                    for (int j = lane; j < s.n; j += lanes) clock[member[j]] = m;
            }
            __syncthreads();
        }
    }
    double m = 0.0;
    for (int w = threadIdx.x; w < s.W; w += blockDim.x) {
        m = fmax(m, clock[w]);
        s.clock[trial * s.W + w] = clock[w];
    }
    __shared__ double part[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)blockDim.x / 32; ++w) m = fmax(m, part[w]);
        s.out[2 * trial] = barrier;
        s.out[2 * trial + 1] = m;
    }
}

// ---- means and standard errors ------------------------------------------------------------------------

constexpr int kStatsThreads = 512, kStatsCtas = 64;

__device__ __forceinline__ double cta_sum(double v) {          // in a fixed order, to every thread
    __shared__ double part[kStatsThreads / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();                                            // part[] may still be read from the call before
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = part[0];
#pragma unroll
    for (int w = 1; w < kStatsThreads / 32; ++w) v += part[w];
    return v;
}

// Sum, and sum of squared deviations from the mean, of each column of rows [r0, r1) of x[][COLS], one slice of
// the rows per CTA; the slices are put together by the next kernel.  stats[cta][column] = {sum, deviations}.
template <int COLS>
__global__ void __launch_bounds__(kStatsThreads)
column_moments_kernel(const double* x, int64_t rows, double2* __restrict__ moments) {
    wait_for_predecessors();
    let_successor_start();
    const int64_t r0 = rows * blockIdx.x / gridDim.x, r1 = rows * (blockIdx.x + 1) / gridDim.x;
    double sum[COLS] = {}, dev[COLS] = {};
#pragma unroll 4
    for (int64_t i = r0 + threadIdx.x; i < r1; i += kStatsThreads)
        for (int c = 0; c < COLS; ++c) sum[c] += x[i * COLS + c];
#pragma unroll
    for (int c = 0; c < COLS; ++c) sum[c] = cta_sum(sum[c]);
#pragma unroll 4
    for (int64_t i = r0 + threadIdx.x; i < r1; i += kStatsThreads) {
        for (int c = 0; c < COLS; ++c) {
            const double d = x[i * COLS + c] - sum[c] / (double)(r1 - r0);
            dev[c] += d * d;
        }
    }
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
        dev[c] = cta_sum(dev[c]);
        if (threadIdx.x == 0) moments[blockIdx.x * COLS + c] = make_double2(sum[c], dev[c]);
    }
}

// Column means to out[c]; the standard error of each mean, sqrt(sample variance / rows), to out[COLS + c].
template <int COLS>
__global__ void __launch_bounds__(32)
column_stats_kernel(const double2* moments, int slices, int64_t rows, double* __restrict__ out) {
    wait_for_predecessors();
    let_successor_start();
    const int c = threadIdx.x;
    if (c >= COLS) return;
    double total = 0.0;
    for (int k = 0; k < slices; ++k) total += moments[k * COLS + c].x;
    const double mean = total / (double)rows;
    double dev = 0.0;
    for (int k = 0; k < slices; ++k) {
        const double n = (double)(rows * (k + 1) / slices - rows * k / slices), d = moments[k * COLS + c].x / n - mean;
        dev += moments[k * COLS + c].y + n * d * d;
    }
    out[c] = mean;
    out[COLS + c] = rows > 1 ? sqrt(dev / (double)(rows - 1) / (double)rows) : 0.0;
}

template <int COLS>
cudaError_t launch_stats(const double* x, int64_t rows, double* out, void* scratch, cudaStream_t stream) {
    const int64_t wanted = rows / 4096;
    const int slices = (int)(wanted < 1 ? 1 : wanted > kStatsCtas ? kStatsCtas : wanted);
    double2* moments = static_cast<double2*>(scratch);
    const cudaError_t e = launch_overlapped(column_moments_kernel<COLS>, dim3((unsigned)slices), kStatsThreads, 0, stream, x,
                                            rows, moments);
    if (e != cudaSuccess) return e;
    return launch_overlapped(column_stats_kernel<COLS>, dim3(1), 32, 0, stream, static_cast<const double2*>(moments), slices, rows,
                             out);
}

// Iterations and trials whose work sums are held at a time.
constexpr int64_t kSlabItems = 1 << 21;

int64_t slab_trials(int W, int64_t trials) {
    const int64_t most = kSlabItems / W;
    return trials < most ? trials : most;
}

int64_t slab_iterations(int W, int T, int64_t trials) {
    const int64_t most = kSlabItems / (W * slab_trials(W, trials));
    return T < most ? T : most;
}

}  // namespace

size_t tree_scratch() { return sizeof(double2) * kStatsCtas; }

cudaError_t launch_tree_allreduce(int W, double mu, double sigma, int64_t trials, uint64_t seed,
                                  double* per_trial, double* stats, void* scratch, cudaStream_t stream) {
    const int blocks = W / 2 > 1 ? W / 2 : 1;
    const int group = blocks < 256 ? blocks : 256;
    const bool lead = W <= kLeadMaxW, tame = LogNormal::tame(mu, sigma);
    const int threads = group <= 128 ? 256 : lead ? 512 : 256;
    const int per_cta = threads / group;
    const size_t smem = sizeof(double) * 2 * (size_t)W * per_cta + 
                        (lead ? sizeof(PhiloxOfC0) * 2 * (size_t)blocks + sizeof(PhiloxOfC1) * 2 * trials_ahead(per_cta) : 0);
    auto kernel = tame ? (lead ? tree_allreduce_kernel<true, true> : tree_allreduce_kernel<true, false>)
                       : (lead ? tree_allreduce_kernel<false, true> : tree_allreduce_kernel<false, false>);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int device = 0, sms = 0, resident = 0;
    e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    const int64_t ctas = (trials + per_cta - 1) / per_cta, most = (int64_t)sms * (resident > 0 ? resident : 1);
    kernel<<<(unsigned)(ctas < most ? ctas : most), threads, smem, stream>>>(W, group, trials, LogNormal::make(mu, sigma), seed,
                                                                            per_trial);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_stats<1>(per_trial, trials, stats, scratch, stream);
}

size_t straggler_scratch(int W, int T, int64_t trials) {
    const size_t rows = (size_t)slab_trials(W, trials) * slab_iterations(W, T, trials);
    return rows * W * (sizeof(double) + sizeof(uint16_t)) + rows * sizeof(double) +
           (size_t)slab_trials(W, trials) * W * sizeof(double) + sizeof(double2) * 2 * kStatsCtas;
}

cudaError_t launch_straggler(int W, int n, int H, int T, double mu, double sigma, int64_t trials, uint64_t seed,
                             double* per_trial, double* stats, void* scratch, cudaStream_t stream) {
    const int64_t group = slab_trials(W, trials), iterations = slab_iterations(W, T, trials);
    Slab s;
    s.W = W; s.n = n; s.H = H;
    const LogNormal q = LogNormal::make(mu, sigma);
    s.seed = seed;
    s.work = static_cast<double*>(scratch);
    s.clock = s.work + group * iterations * W;
    s.longest = s.clock + group * W;
    s.order = reinterpret_cast<uint16_t*>(s.longest + group * iterations);
    const bool tame = LogNormal::tame(mu, sigma);
    const int threads = W >= 1024 ? 1024 : (W + 31) / 32 * 32;
    int device = 0, sms = 0, resident = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, tame ? straggler_work_kernel<true> : straggler_work_kernel<false>,
                                                          kSimThreads, 0);
    if (e != cudaSuccess) return e;
    const int64_t work_ctas = (int64_t)sms * (resident > 0 ? resident : 1);
    int lanes = 1;
    while (2 * lanes <= n && lanes < 32) lanes *= 2;
    for (int64_t trial0 = 0; trial0 < trials; trial0 += group) {
        s.trial0 = trial0;
        s.trials = trials - trial0 < group ? trials - trial0 : group;
        s.out = per_trial + 2 * trial0;
        for (int64_t t0 = 0; t0 < T; t0 += iterations) {
            s.t0 = t0;
            s.iterations = (int)(T - t0 < iterations ? T - t0 : iterations);
            const int64_t rows = s.trials * s.iterations, items = rows * W;
            // Threads per item: enough to fill the chip about twice, at most one per block of the item.
            int split = 1;
            while (items * split < (1 << 18) && split < 32 && 4 * split < H) split *= 2;
            const bool shared = split == 1 && W >= kSharedRowsW;
            const int64_t units = shared ? s.trials * (((int64_t)s.iterations * W + kSimThreads - 1) / kSimThreads)
                                         : (items * split + kSimThreads - 1) / kSimThreads;
            const unsigned ctas = (unsigned)(units < 3 * work_ctas ? units : 3 * work_ctas);   // a CTA that falls behind holds up less
            if (shared)
                (tame ? straggler_work_kernel<true> : straggler_work_kernel<false>)<<<ctas, kSimThreads, 0, stream>>>(s, q);
            else
                (tame ? straggler_split_work_kernel<true>
                      : straggler_split_work_kernel<false>)<<<ctas, kSimThreads, 0, stream>>>(s, q, split, items);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            auto order = [&](auto kernel, int order_threads) {
                return launch_overlapped(kernel, dim3((unsigned)rows), order_threads, draw_scratch_bytes(W, order_threads), stream, s);
            };
            e = W <= 32 ? launch_overlapped(straggler_order_warp_kernel, dim3((unsigned)((rows * 32 + kSimThreads - 1) / kSimThreads)),
                                            kSimThreads, 0, stream, s, rows)
              : W <= 512  ? order(straggler_order_kernel<128>, 128)
              : W <= 1024 ? order(straggler_order_kernel<256>, 256)
              : W <= 2048 ? order(straggler_order_kernel<512>, 512)
                          : order(straggler_order_kernel<1024>, 1024);
            if (e != cudaSuccess) return e;
            // Not ahead of the order kernel's end: CTAs that come in as it leaves crowd on the first free SMs, and these
            // run for long (1.03 -> 1.16 ms in all for (4, 2, 100, 500, 592)).
            auto clock = [&](auto kernel) { kernel<<<(unsigned)s.trials, threads, (size_t)W * 10, stream>>>(s, lanes); };
            if (W <= 1024) clock(straggler_clock_kernel<1, 4>);
            else clock(straggler_clock_kernel<NOLO_MAX_WORKERS / 1024, 1>);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    }
    return launch_stats<2>(per_trial, trials, stats, scratch, stream);      // the slabs are done with it
}

}  // namespace nolo
