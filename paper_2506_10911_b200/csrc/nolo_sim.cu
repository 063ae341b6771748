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
// The edges of one direction are indexed like a binary heap (root 1, children of p are 2p and 2p + 1, leaves W .. 2W - 1);
// Philox block q holds the times above the nodes 4q .. 4q + 3.  Either direction is the same recursion from the leaves
// to the root: a node is ready when the later of its children's messages is there, and the last leaf has the result at
// the time of the longest way down, which is found from below like the longest way up.  So a trial is two sums of
// longest ways, and no time is kept for a second sweep.
//
// `lanes` lanes (a power of two, at most kTreeMostLanes and W / 2) take one direction of one trial.  Every lane has a subtree of W / lanes
// leaves, whose blocks it visits children first, with the finished halves of what is above them on a stack
// of its own; then every lane makes one of the `lanes` blocks of the nodes below 4 lanes, which they reduce by shuffles.
// So all lanes work all the time and nothing waits for another warp, but for the two directions of a trial
// of 32 lanes, which meet every kTreeRounds trials.  Where few trials leave most of the chip idle, several warps share a direction and
// meet in shared memory for the nodes below 2 lanes / 32 (WIDE): (2048, 148) 66 -> 28 us, (4096, 148) 108 -> 34 (46 and
// 50 with 256 threads that swept the nodes).  What Philox makes of a block's number is the same for all trials and is kept (LEAD).
// Bound by the log-normal times: 363 thread-instructions per four (those of the stragglers 317); a sweep up and one down
// over nodes in shared memory with barriers between the levels took 464.  Whole call, (W, trials): (1024, 20 000) 0.51 -> 0.37 ms,
// (256, 100 000) 0.77 -> 0.50, (64, 300 000) 0.70 -> 0.48 (0.3 of it the copy of the trials).
constexpr int kTreeThreads = 512, kTreeWarps = kTreeThreads / 32, kTreeRounds = 32;
constexpr int kTreeMostLanes = kTreeThreads / 2;      // both directions of a trial in a CTA
constexpr int kLeadMaxW = 1024;      // 32 KB of shared memory
constexpr int kTreeMostDepth = 10;    // log2(NOLO_MAX_WORKERS / 4)
static_assert(4 << kTreeMostDepth == NOLO_MAX_WORKERS, "a lane's subtree has at most NOLO_MAX_WORKERS / 4 leaf blocks");

__device__ __forceinline__ double later(double a, double b) { return a > b ? a : b; }      // no NaN here

template <bool TAME, bool LEAD, bool WIDE>
__global__ void __launch_bounds__(kTreeThreads, 2)
tree_allreduce_kernel(int W, int lanes, int64_t trials, LogNormal q, uint64_t seed, double* __restrict__ out, unsigned* arrived) {
    extern __shared__ double2 dynamic[];
    __shared__ LogNormalTables tables;
    __shared__ double ways[kTreeRounds][kTreeWarps];
    const int blocks = W / 2, leaves = W / (4 * lanes);       // leaf blocks of a lane
    // [direction][block] a, b and c, d, a level's blocks in the order in which the lanes take them; then [depth][thread]
    ulonglong2* lead_ab = reinterpret_cast<ulonglong2*>(dynamic);
    ulonglong2* lead_cd = lead_ab + (LEAD ? 2 * blocks : 0);
    double2* stack = reinterpret_cast<double2*>(lead_cd + (LEAD ? 2 * blocks : 0)) + threadIdx.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) *arrived = 0;
    fill_tables(tables, q);
    if constexpr (LEAD) {
        for (int i = threadIdx.x; i < 2 * blocks; i += kTreeThreads) {
            const int direction = i / blocks, slot = i % blocks;
            const int first = slot < lanes ? 0 : 1 << (31 - __clz(slot)), each = first / lanes;
            const int block = first == 0 ? slot : first + slot % lanes * each + (slot - first) / lanes;
            const PhiloxOfC0 l = philox_of_c0(block, direction, kDomainTree, seed, 0);
            lead_ab[i] = make_ulonglong2(l.a, l.b);
            lead_cd[i] = make_ulonglong2(l.c, l.d);
        }
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mine = threadIdx.x % lanes;
    // A warp's tasks of a round: one, or both directions of 16 / lanes trials next to each other.  WIDE: the CTA's, both directions of
    // its trials next to each other.
    const int64_t per_warp = WIDE ? 1 : 32 / lanes, per_cta = kTreeThreads / lanes;
    const int64_t rounds = (2 * trials + per_cta * gridDim.x - 1) / (per_cta * gridDim.x);
    for (int64_t round = 0; round < rounds; ++round) {
        int direction;
        int64_t trial;
        if (WIDE) {
            const int64_t task = (round * gridDim.x + blockIdx.x) * per_cta + threadIdx.x / lanes;
            direction = (int)(task & 1);
            trial = task >> 1;
        } else if (lanes == 32) {
            direction = warp & 1;
            trial = (round * (kTreeWarps / 2) + (warp >> 1)) * gridDim.x + blockIdx.x;
        } else {
            const int64_t task = ((round * kTreeWarps + warp) * gridDim.x + blockIdx.x) * per_warp + lane / lanes;
            direction = (int)(task & 1);
            trial = task >> 1;
        }
        double way = 0.0;
        if (WIDE || lanes < 32 || trial < trials) {
            const PhiloxOfC1 of_trial = philox_of_c1(trial, direction, seed);
            auto words = [&](int block, int slot) {
                if constexpr (LEAD) {
                    const ulonglong2 ab = lead_ab[direction * blocks + slot], cd = lead_cd[direction * blocks + slot];
                    return philox_join({ab.x, ab.y, cd.x, cd.y}, of_trial, seed, 0);
                } else {
                    return philox4x64_10(block, trial, direction, kDomainTree, seed, 0);
                }
            };
            // when the two parents of the block last made are ready, seen from the leaves
            double x0 = 0.0, x1 = 0.0;
            int first = W / 4, turn = 0, done = 0, depth = 0;      // the level's first block, the lane's turn in it
            double t[4];
            for (int left = 2 * leaves - 1; left > 0; --left) {
                const int each = first / lanes;
                lognormal4<TAME>(tables, words(first + mine * each + turn, first + turn * lanes + mine), q, t);
                if (first == W / 4) {
                    x0 = later(t[0], t[1]);
                    x1 = later(t[2], t[3]);
                } else {
                    const double2 y = stack[--depth * kTreeThreads];
                    const double x = later(x0 + t[2], x1 + t[3]);
                    x0 = later(y.x + t[0], y.y + t[1]);
                    x1 = x;
                }
                if (turn & 1) {                                    // both halves of the block above are there
                    turn >>= 1;
                    first >>= 1;
                } else if (left > 1) {
                    stack[depth++ * kTreeThreads] = make_double2(x0, x1);
                    first = W / 4;
                    turn = ++done;
                }
            }
            // the nodes below 4 * lanes
            const Philox4 x = words(mine, mine);
            if (W > 2) lognormal2<TAME>(tables, x.w0, x.w1, q, t[0], t[1]);
            lognormal2<TAME>(tables, x.w2, x.w3, q, t[2], t[3]);
            __syncwarp();
            double2* own = stack - mine;                           // of the lanes, [2][lanes]: the times above nodes 2i and 2i + 1
            auto pair = [&](int i) -> double2& { return own[(i & 1) * kTreeThreads + (i >> 1)]; };
            pair(2 * mine) = make_double2(t[0], t[1]);
            pair(2 * mine + 1) = make_double2(t[2], t[3]);
            if constexpr (WIDE) __syncthreads();
            else __syncwarp();
            auto above = [&](int node) { return reinterpret_cast<const double*>(&pair(node >> 1))[node & 1]; };
            const double2 leaf = pair(lanes + mine);
            way = later(x0 + leaf.x, x1 + leaf.y);
            for (int o = 1; o < (WIDE ? 32 : lanes); o <<= 1) {
                way += above((lanes + mine) / o);
                way = later(way, __shfl_xor_sync(0xffffffffu, way, o));
            }
            __syncwarp();
            if constexpr (WIDE) {                                  // the nodes that a warp each has come to
                const int warps = lanes / 32;
                if (lane == 0) ways[0][warp] = way;
                __syncthreads();
                if (mine < 32) {
                    const int i = lane % warps;
                    way = ways[0][warp + i];
                    for (int o = 1; o < warps; o <<= 1) {
                        way += above((warps + i) / o);
                        way = later(way, __shfl_xor_sync(0xffffffffu, way, o));
                    }
                    if (lane == 0) ways[1][threadIdx.x / lanes] = way;
                }
                __syncthreads();
            }
        }
        if (WIDE) {
            if (mine == 0 && direction == 0 && trial < trials) out[trial] = ways[1][threadIdx.x / lanes] + ways[1][threadIdx.x / lanes + 1];
        } else if (lanes < 32) {
            way += __shfl_xor_sync(0xffffffffu, way, lanes);
            if (lane % (2 * lanes) == 0 && trial < trials) out[trial] = way;
        } else {
            if (lane == 0) ways[round % kTreeRounds][warp] = way;
            if (round % kTreeRounds == kTreeRounds - 1 || round == rounds - 1) {
                __syncthreads();
                for (int i = threadIdx.x; i < kTreeRounds * kTreeWarps / 2; i += kTreeThreads) {
                    const int64_t r = round - round % kTreeRounds + i / (kTreeWarps / 2);
                    const int p = i % (kTreeWarps / 2);
                    const int64_t at = (r * (kTreeWarps / 2) + p) * gridDim.x + blockIdx.x;
                    if (r <= round && at < trials) out[at] = ways[r % kTreeRounds][2 * p] + ways[r % kTreeRounds][2 * p + 1];
                }
                __syncthreads();
            }
        }
    }
}

// ---- straggler simulation --------------------------------------------------------------------------
//
// Only the clocks depend on the iteration before: the work of every worker in every iteration and the
// partitions do not.  So a slab of iterations is done by three kernels: the work sums (all of the random
// times; any number of trials fills the chip), the partitions with the longest
// work of each iteration (a CTA, a warp or a part of one each), and the clocks (one CTA per trial, one exchange
// through shared memory per iteration for pairs and for the members of small subgroups, two for other subgroups).
// Whole call, one CTA per trial for everything -> three kernels -> now, (W, n, H, T, trials): (1024, 2, 100, 250, 148) 39.0 -> 16.1 -> 14.5 ms, (1024, 512, 100, 500, 8) 91.7 ->
// 2.9 -> 2.3, (100, 100, 100, 500, 50) 16.9 -> 1.55 -> 0.97, (4, 2, 100, 500, 592) 15.7 -> 0.95 -> 0.57,
// (64, 2, 50, 100, 8) 2.3 -> 0.11 -> 0.065.
struct Slab {
    int W, n, H;
    int iterations;            // of this slab, from t0 on
    int64_t t0, trial0, trials;
    uint64_t seed;
    double* work;              // [trials][iterations][W]
    uint32_t* rank;            // [trials][iterations][W]: each worker's position in the partition
    double* longest;           // [trials][iterations]
    double* clock;             // [trials][W], from slab to slab
    double* out;               // [trials][2]: barrier and subgroup time so far
    unsigned* arrived;         // counter of the statistics
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

// A thread per item (iteration, worker), for W >= kSharedRowsW.  A CTA's kSimThreads items lie in few rows
// (iterations), so the part of the Philox rounds that depends on the row and the block only is made once for
// the CTA, up to kSharedBlocks blocks at a time.  They are of one trial, so that the round keys are the same for the CTA, unless
// that would leave threads idle: many trials leave a slab few iterations, and a trial of it fewer items than threads (ACROSS).
// Bound as nolo_lognormal.cuh says: 317 thread-instructions per four times, 0.60 of the issue slots.  The tables are filled
// once for several units of 256 items.  (1024, 2, 100, 250, 148) 16.1 -> 14.5 ms; with 3 CTAs
// per SM 1 % more, with 5 the same, with 2 of 512 threads 0.3 % less.
// Few workers (from kSharedRowsW on) lie in many rows, a few blocks of which are made at a time: (4, 2, 100, 500, 592)
// 611 -> 570 us, (16, 2, 50, 250, 500) 540 -> 493 against whole Philox blocks in the kernel below.
constexpr int kSharedRowsW = 4;
constexpr int kSharedBlocks = 32, kSharedLead = 400;
static_assert(kSharedLead >= 4 * ((kSimThreads - 2) / kSharedRowsW + 2), "at least four blocks of every row");

template <bool TAME, bool ACROSS>
__global__ void __launch_bounds__(kSimThreads, 4)
straggler_work_kernel(const Slab s, const LogNormal q, int items, int chunks, int64_t units) {
    __shared__ LogNormalTables tables;
    if (blockIdx.x == 0 && threadIdx.x == 0) *s.arrived = 0;
    __shared__ PhiloxOfC0 lead[kSharedLead];                         // [row][at_once]
    const int at_once = min(kSharedBlocks, kSharedLead / ((kSimThreads - 2) / s.W + 2));
    fill_tables(tables, q);
    const int blocks = step_blocks(s.H);
    for (int64_t unit = blockIdx.x; unit < units; unit += gridDim.x) {
        const int64_t unit_trial = ACROSS ? 0 : unit / chunks;
        const int base = (int)(unit - unit_trial * chunks) * kSimThreads, item = base + threadIdx.x;
        const int row0 = base / s.W, rows = (min(base + kSimThreads, items) - 1) / s.W - row0 + 1;
        const int row = item / s.W, mine = item < items ? row - row0 : 0;
        // of a row, counted from the unit's trial on
        auto trial_of = [&](int r) { return ACROSS ? r / s.iterations : 0; };
        auto iteration_of = [&](int r) { return s.t0 + (ACROSS ? r % s.iterations : r); };
        const PhiloxOfC1 of_worker = philox_of_c1(item - row * s.W, iteration_of(row), s.seed);
        const uint64_t key1 = s.trial0 + unit_trial + trial_of(row);
        double work = 0.0;
        for (int b0 = 0; b0 < blocks; b0 += at_once) {
            __syncthreads();
            const int here = blocks - b0 < at_once ? blocks - b0 : at_once;
            for (int i = threadIdx.x; i < rows * here; i += kSimThreads) {
                const int r = i / here, k = i - r * here;
                lead[r * at_once + k] = philox_of_c0(b0 + k, iteration_of(row0 + r), kDomainStraggler, s.seed,
                                                     s.trial0 + unit_trial + trial_of(row0 + r));
            }
            __syncthreads();
            const int last = steps_in_block(s.H, b0 + here - 1), full = last < 4 ? here - 1 : here;
            for (int k = 0; k < full; ++k)                           // inner steps 4 (b0 + k) .. + 3 share a block
                work += block_work<TAME>(tables, philox_join(lead[mine * at_once + k], of_worker, s.seed, key1), q);
            if (full < here) work += part_work<TAME>(tables, philox_join(lead[mine * at_once + full], of_worker, s.seed, key1), q, last);
        }
        if (item < items) s.work[unit_trial * items + item] = work;
    }
}

// The same for any W: `lanes` (a power of two, at most 32) threads share the blocks of an item, so that few
// items fill the chip too.
template <bool TAME>
__global__ void __launch_bounds__(kSimThreads, 4)
straggler_split_work_kernel(const Slab s, const LogNormal q, int lanes, int64_t items) {
    __shared__ LogNormalTables tables;
    if (blockIdx.x == 0 && threadIdx.x == 0) *s.arrived = 0;
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

// One row (trial, iteration) per CTA of THREADS; up to 32 workers, 32 / width rows per warp.
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
            s.rank[row * s.W + w] = (uint32_t)rank[k];
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
straggler_order_warp_kernel(const Slab s, int64_t rows, int width) {
    const int lane = threadIdx.x & (width - 1);
    const int64_t row = ((int64_t)blockIdx.x * kSimThreads + threadIdx.x) / width;
    const int64_t trial = row / s.iterations, t = row - trial * s.iterations;
    const uint64_t key = draw_key(lane, s.trial0 + trial, 0, kDomainGroups, s.seed, s.t0 + t);
    int rank = 0;
    for (int j = 0; j < s.W; ++j) {
        const uint64_t other = __shfl_sync(0xffffffffu, key, j, width);
        rank += other < key || (other == key && j < lane);
    }
    wait_for_predecessors();
    let_successor_start();
    const bool mine = row < rows && lane < s.W;
    double m = mine ? s.work[row * s.W + lane] : 0.0;
    if (mine) s.rank[row * s.W + lane] = (uint32_t)rank;
    for (int o = width / 2; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (row < rows && lane == 0) s.longest[row] = m;
}

// The sum of the longest work of a trial's iterations, in their order, added to `sum`; by one warp.
__device__ __forceinline__ double barrier_time(const Slab& s, int64_t trial, double sum) {
    const int lane = threadIdx.x & 31;
    for (int i0 = 0; i0 < s.iterations; i0 += 32) {
        const double longest = i0 + lane < s.iterations ? s.longest[trial * s.iterations + i0 + lane] : 0.0;
#pragma unroll
        for (int k = 0; k < 32; ++k) sum += __shfl_sync(0xffffffffu, longest, k);
    }
    return sum;
}

// The clocks of one trial per CTA, each in a register of its worker's thread; the members of a subgroup meet in
// shared memory, in the order of the partition.  Bound by the latency of that exchange, iteration after iteration, so
// the work and the ranks are copied to shared memory AHEAD iterations ahead, each by the thread that will use it (loads into
// registers are waited for by six counters, whoever shares one waits for the latest: no more than four iterations ahead).
// LOOK > 0: subgroups of at most that many, each of whose members looks at all the others: one barrier per iteration, two buffers.
// Else `lanes` (a power of two, at most 32) threads share a subgroup, with shuffles and two barriers: from 512 workers on the
// faster for more than pairs, since members who look at all take n accesses each.  Whole call, us, shared / looked at: (16, 8, 10, 500,
// 100) 299 / 233, (100, 5, 10, 250, 50) 241 / 204, (256, 8, 10, 250, 50) 377 / 360, (1024, 4, 10, 100, 20) 275 / 294.  Pairs of 16
// workers, a kernel of 500 iterations: 246 -> 60 us.
constexpr int kLookMost = 8, kLookMaxW = 256;

template <int BYTES>
__device__ __forceinline__ void copy_ahead(void* to, const void* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from), "n"(BYTES)
                 : "memory");
}

__host__ __device__ constexpr size_t clock_bytes(int W, int groups, int ahead, bool look) {
    return (size_t)W * ahead * (sizeof(double) + sizeof(uint32_t)) + (look ? 2 * (W + groups) : W + groups) * sizeof(double);
}

template <int MOST, int AHEAD, int LOOK>
__global__ void __launch_bounds__(1024)
straggler_clock_kernel(const Slab s, int lanes, unsigned inverse_n) {
    extern __shared__ double shared[];
    const int64_t trial = blockIdx.x;
    const int lane = threadIdx.x % lanes, turn = threadIdx.x / lanes, per_turn = blockDim.x / lanes, groups = s.W / s.n;
    // [W], or twice [groups][pitch]: an odd pitch spreads the subgroups over the banks
    const int pitch = LOOK > 2 ? s.n | 1 : s.n, half = LOOK > 2 ? s.W + groups : s.W;
    double* buffer = shared;
    double* longest_of = shared + s.W;                        // [groups], unless LOOK
    double* works = shared + (LOOK ? 2 * half : s.W + groups);            // [AHEAD][W]
    uint32_t* ranks = reinterpret_cast<uint32_t*>(works + AHEAD * s.W);      // [AHEAD][W]
    const double* next_work = s.work + trial * s.iterations * s.W + threadIdx.x;
    const uint32_t* next_rank = s.rank + trial * s.iterations * s.W + threadIdx.x;
    double clock[MOST];
    bool mine[MOST];
#pragma unroll
    for (int k = 0; k < MOST; ++k) {
        const int w = threadIdx.x + k * blockDim.x;
        mine[k] = w < s.W;
        clock[k] = s.t0 && mine[k] ? s.clock[trial * s.W + w] : 0.0;
    }
    auto ahead = [&](int slot, int i) {
        if (i < s.iterations) {
#pragma unroll
            for (int k = 0; k < MOST; ++k) {
                const int w = threadIdx.x + k * blockDim.x;
                if (mine[k]) {
                    copy_ahead<8>(works + slot * s.W + w, next_work + k * blockDim.x);
                    copy_ahead<4>(ranks + slot * s.W + w, next_rank + k * blockDim.x);
                }
            }
            next_work += s.W;
            next_rank += s.W;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int u = 0; u < AHEAD; ++u) ahead(u, u);
    int slot = 0;
    for (int i = 0; i < s.iterations; ++i) {
        asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
        int at[MOST];
#pragma unroll
        for (int k = 0; k < MOST; ++k) {
            if (mine[k]) {
                const int w = threadIdx.x + k * blockDim.x;
                at[k] = (int)ranks[slot * s.W + w];
                clock[k] += works[slot * s.W + w];
                const int group = LOOK != 2 && inverse_n ? (int)__umulhi((unsigned)at[k], inverse_n) : at[k];
                buffer[LOOK > 2 ? at[k] + group * (pitch - s.n) : at[k]] = clock[k];
                if (LOOK != 2) at[k] = group;
            }
        }
        ahead(slot, i + AHEAD);
        slot = slot + 1 == AHEAD ? 0 : slot + 1;
        __syncthreads();
        if constexpr (LOOK > 0) {
#pragma unroll
            for (int k = 0; k < MOST; ++k) {
                if (mine[k]) {
                    if constexpr (LOOK == 2) {
                        clock[k] = later(clock[k], buffer[at[k] ^ 1]);
                    } else {
                        const double* member = buffer + at[k] * pitch;
                        double c[LOOK];
#pragma unroll
                        for (int j = 0; j < LOOK; ++j) c[j] = j < s.n ? member[j] : 0.0;
#pragma unroll
                        for (int j = 0; j < LOOK; ++j) clock[k] = later(clock[k], c[j]);
                    }
                }
            }
            buffer = buffer == shared ? shared + half : shared;
        } else {
            for (int g0 = 0; g0 < groups; g0 += per_turn) {               // every lane of a subgroup takes the same turns
                const int g = g0 + turn;
                double m = 0.0;
                if (g < groups)
                    for (int j = lane; j < s.n; j += lanes) m = later(m, buffer[g * s.n + j]);
                for (int o = lanes / 2; o > 0; o >>= 1) m = later(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (g < groups && lane == 0) longest_of[g] = m;
            }
            __syncthreads();
#pragma unroll
            for (int k = 0; k < MOST; ++k)
                if (mine[k]) clock[k] = longest_of[at[k]];
        }
    }
    double m = 0.0;
#pragma unroll
    for (int k = 0; k < MOST; ++k) {
        const int w = threadIdx.x + k * blockDim.x;
        if (w < s.W) {
            m = fmax(m, clock[k]);
            s.clock[trial * s.W + w] = clock[k];
        }
    }
    __shared__ double part[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        const double barrier = barrier_time(s, trial, s.t0 ? s.out[2 * trial] : 0.0);
        if (threadIdx.x == 0) {
            for (int w = 1; w < (int)blockDim.x / 32; ++w) m = fmax(m, part[w]);
            s.out[2 * trial] = barrier;
            s.out[2 * trial + 1] = m;
        }
    }
}

// One subgroup of all workers waits for the longest work of every iteration, as the barrier does: no partition and
// no clocks, and the two times are the same.  The longest work of a row per warp, then the sum over the
// iterations, in their order, per warp.  (512, 512, 50, 500, 83) 5.6 -> 4.2 ms, (100, 100, 100, 500, 50) 1.46 -> 0.97.
__global__ void __launch_bounds__(kSimThreads)
straggler_longest_kernel(const Slab s, int64_t rows) {
    wait_for_predecessors();
    let_successor_start();
    const int64_t row = ((int64_t)blockIdx.x * kSimThreads + threadIdx.x) >> 5;
    if (row >= rows) return;
    double m = 0.0;
    for (int w = threadIdx.x & 31; w < s.W; w += 32) m = fmax(m, s.work[row * s.W + w]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) s.longest[row] = m;
}

__global__ void __launch_bounds__(kSimThreads)
straggler_barrier_kernel(const Slab s) {
    wait_for_predecessors();
    let_successor_start();
    const int64_t trial = ((int64_t)blockIdx.x * kSimThreads + threadIdx.x) >> 5;
    if (trial >= s.trials) return;
    const double barrier = barrier_time(s, trial, s.t0 ? s.out[2 * trial] : 0.0);
    if ((threadIdx.x & 31) < 2) s.out[2 * trial + (threadIdx.x & 31)] = barrier;
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

// Means of the columns of x[rows][COLS] to out[c], the standard error of each, sqrt(sample variance / rows), to
// out[COLS + c]; x itself to `copy`, unless that is NULL.  out and copy may be page-locked host memory.  One slice of the rows
// per CTA gives its sum and the squared deviations from its mean, which the last CTA to be done puts together in
// a fixed order.  `arrived` counts them, from zero.  One kernel whose results are there when it ends, instead of two kernels
// and two copies through the driver's buffer: tree of (64, 2000) 46 -> 27 us a call, (2, 45 226) 71 -> 43.
template <int COLS>
__global__ void __launch_bounds__(kStatsThreads)
trial_stats_kernel(const double* x, int64_t rows, double2* moments, unsigned* arrived, double* out, double* copy) {
    static_assert(COLS == 1 || COLS == 2, "a row is one access");
    wait_for_predecessors();
    let_successor_start();
    const int64_t r0 = rows * blockIdx.x / gridDim.x, r1 = rows * (blockIdx.x + 1) / gridDim.x;
    double sum[COLS] = {}, dev[COLS] = {};
#pragma unroll 8
    for (int64_t i = r0 + threadIdx.x; i < r1; i += kStatsThreads) {
        if constexpr (COLS == 1) {
            const double v = x[i];
            if (copy) copy[i] = v;
            sum[0] += v;
        } else {
            const double2 v = reinterpret_cast<const double2*>(x)[i];
            if (copy) reinterpret_cast<double2*>(copy)[i] = v;
            sum[0] += v.x;
            sum[1] += v.y;
        }
    }
#pragma unroll
    for (int c = 0; c < COLS; ++c) sum[c] = cta_sum(sum[c]);
#pragma unroll 8
    for (int64_t i = r0 + threadIdx.x; i < r1; i += kStatsThreads) {
#pragma unroll
        for (int c = 0; c < COLS; ++c) {
            const double d = x[i * COLS + c] - sum[c] / (double)(r1 - r0);
            dev[c] += d * d;
        }
    }
    __shared__ bool last;
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
        dev[c] = cta_sum(dev[c]);
        if (gridDim.x == 1) {
            if (threadIdx.x == 0) {
                out[c] = sum[c] / (double)rows;
                out[COLS + c] = rows > 1 ? sqrt(dev[c] / (double)(rows - 1) / (double)rows) : 0.0;
            }
            continue;
        }
        if (threadIdx.x == 0) moments[blockIdx.x * COLS + c] = make_double2(sum[c], dev[c]);
    }
    if (gridDim.x == 1) return;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(arrived, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int k = threadIdx.x, slices = gridDim.x;
    const double n = (double)(rows * (k + 1) / slices - rows * k / slices);
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
        const double2 m = k < slices ? __ldcg(moments + k * COLS + c) : make_double2(0.0, 0.0);
        const double mean = cta_sum(m.x) / (double)rows;
        const double d = k < slices ? m.x / n - mean : 0.0;
        const double total = cta_sum(k < slices ? m.y + n * d * d : 0.0);
        if (threadIdx.x == 0) {
            out[c] = mean;
            out[COLS + c] = rows > 1 ? sqrt(total / (double)(rows - 1) / (double)rows) : 0.0;
        }
    }
}

constexpr size_t kStatsScratch = sizeof(double2) * (2 * kStatsCtas + 1);      // moments, then the counter

unsigned* stats_counter(void* scratch) { return reinterpret_cast<unsigned*>(static_cast<double2*>(scratch) + 2 * kStatsCtas); }

template <int COLS>
cudaError_t launch_stats(const double* x, int64_t rows, double* out, double* copy, void* scratch, cudaStream_t stream) {
    const int64_t wanted = rows / 4096;
    const int slices = (int)(wanted < 1 ? 1 : wanted > kStatsCtas ? kStatsCtas : wanted);
    return launch_overlapped(trial_stats_kernel<COLS>, dim3((unsigned)slices), kStatsThreads, 0, stream, x, rows,
                             static_cast<double2*>(scratch), stats_counter(scratch), out, copy);
}

// Iterations and trials whose work sums are held at a time: as many as keep a call's scratch with its results below the 64 MB that are kept
// between calls (67.0e6 bytes at one worker, 2 iterations, 1 046 528 trials).
constexpr int64_t kSlabItems = (1 << 21) - (1 << 12);

// As few slabs as that allows, of equal sizes.
int64_t even_share(int64_t all, int64_t most) {
    const int64_t parts = (all + most - 1) / most;
    return (all + parts - 1) / parts;
}

int64_t slab_trials(int W, int64_t trials) { return even_share(trials, kSlabItems / W); }

int64_t slab_iterations(int W, int T, int64_t trials) {
    return even_share(T, kSlabItems / (W * slab_trials(W, trials)));
}

}  // namespace

size_t tree_scratch() { return kStatsScratch; }

cudaError_t launch_tree_allreduce(int W, double mu, double sigma, int64_t trials, uint64_t seed,
                                  double* per_trial, double* stats, double* copy, void* scratch, cudaStream_t stream) {
    const bool lead = W <= kLeadMaxW, tame = LogNormal::tame(mu, sigma);
    // Lanes per direction of a trial.  What several do together costs about 0.14 of a block for each of their log2(lanes)
    // exchanges, few lanes per trial leave the last turn of the chip's warps emptier.
    int device = 0, sms = 0, resident = 0, lanes = 1;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    double least = 0.0;
    for (int l = 1, log2 = 0; l <= W / 2 && l <= kTreeMostLanes; l *= 2, ++log2) {
        const int64_t threads = (int64_t)sms * 2 * kTreeThreads;
        const double cost = (double)((2 * trials * l + threads - 1) / threads) * (W / (2 * l) + 0.14 * log2);
        if (l == 1 || cost <= least) {
            least = cost;
            lanes = l;
        }
    }
    int depth = 2;                       // of a lane's stack, as much as it needs for the last exchange
    for (int leaves = W / (4 * lanes); leaves > 4; leaves /= 2) ++depth;
    const size_t smem = sizeof(double2) * depth * kTreeThreads + (lead ? sizeof(PhiloxOfC0) * W : 0);
    auto kernel = lanes > 32 ? (tame ? (lead ? tree_allreduce_kernel<true, true, true> : tree_allreduce_kernel<true, false, true>)
                                     : (lead ? tree_allreduce_kernel<false, true, true> : tree_allreduce_kernel<false, false, true>))
                             : (tame ? (lead ? tree_allreduce_kernel<true, true, false> : tree_allreduce_kernel<true, false, false>)
                                     : (lead ? tree_allreduce_kernel<false, true, false> : tree_allreduce_kernel<false, false, false>));
    // the most that any call needs (lanes = 1), so that calls of different sizes from several threads do not undo each other's
    const int most_smem = (int)sizeof(double2) * kTreeMostDepth * kTreeThreads + (lead ? (int)sizeof(PhiloxOfC0) * kLeadMaxW : 0);
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most_smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kernel, kTreeThreads, smem);
    if (e != cudaSuccess) return e;
    // whole CTAs of busy warps, for each fills its tables: (16, 1855) 26.2 us with as many CTAs as run at a time, 23.4 so
    const int64_t ctas = (2 * trials * lanes + kTreeThreads - 1) / kTreeThreads;
    const int64_t most = (int64_t)sms * (resident > 0 ? resident : 1);
    kernel<<<(unsigned)(ctas < most ? ctas : most), kTreeThreads, smem, stream>>>(W, lanes, trials, LogNormal::make(mu, sigma), seed,
                                                                                 per_trial, stats_counter(scratch));
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_stats<1>(per_trial, trials, stats, copy, scratch, stream);
}

size_t straggler_scratch(int W, int T, int64_t trials) {
    const size_t rows = (size_t)slab_trials(W, trials) * slab_iterations(W, T, trials);
    return rows * W * (sizeof(double) + sizeof(uint32_t)) + rows * sizeof(double) +
           (size_t)slab_trials(W, trials) * W * sizeof(double) + kStatsScratch;
}

cudaError_t launch_straggler(int W, int n, int H, int T, double mu, double sigma, int64_t trials, uint64_t seed,
                             double* per_trial, double* stats, double* copy, void* scratch, cudaStream_t stream) {
    const int64_t group = slab_trials(W, trials), iterations = slab_iterations(W, T, trials);
    Slab s;
    s.W = W; s.n = n; s.H = H;
    const LogNormal q = LogNormal::make(mu, sigma);
    s.seed = seed;
    s.arrived = stats_counter(scratch);
    s.work = static_cast<double*>(scratch) + kStatsScratch / sizeof(double);
    s.clock = s.work + group * iterations * W;
    s.longest = s.clock + group * W;
    s.rank = reinterpret_cast<uint32_t*>(s.longest + group * iterations);
    const bool tame = LogNormal::tame(mu, sigma);
    const int threads = W >= 1024 ? 1024 : (W + 31) / 32 * 32;
    int device = 0, sms = 0, resident = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, tame ? straggler_work_kernel<true, false> : straggler_work_kernel<false, false>,
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
            const WorkUnits u = WorkUnits::of(W, s.iterations, s.trials, kSimThreads);
            const bool shared = split == 1 && W >= kSharedRowsW;
            const int64_t units = shared ? u.count : (items * split + kSimThreads - 1) / kSimThreads;
            // Every CTA fills its tables (2 us), but of three per place one that falls behind holds up less: 2744 units, (100, 100, 50,
            // 250, 28), 176 us with one CTA per place, 170 with three; 1775 units, (4, 2, 100, 100, 71), 58 and 65.
            const int64_t most = units >= 4 * work_ctas ? 3 * work_ctas : work_ctas;
            const unsigned ctas = (unsigned)(units < most ? units : most);
            if (shared)
                (tame ? (u.across ? straggler_work_kernel<true, true> : straggler_work_kernel<true, false>)
                      : (u.across ? straggler_work_kernel<false, true>
                                  : straggler_work_kernel<false, false>))<<<ctas, kSimThreads, 0, stream>>>(s, q, (int)u.items,
                                                                                                           (int)u.chunks, units);
            else
                (tame ? straggler_split_work_kernel<true>
                      : straggler_split_work_kernel<false>)<<<ctas, kSimThreads, 0, stream>>>(s, q, split, items);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            if (n == W) {
                auto warps = [&](auto kernel, int64_t count, auto... args) {
                    return launch_overlapped(kernel, dim3((unsigned)((count * 32 + kSimThreads - 1) / kSimThreads)), kSimThreads, 0,
                                             stream, args...);
                };
                e = warps(straggler_longest_kernel, rows, s, rows);
                if (e == cudaSuccess) e = warps(straggler_barrier_kernel, s.trials, s);
                if (e != cudaSuccess) return e;
                continue;
            }
            auto order = [&](auto kernel, int order_threads) {
                return launch_overlapped(kernel, dim3((unsigned)rows), order_threads, draw_scratch_bytes(W, order_threads), stream, s);
            };
            int width = 4;
            while (width < W) width *= 2;
            e = W <= 32 ? launch_overlapped(straggler_order_warp_kernel,
                                            dim3((unsigned)((rows * width + kSimThreads - 1) / kSimThreads)), kSimThreads, 0,
                                            stream, s, rows, width)
              : W <= 512  ? order(straggler_order_kernel<128>, 128)
              : W <= 1024 ? order(straggler_order_kernel<256>, 256)
              : W <= 2048 ? order(straggler_order_kernel<512>, 512)
                          : order(straggler_order_kernel<1024>, 1024);
            if (e != cudaSuccess) return e;
            // Not ahead of the order kernel's end: CTAs that come in as it leaves crowd on the first free SMs, and these
            // run for long (1.03 -> 1.16 ms in all for (4, 2, 100, 500, 592)).
            auto clock = [&](auto kernel, int ahead, bool look) {
                const size_t bytes = clock_bytes(W, W / n, ahead, look);
                const int most = W > 1024 ? NOLO_MAX_WORKERS : 1024;         // as above: for any call of this kernel
                cudaError_t set = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)clock_bytes(most, most, ahead, look));
                if (set != cudaSuccess) return set;
                kernel<<<(unsigned)s.trials, threads, bytes, stream>>>(s, lanes, n > 1 ? 0xffffffffu / n + 1 : 0u);
                return cudaGetLastError();
            };
            e = W > 1024                         ? clock(straggler_clock_kernel<NOLO_MAX_WORKERS / 1024, 2, 0>, 2, false)
              : n == 2                           ? clock(straggler_clock_kernel<1, 4, 2>, 4, true)
              : n <= kLookMost && W <= kLookMaxW ? clock(straggler_clock_kernel<1, 4, kLookMost>, 4, true)
                                                 : clock(straggler_clock_kernel<1, 4, 0>, 4, false);
            if (e != cudaSuccess) return e;
        }
    }
    return launch_stats<2>(per_trial, trials, stats, copy, scratch, stream);
}

}  // namespace nolo
