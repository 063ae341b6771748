// Fused NoLoCo outer step (Section 3.2, Eq. 1-3) for W workers resident in one GPU's memory.
//
// Work decomposition: one CTA owns one subgroup x one tile of parameters.  Every member's
// phi / theta / delta element is fetched from HBM exactly once (128- or 256-bit coalesced, streaming
// cache policy) and every output element stored exactly once; the pseudo-gradients, their sum
// and the subgroup mean of phi exist only on chip.  The path is bandwidth bound (about 15 flops
// per 20-24 bytes), so there is no tensor-core work here.
//
//   Delta_j  = phi_j - theta_j                                            (Eq. 1)
//   delta_i' = alpha*delta_i - (beta/n) sum_j Delta_j - gamma*(phi_i - (1/n) sum_j phi_j)   (Eq. 2)
//   phi_i'   = phi_i + delta_i'                                           (Eq. 3)
//   theta_i' = phi_i'   (start of the next inner phase)
//
// Three kernels cover the subgroup sizes:
//   n <= 8        register-resident: one thread holds its oct of every member;
//   n > 8         two passes over the members, the second read of phi served by L1/L2;
//                 with few columns the threads of a CTA hold all members, and the sums are taken in shared memory.
//
// Arithmetic.  Delta_j is formed per member and summed in float32 in short fixed-order partial
// sums.  gamma * (phi_i - mean phi) is a small number formed from large ones: a mean rounded to
// float32 would pass half an ulp of |phi| straight into delta', whose tolerance does not grow
// with |phi|.  So the mean is carried as an unevaluated float32 pair hi + lo (about 46 bits):
// the register kernel refines a float32 mean by the mean of the residuals phi_j - mean, the
// two-pass kernel sums phi with error-free additions (Knuth's two-sum: the rounding error of every
// addition is recovered exactly and kept in lo).  Float64 accumulators would do the same, but
// the float32 <-> float64 conversions they need run at 16 per clock per SM on B200 and cost
// the wide-subgroup kernels 20-35 % of their bandwidth when measured.
#include "nolo_draw.cuh"
#include "nolo_internal.h"
#include "nolo_launch.cuh"

#include <cuda_bf16.h>

namespace nolo {

namespace {

constexpr int kMostSlots = 32;  // of a two-pass CTA
constexpr int kThreads = 256;   // CTA size of the subgroup-mean kernel

struct KArgs {
    float* phi;
    void* theta;
    float* delta;
    int32_t* perm;
    uint64_t seed, step;      // kernels that draw the partition themselves (DRAW)
    int W;
    const double* mean_phi;   // subgroup means of phi prepared in advance, [groups][mean_stride]; or NULL
    int64_t mean_stride;
    int64_t stride;
    int64_t P;
    int n;
    int tail;                 // 1 when P is no multiple of a thread's columns: the first CTA of every subgroup takes the rest
    float alpha, beta_over_n, gamma, inv_n, n_f;
    double inv_n_d;
};

__device__ __forceinline__ void f4_add(float4& s, const float4 v) {
    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
}
__device__ __forceinline__ float4 f4_sub(const float4 a, const float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float4 f4_zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// ---- the mean of phi as a float32 pair ----------------------------------------------------

// hi + x with the rounding error of the addition added to lo (error-free: hi_new + error == hi + x).
__device__ __forceinline__ void two_sum(float& hi, float& lo, const float x) {
    const float s = hi + x;
    const float bb = s - hi;
    lo += (hi - (s - bb)) + (x - bb);
    hi = s;
}

// Running sum of the phi quads of some members, later the mean: value = hi + lo.
struct PairSum {
    float4 hi, lo;
    __device__ __forceinline__ void clear() { hi = f4_zero(); lo = f4_zero(); }
    __device__ __forceinline__ void add(const float4 v) {
        two_sum(hi.x, lo.x, v.x); two_sum(hi.y, lo.y, v.y); two_sum(hi.z, lo.z, v.z); two_sum(hi.w, lo.w, v.w);
    }
    __device__ __forceinline__ void add(const PairSum& o) { add(o.hi); f4_add(lo, o.lo); }
    // sum -> sum / n.  m = fl(hi / n) leaves hi - m*n, which the fused multiply-add returns exactly.
    static __device__ __forceinline__ void divide1(float& h, float& l, const float inv_n, const float n_f) {
        const float m = h * inv_n;
        const float r = fmaf(-m, n_f, h);
        l = (r + l) * inv_n;
        h = m;
    }
    __device__ __forceinline__ void divide(const KArgs& a) {
        divide1(hi.x, lo.x, a.inv_n, a.n_f); divide1(hi.y, lo.y, a.inv_n, a.n_f);
        divide1(hi.z, lo.z, a.inv_n, a.n_f); divide1(hi.w, lo.w, a.inv_n, a.n_f);
    }
    // phi - mean
    __device__ __forceinline__ float4 deviation(const float4 phi) const { return f4_sub(f4_sub(phi, hi), lo); }
};

// The mean of subgroup g for quad q prepared in advance (float64 in memory), split into hi + lo.
__device__ __forceinline__ PairSum load_prepared_mean(const KArgs& a, int g, int64_t q) {
    const double2* m = reinterpret_cast<const double2*>(a.mean_phi + (int64_t)g * a.mean_stride) + 2 * q;
    const double2 u = load_written(m), v = load_written(m + 1);
    PairSum p;
    p.hi = make_float4((float)u.x, (float)u.y, (float)v.x, (float)v.y);
    p.lo = make_float4((float)(u.x - (double)p.hi.x), (float)(u.y - (double)p.hi.y),
                       (float)(v.x - (double)p.hi.z), (float)(v.y - (double)p.hi.w));
    return p;
}

// ---- theta access: 4 consecutive parameters as float4, fp32 or bf16 storage -------------

__device__ __forceinline__ float4 widen(float4 v) { return v; }
__device__ __forceinline__ float4 widen(uint2 v) {
    float4 r;
    r.x = __uint_as_float(v.x << 16);
    r.y = __uint_as_float(v.x & 0xffff0000u);
    r.z = __uint_as_float(v.y << 16);
    r.w = __uint_as_float(v.y & 0xffff0000u);
    return r;
}
// Raw (unconverted) loads, so that the conversion sits with the arithmetic and never between loads
// (a conversion placed between the loads serialised them when measured).
__device__ __forceinline__ float4 load_theta_raw(const float* row, int64_t q) {
    return __ldcs(reinterpret_cast<const float4*>(row) + q);
}
__device__ __forceinline__ uint2 load_theta_raw(const __nv_bfloat16* row, int64_t q) {
    return __ldcs(reinterpret_cast<const uint2*>(row) + q);
}
template <typename ThetaT> struct ThetaRaw { using type = float4; };
template <> struct ThetaRaw<__nv_bfloat16> { using type = uint2; };

__device__ __forceinline__ void store_theta4(float* row, int64_t q, float4 v) {
    __stcs(reinterpret_cast<float4*>(row) + q, v);
}
__device__ __forceinline__ void store_theta4(__nv_bfloat16* row, int64_t q, float4 v) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y);   // round to nearest even
    const __nv_bfloat162 hi = __floats2bfloat162_rn(v.z, v.w);
    uint2 u;
    u.x = *reinterpret_cast<const uint32_t*>(&lo);
    u.y = *reinterpret_cast<const uint32_t*>(&hi);
    __stcs(reinterpret_cast<uint2*>(row) + q, u);
}
__device__ __forceinline__ float load_theta1(const float* row, int64_t c) { return row[c]; }
__device__ __forceinline__ float load_theta1(const __nv_bfloat16* row, int64_t c) {
    return __bfloat162float(row[c]);
}
__device__ __forceinline__ void store_theta1(float* row, int64_t c, float v) { row[c] = v; }
__device__ __forceinline__ void store_theta1(__nv_bfloat16* row, int64_t c, float v) {
    row[c] = __float2bfloat16_rn(v);
}

// ---- 8 consecutive parameters -------------------------------------------------------------
//
// WIDE: one 256-bit access (rows are 32-byte aligned); else two 128-bit ones.
struct Oct { float v[8]; };

template <bool WIDE>
__device__ __forceinline__ Oct load8(const float* p) {
    Oct o;
    if constexpr (WIDE) {
        asm volatile("ld.global.cs.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=f"(o.v[0]), "=f"(o.v[1]), "=f"(o.v[2]), "=f"(o.v[3]), "=f"(o.v[4]), "=f"(o.v[5]), "=f"(o.v[6]),
                       "=f"(o.v[7])
                     : "l"(p));
    } else {
        const float4 x = __ldcs(reinterpret_cast<const float4*>(p)), y = __ldcs(reinterpret_cast<const float4*>(p) + 1);
        o.v[0] = x.x; o.v[1] = x.y; o.v[2] = x.z; o.v[3] = x.w;
        o.v[4] = y.x; o.v[5] = y.y; o.v[6] = y.z; o.v[7] = y.w;
    }
    return o;
}
template <bool WIDE>
__device__ __forceinline__ void store8(float* p, const Oct& o) {
    if constexpr (WIDE) {
        asm volatile("st.global.cs.v8.f32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"f"(o.v[0]), "f"(o.v[1]), "f"(o.v[2]),
                     "f"(o.v[3]), "f"(o.v[4]), "f"(o.v[5]), "f"(o.v[6]), "f"(o.v[7]), "l"(p)
                     : "memory");
    } else {
        __stcs(reinterpret_cast<float4*>(p), make_float4(o.v[0], o.v[1], o.v[2], o.v[3]));
        __stcs(reinterpret_cast<float4*>(p) + 1, make_float4(o.v[4], o.v[5], o.v[6], o.v[7]));
    }
}
template <typename ThetaT> struct ThetaOct { using type = Oct; };
template <> struct ThetaOct<__nv_bfloat16> { using type = uint4; };
template <bool WIDE>
__device__ __forceinline__ Oct load_theta8(const float* p) { return load8<WIDE>(p); }
template <bool WIDE>
__device__ __forceinline__ uint4 load_theta8(const __nv_bfloat16* p) { return __ldcs(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ float widened(const Oct& o, int e) { return o.v[e]; }
__device__ __forceinline__ float widened(const uint4& o, int e) {
    const uint32_t w = e < 2 ? o.x : e < 4 ? o.y : e < 6 ? o.z : o.w;
    return __uint_as_float(e & 1 ? w & 0xffff0000u : w << 16);
}
template <bool WIDE>
__device__ __forceinline__ void store_theta8(float* p, const Oct& o) { store8<WIDE>(p, o); }
template <bool WIDE>
__device__ __forceinline__ void store_theta8(__nv_bfloat16* p, const Oct& o) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 b = __floats2bfloat162_rn(o.v[2 * i], o.v[2 * i + 1]);   // round to nearest even
        w[i] = *reinterpret_cast<const uint32_t*>(&b);
    }
    __stcs(reinterpret_cast<uint4*>(p), make_uint4(w[0], w[1], w[2], w[3]));
}
template <bool WIDE>
__device__ __forceinline__ void load_means8(double (&m)[8], const double* p) {
    if constexpr (WIDE) {
#pragma unroll
        for (int i = 0; i < 8; i += 4)
            asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
                         : "=d"(m[i]), "=d"(m[i + 1]), "=d"(m[i + 2]), "=d"(m[i + 3]) : "l"(p + i));
    } else {
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const double2 x = load_written(reinterpret_cast<const double2*>(p + i));
            m[i] = x.x; m[i + 1] = x.y;
        }
    }
}

// Eq. 2 and Eq. 3 for one parameter; dev = phi_i - mean phi.
__device__ __forceinline__ float update1(float phi, float dev, float delta, float sum_Delta,
                                         const KArgs& a, float* delta_out) {
    const float d = a.alpha * delta - a.beta_over_n * sum_Delta - a.gamma * dev;
    *delta_out = d;
    return phi + d;
}
__device__ __forceinline__ float4 update4(const float4 phi, const float4 dev, const float4 delta,
                                          const float4 sum_Delta, const KArgs& a, float4* delta_out) {
    float4 p;
    p.x = update1(phi.x, dev.x, delta.x, sum_Delta.x, a, &delta_out->x);
    p.y = update1(phi.y, dev.y, delta.y, sum_Delta.y, a, &delta_out->y);
    p.z = update1(phi.z, dev.z, delta.z, sum_Delta.z, a, &delta_out->z);
    p.w = update1(phi.w, dev.w, delta.w, sum_Delta.w, a, &delta_out->w);
    return p;
}
// update and store one member's quad
template <typename ThetaT>
__device__ __forceinline__ void update_store(const KArgs& a, int64_t row_off, int64_t q, const float4 phi,
                                             const float4 dev, const float4 delta, const float4 sum_Delta) {
    float4 d;
    const float4 p = update4(phi, dev, delta, sum_Delta, a, &d);
    __stcs(reinterpret_cast<float4*>(a.phi + row_off) + q, p);
    __stcs(reinterpret_cast<float4*>(a.delta + row_off) + q, d);
    store_theta4(static_cast<ThetaT*>(a.theta) + row_off, q, p);
}

// ---- the members of a subgroup --------------------------------------------------------------
//
// DRAW = false: read from the table.  DRAW = true (at most 32 workers): the first warp of every CTA draws
// the partition, before it waits for the kernels ahead of it, and keeps its subgroup's members in
// shared memory; the first CTA writes the table as well.  Both wait for the kernels ahead of this one.
// (Having phi and theta of the first tiles brought to L2 ahead of the wait measured no gain since the kernel ahead is
// mostly done by then: 61.0 us with, 60.5 without for steps that follow each other, W = 4, P = 2^22, n = 2; 63.6 / 63.9
// behind a routing copy.)
template <bool DRAW> struct Members;
template <> struct Members<false> {
    const int32_t* list;
    __device__ __forceinline__ void init(const KArgs& a, int g, int*) {
        list = a.perm + (int64_t)g * a.n;
        wait_for_predecessors();
    }
    __device__ __forceinline__ int operator[](int j) const { return load_written(list + j); }
};
template <> struct Members<true> {
    const int* list;                     // shared memory
    __device__ __forceinline__ void init(const KArgs& a, int g, int* shared) {
        list = shared;
        int rank = 0;
        if (threadIdx.x < 32) {
            rank = rank_by_warp(a.W, 0, 0, kDomainGroups, a.seed, a.step);
            if ((int)threadIdx.x < a.W && rank / a.n == g) shared[rank - g * a.n] = threadIdx.x;
        }
        wait_for_predecessors();
        if (blockIdx.x == 0 && g == 0 && (int)threadIdx.x < a.W) a.perm[rank] = threadIdx.x;
        __syncthreads();
    }
    __device__ __forceinline__ int operator[](int j) const { return list[j]; }
};

// Columns P - (P % VEC) .. P-1 of one subgroup (a thread has VEC columns elsewhere), element by element
// with float64 sums (rows are only guaranteed to be padded to a multiple of 8, and padding must not be
// written).  Done by a CTA of its own, the first of the subgroup: VEC neighbouring threads per member, so
// a pass over the members is one or a few loads in flight per thread.  One thread walking the members
// column by column is a serial chain of loads; one CTA is not: 3 extra columns cost 7.7 us before and
// nothing measurable now at n = 20 (73.5 -> 67.4 us for W = 60, P = 2^18 + 3), 197 us at n = 256, 1.42 ms
// at n = 1024 (2531 -> 1056 us for P = 2^18 + 3).
template <typename ThetaT, int THREADS, int VEC, typename M>
__device__ __forceinline__ void ragged_tail(const KArgs& a, int g, const M& members) {
    constexpr int WARPS = THREADS / 32, ROWS = THREADS / VEC;
    __shared__ double2 part[WARPS][VEC];
    const int n = a.n;
    const int64_t c = (a.P & ~int64_t(VEC - 1)) + threadIdx.x % VEC;
    const int first = threadIdx.x / VEC;
    const bool mine = c < a.P;
    double sD = 0.0, sP = 0.0;
    if (mine) {
#pragma unroll 4
        for (int j = first; j < n; j += ROWS) {
            const int64_t at = (int64_t)members[j] * a.stride + c;
            const float p = a.phi[at];
            sD += (double)(p - load_theta1(static_cast<const ThetaT*>(a.theta), at));
            sP += (double)p;
        }
    }
#pragma unroll
    for (int o = VEC; o < 32; o <<= 1) {
        sD += __shfl_xor_sync(0xffffffffu, sD, o);
        sP += __shfl_xor_sync(0xffffffffu, sP, o);
    }
    if ((threadIdx.x & 31) < VEC) part[threadIdx.x >> 5][threadIdx.x % VEC] = make_double2(sD, sP);
    __syncthreads();
    if (!mine) return;
    sD = sP = 0.0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) { sD += part[w][threadIdx.x % VEC].x; sP += part[w][threadIdx.x % VEC].y; }
    const double mP = a.mean_phi ? a.mean_phi[(int64_t)g * a.mean_stride + c] : sP * a.inv_n_d;
    for (int j0 = first; j0 < n; j0 += 4 * ROWS) {        // four rows in flight
        float p[4], d[4];
        int64_t at[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (j0 + i * ROWS < n) {
                at[i] = (int64_t)members[j0 + i * ROWS] * a.stride + c;
                p[i] = a.phi[at[i]];
                d[i] = a.delta[at[i]];
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (j0 + i * ROWS < n) {
                float dn;
                const float pn = update1(p[i], (float)((double)p[i] - mP), d[i], (float)sD, a, &dn);
                a.phi[at[i]] = pn;
                a.delta[at[i]] = dn;
                store_theta1(static_cast<ThetaT*>(a.theta), at[i], pn);
            }
        }
    }
}

// ---- n <= 8: register-resident, subgroup size N known at compile time --------------------
//
// Each thread handles one oct (8 consecutive parameters) for all N members: phi_j stays in registers
// between the reduction and the update, so nothing is read twice.  All loads of a thread are issued
// before the first use to keep many bytes in flight.
//
// Bound by DRAM.  256-bit accesses make a row piece of one warp 1 KB long and halve the requests, and the rate rises
// with what is in flight per thread: 6923 GB/s for pairs with float32 theta (W = 16, P = 2^25), 6822 in quads by 128-bit
// accesses; 6739 against 5568 with n = 8 and bfloat16 theta, where quads left one CTA of 256 threads per SM.
template <int N, typename ThetaT, int THREADS, bool PREPARED, bool WIDE, bool DRAW>
__global__ void __launch_bounds__(THREADS, 1)
outer_step_reg_kernel(const KArgs a) {
    const int g = blockIdx.y;
    __shared__ int drawn[DRAW ? N : 1];
    Members<DRAW> members;
    members.init(a, g, drawn);
    if (a.tail && blockIdx.x == 0) {
        ragged_tail<ThetaT, THREADS, 8>(a, g, members);
        return;
    }
    const int64_t c = ((int64_t)(blockIdx.x - a.tail) * THREADS + threadIdx.x) * 8;
    if (c + 8 > a.P) return;

    int64_t at[N];
#pragma unroll
    for (int j = 0; j < N; ++j) at[j] = (int64_t)members[j] * a.stride + c;
    Oct phi[N], dlt[N];
    typename ThetaOct<ThetaT>::type the[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        phi[j] = load8<WIDE>(a.phi + at[j]);
        the[j] = load_theta8<WIDE>(static_cast<const ThetaT*>(a.theta) + at[j]);
    }
#pragma unroll
    for (int j = 0; j < N; ++j) dlt[j] = load8<WIDE>(a.delta + at[j]);
    double mean[PREPARED ? 8 : 1];
    if constexpr (PREPARED) load_means8<WIDE>(mean, a.mean_phi + (int64_t)g * a.mean_stride + c);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        // Sums in the fixed member order (deterministic).  The mean of phi is formed in two
        // passes over the registers: a plain float32 mean, then the mean of the residuals
        // phi_j - mean, so that hi + lo keeps the precision of the spread of the replicas.
        float sD = 0.f, s0 = 0.f, hi, lo;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            sD += phi[j].v[e] - widened(the[j], e);                      // Eq. 1
            s0 += phi[j].v[e];
        }
        if constexpr (PREPARED) {
            hi = (float)mean[e];
            lo = (float)(mean[e] - (double)hi);
        } else {
            hi = s0 * a.inv_n;
            float sR = 0.f;
#pragma unroll
            for (int j = 0; j < N; ++j) sR += phi[j].v[e] - hi;
            lo = sR * a.inv_n;
        }
#pragma unroll
        for (int j = 0; j < N; ++j)
            phi[j].v[e] = update1(phi[j].v[e], (phi[j].v[e] - hi) - lo, dlt[j].v[e], sD, a, &dlt[j].v[e]);
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
        store8<WIDE>(a.phi + at[j], phi[j]);
        store8<WIDE>(a.delta + at[j], dlt[j]);
        store_theta8<WIDE>(static_cast<ThetaT*>(a.theta) + at[j], phi[j]);
    }
}

// ---- n > 8: two passes over the members, the second read of phi served by L1 / L2 ----------
//
// One CTA owns one subgroup x ROWQ quads.  Its THREADS threads form THREADS/ROWQ slots of ROWQ
// consecutive quads; slot s walks members s, s + SLOTS, ... in chunks of U rows in flight.  Pass 1
// reads phi and theta and accumulates the two sums; the slots' partial sums meet in shared memory;
// pass 2 reads phi again together with delta and writes the update.  Between the two reads of a
// phi element lie only the other rows of the same CTA's tile (n x ROWQ x 16 bytes), so the second
// read is served by L1 or L2 as long as the tiles of all resident CTAs fit there: profiled DRAM
// traffic equals the algorithmic 24 / 20 bytes per worker-parameter, and nothing has to be parked
// in registers or shared memory, whatever n is.  The first chunk of pass 2 depends on no sum, so
// its loads are issued before the partial sums meet and are in flight across the CTA barrier.
// No bulk copies, no clusters and no waits other than that one barrier (none at all with one slot).
//
// The shape trades three things: bytes in flight (threads x U), the width of the piece of a row
// that one CTA streams (ROWQ x 16 bytes: DRAM likes 1-2 KB pieces better than 512-byte ones, and
// 256-byte ones least) and the L2 footprint of the resident tiles
// (CTAs per SM x n x ROWQ x 16 bytes x 148 SMs), which must stay well below the 126 MB of L2 or
// the re-read goes to DRAM.  Small subgroups therefore take wide pieces and few slots, large
// ones narrow pieces; the best shapes have SLOTS x U close to n, so that a slot walks its rows
// in one to four chunks.  Measured on B200 as a fraction of a plain copy (float32 / bfloat16
// theta): 0.96-0.97 / 0.94-0.96 up to 48 members, 0.95 / 0.94 at 64 and at 96, 0.93 at 128,
// 0.92 up to 224, 0.93-0.88 up to 640, 0.89 / 0.84 at 1024.
//
// Tried and measured slower on this access pattern: members held in registers by the warps of a
// CTA, one pass (0.94 for 9-64 members: 512-byte pieces); rings of asynchronous copies (cp.async)
// that keep several chunks in flight per thread (same rate: the kernel is not short of loads in
// flight); phi parked in shared memory; phi parked in tensor memory (tcgen05.st / tcgen05.ld;
// exact, but two CTAs of eight warps per SM are too few warps: 0.78-0.85); a persistent grid
// (0.5-0.7: all CTAs in the same phase at once).  With the re-read of phi left out altogether
// the 512-byte-piece loops reach only 0.92 / 0.91 / 0.89 of a plain copy at n = 128 / 256 / 1024:
// what is lost is lost to streaming n x 3 rows in narrow pieces, not to the second read.
template <typename ThetaT, int THREADS, int ROWQ, int U, int MINB, bool DRAW>
__global__ void __launch_bounds__(THREADS, MINB)
outer_step_twopass_kernel(const KArgs a) {
    static_assert(THREADS % 32 == 0 && THREADS % ROWQ == 0, "slots tile the CTA");
    static_assert(ROWQ >= 32 ? ROWQ % 32 == 0 : 32 % ROWQ == 0, "a slot is whole warps or a whole fraction of one");
    constexpr int SLOTS = THREADS / ROWQ;
    constexpr int WARPS = THREADS / 32;
    // Partial sums that meet in shared memory: one per slot when slots are whole warps, one per warp
    // when a warp holds several slots (those are first added by shuffles).
    constexpr int PARTS = ROWQ >= 32 ? SLOTS : WARPS;
    __shared__ float4 part_D[PARTS][ROWQ];
    __shared__ PairSum part_P[PARTS][ROWQ];
    const int lane = threadIdx.x & 31;
    const int ql = threadIdx.x % ROWQ;
    const int slot = threadIdx.x / ROWQ;
    const int part = ROWQ >= 32 ? slot : (threadIdx.x >> 5);
    const int g = blockIdx.y;
    const int n = a.n;
    __shared__ int drawn[DRAW ? 32 : 1];
    Members<DRAW> members;
    members.init(a, g, drawn);
    if (a.tail && blockIdx.x == 0) {
        ragged_tail<ThetaT, THREADS, 4>(a, g, members);
        return;
    }
    const int64_t q = (int64_t)(blockIdx.x - a.tail) * ROWQ + ql;
    const bool ok = q < (a.P >> 2);

    float4 sD = f4_zero();
    PairSum sP;
    sP.clear();
    if (ok) {
        for (int j = slot; j < n; j += SLOTS * U) {
            float4 p[U];
            typename ThetaRaw<ThetaT>::type t[U];
#pragma unroll
            for (int i = 0; i < U; ++i) {
                const int jj = j + i * SLOTS;
                if (jj < n) {
                    const int64_t off = (int64_t)members[jj] * a.stride;
                    p[i] = reinterpret_cast<const float4*>(a.phi + off)[q];     // default policy: stays cached for pass 2
                    t[i] = load_theta_raw(static_cast<const ThetaT*>(a.theta) + off, q);
                }
            }
#pragma unroll
            for (int i = 0; i < U; ++i) {
                if (j + i * SLOTS < n) {
                    f4_add(sD, f4_sub(p[i], widen(t[i])));              // Eq. 1
                    sP.add(p[i]);
                }
            }
        }
    }
    // pass 2, chunk by chunk: phi (from L1 / L2) and delta of U rows
    float4 p2[U], d2[U];
    int64_t off2[U];
    auto load_chunk = [&](int j) {
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int jj = j + i * SLOTS;
            if (jj < n) {
                off2[i] = (int64_t)members[jj] * a.stride;
                p2[i] = __ldcs(reinterpret_cast<const float4*>(a.phi + off2[i]) + q);
                d2[i] = __ldcs(reinterpret_cast<const float4*>(a.delta + off2[i]) + q);
            }
        }
    };
    if (ok) load_chunk(slot);      // in flight while the partial sums meet
    if constexpr (ROWQ < 32) {
        // the slots of one warp that share a quad, in a fixed order
#pragma unroll
        for (int o = ROWQ; o < 32; o <<= 1) {
            PairSum t;
            float4 d;
            d.x = __shfl_xor_sync(0xffffffffu, sD.x, o); d.y = __shfl_xor_sync(0xffffffffu, sD.y, o);
            d.z = __shfl_xor_sync(0xffffffffu, sD.z, o); d.w = __shfl_xor_sync(0xffffffffu, sD.w, o);
            t.hi.x = __shfl_xor_sync(0xffffffffu, sP.hi.x, o); t.hi.y = __shfl_xor_sync(0xffffffffu, sP.hi.y, o);
            t.hi.z = __shfl_xor_sync(0xffffffffu, sP.hi.z, o); t.hi.w = __shfl_xor_sync(0xffffffffu, sP.hi.w, o);
            t.lo.x = __shfl_xor_sync(0xffffffffu, sP.lo.x, o); t.lo.y = __shfl_xor_sync(0xffffffffu, sP.lo.y, o);
            t.lo.z = __shfl_xor_sync(0xffffffffu, sP.lo.z, o); t.lo.w = __shfl_xor_sync(0xffffffffu, sP.lo.w, o);
            // both partners add (lower slot) + (higher slot) in that order, so they agree bit for bit
            if (lane & o) {
                PairSum mine = sP;
                sP = t;
                sP.add(mine);
                d.x += sD.x; d.y += sD.y; d.z += sD.z; d.w += sD.w;
                sD = d;
            } else {
                sP.add(t);
                f4_add(sD, d);
            }
        }
    }
    if constexpr (PARTS > 1) {
        // the partial sums of the slots (or warps) meet in shared memory
        if (ROWQ >= 32 || lane < ROWQ) {
            part_D[part][ql] = sD;
            part_P[part][ql] = sP;
        }
        __syncthreads();
    }
    if (ok) {
        if constexpr (PARTS > 1) {          // added in index order: the same result in every slot
            sD = part_D[0][ql];
            sP = part_P[0][ql];
#pragma unroll
            for (int w = 1; w < PARTS; ++w) {
                f4_add(sD, part_D[w][ql]);
                sP.add(part_P[w][ql]);
            }
        }
        if (a.mean_phi) sP = load_prepared_mean(a, g, q);
        else sP.divide(a);
        for (int j = slot; j < n; j += SLOTS * U) {
            if (j != slot) load_chunk(j);
#pragma unroll
            for (int i = 0; i < U; ++i) {
                if (j + i * SLOTS < n) update_store<ThetaT>(a, off2[i], q, p2[i], sP.deviation(p2[i]), d2[i], sD);
            }
        }
    }
}

// ---- n > 8, few columns: every row in flight at once ------------------------------------------
//
// One CTA owns one subgroup x ROWQ quads, and its threads hold every member's piece: ROWS members each, phi and delta in
// registers, phi and Delta in shared memory as well.  There the sums are taken column by column, by a thread for each column,
// slot and kind of sum; the slots are those of the two-pass shape that these states would have otherwise, and their sums meet in
// its order, so every bit is the same, whatever the number of columns.
//
// Bound by latency: the table's, one read of all rows, three barriers.  (W, n, P) float32, us in a train, two passes / this: (32, 32, 3125)
// 5.6 / 3.4, (60, 60, 1667) 10.3 / 5.5, (96, 96, 4166) 13.2 / 5.8, (256, 256, 1562) 11.1 / 7.2, (512, 512, 3125) 18.9 / 15.6,
// (1024, 1024, 1563) 30.6 / 16.1.
template <typename ThetaT, int THREADS, int ROWQ, int ROWS, bool DRAW>
__global__ void __launch_bounds__(THREADS, 1)
outer_step_staged_kernel(const KArgs a, int slots) {
    constexpr int WALK = THREADS / ROWQ, COLS = 4 * ROWQ;
    extern __shared__ float4 staged[];                         // [n][ROWQ] phi, [n][ROWQ] Delta
    __shared__ float part_D[kMostSlots][COLS], part_hi[kMostSlots][COLS], part_lo[kMostSlots][COLS];
    __shared__ float4 total_D[ROWQ], total_hi[ROWQ], total_lo[ROWQ];
    const int g = blockIdx.y, n = a.n;
    __shared__ int drawn[DRAW ? 32 : 1];
    Members<DRAW> members;
    members.init(a, g, drawn);
    if (a.tail && blockIdx.x == 0) {
        ragged_tail<ThetaT, THREADS, 4>(a, g, members);
        return;
    }
    const int ql = threadIdx.x % ROWQ, walk = threadIdx.x / ROWQ;
    const int64_t q = (int64_t)(blockIdx.x - a.tail) * ROWQ + ql;
    const bool ok = q < (a.P >> 2);
    float4 p[ROWS], d[ROWS];
    typename ThetaRaw<ThetaT>::type t[ROWS];
    int row[ROWS];
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        const int j = walk + i * WALK;
        if (ok && j < n) row[i] = members[j];
    }
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        if (ok && walk + i * WALK < n) {
            const int64_t off = row[i] * a.stride;
            p[i] = __ldcs(reinterpret_cast<const float4*>(a.phi + off) + q);
            t[i] = load_theta_raw(static_cast<const ThetaT*>(a.theta) + off, q);
            d[i] = __ldcs(reinterpret_cast<const float4*>(a.delta + off) + q);
        }
    }
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
        const int j = walk + i * WALK;
        if (ok && j < n) {
            staged[j * ROWQ + ql] = p[i];
            staged[(n + j) * ROWQ + ql] = f4_sub(p[i], widen(t[i]));                    // Eq. 1
        }
    }
    __syncthreads();
    const float* phi = reinterpret_cast<const float*>(staged);
    const float* Delta = phi + n * COLS;
    for (int task = threadIdx.x; task < 2 * slots * COLS; task += THREADS) {
        const int c = task % COLS, slot = task / COLS % slots;
        if (task < slots * COLS) {
            float sum = 0.f;
            for (int j = slot; j < n; j += slots) sum += Delta[j * COLS + c];
            part_D[slot][c] = sum;
        } else {
            float hi = 0.f, lo = 0.f;
            for (int j = slot; j < n; j += slots) two_sum(hi, lo, phi[j * COLS + c]);
            part_hi[slot][c] = hi;
            part_lo[slot][c] = lo;
        }
    }
    __syncthreads();
    if (threadIdx.x < COLS) {
        // as the two-pass kernel does it: the two slots of a warp first, where it has 16 quads per slot
        const int c = threadIdx.x, pair = slots >= 16 ? 2 : 1;
        float sD = 0.f, hi = 0.f, lo = 0.f;
        for (int w = 0; w < slots; w += pair) {
            float D = part_D[w][c], h = part_hi[w][c], l = part_lo[w][c];
            if (pair == 2) {
                D += part_D[w + 1][c];
                two_sum(h, l, part_hi[w + 1][c]);
                l += part_lo[w + 1][c];
            }
            if (w == 0) {
                sD = D; hi = h; lo = l;
            } else {
                sD += D;
                two_sum(hi, lo, h);
                lo += l;
            }
        }
        reinterpret_cast<float*>(total_D)[c] = sD;
        reinterpret_cast<float*>(total_hi)[c] = hi;
        reinterpret_cast<float*>(total_lo)[c] = lo;
    }
    __syncthreads();
    if (!ok) return;
    const float4 sD = total_D[ql];
    PairSum sP;
    sP.hi = total_hi[ql];
    sP.lo = total_lo[ql];
    if (a.mean_phi) sP = load_prepared_mean(a, g, q);
    else sP.divide(a);
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
        if (walk + i * WALK < n) update_store<ThetaT>(a, row[i] * a.stride, q, p[i], sP.deviation(p[i]), d[i], sD);
}

// ---- subgroup means of phi alone (first half of the split-phase step) ------------------------
//
// mean[g][p] = (1/n) sum_{j in subgroup g} phi_j[p], stored as float64.  Section 3.2 notes that
// the slow weights of the partners are known as soon as the previous outer step has finished, so
// this part of Eq. 2 can be exchanged early; only the pseudo-gradients have to wait for the inner
// phase.  Read-only on phi: 4 bytes read per worker-parameter, 8/n bytes written.
constexpr int kMeanUnroll = 4;   // member rows in flight per quad

// Four consecutive float64 means with one 256-bit store (one whole 32-byte sector per lane) where
// the row is 32-byte aligned, else as two 128-bit stores.
template <bool WIDE>
__device__ __forceinline__ void store_mean4(double* out, double a, double b, double c, double d) {
    if (WIDE) {
        asm volatile("st.global.cs.v4.f64 [%0], {%1, %2, %3, %4};" :: "l"(out), "d"(a), "d"(b), "d"(c), "d"(d) : "memory");
    } else {
        __stcs(reinterpret_cast<double2*>(out), make_double2(a, b));
        __stcs(reinterpret_cast<double2*>(out) + 1, make_double2(c, d));
    }
}

__device__ __forceinline__ void copy_ahead16(void* to, const void* from) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from) : "memory");
}

// The columns of the partial quad, one warp per column.
__device__ __forceinline__ void mean_tail(const float* phi, const int32_t* members, int n, int64_t stride, int64_t P, double* mean,
                                          double inv_n) {
    const int64_t c = (P & ~int64_t(3)) + (threadIdx.x >> 5);
    if (c >= P) return;
    double t = 0.0;
#pragma unroll 4
    for (int j = threadIdx.x & 31; j < n; j += 32) t += (double)phi[(int64_t)load_written(members + j) * stride + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) mean[c] = t * inv_n;
}

// A thread adds the members of ITEMS quads, 256 quads apart: small subgroups have few rows to keep in flight per
// quad, so each thread takes two quads up to n = 4.
template <int ITEMS, bool WIDE>
__global__ void __launch_bounds__(kThreads)
group_mean_kernel(const float* phi, const int32_t* perm, int n, int64_t stride,
                  int64_t P, double* __restrict__ mean, int64_t mean_stride, double inv_n) {
    wait_for_predecessors();
    let_successor_start();
    const int g = blockIdx.y;
    const int32_t* members = perm + (int64_t)g * n;
    mean += (int64_t)g * mean_stride;
    const int tail = (P & 3) != 0;
    if (tail && blockIdx.x == 0) return mean_tail(phi, members, n, stride, P, mean, inv_n);
    const int64_t q0 = (int64_t)(blockIdx.x - tail) * (kThreads * ITEMS) + threadIdx.x;
    const int64_t quads = P >> 2;
    PairSum s[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) s[it].clear();
    for (int j = 0; j < n; j += kMeanUnroll) {
        float4 v[ITEMS][kMeanUnroll];
#pragma unroll
        for (int i = 0; i < kMeanUnroll; ++i) {
            if (j + i < n) {
                const float4* row = reinterpret_cast<const float4*>(phi + (int64_t)load_written(members + j + i) * stride);
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    const int64_t q = q0 + (int64_t)it * kThreads;
                    if (q < quads) v[it][i] = __ldcs(row + q);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < kMeanUnroll; ++i) {
            if (j + i < n) {
#pragma unroll
                for (int it = 0; it < ITEMS; ++it)
                    if (q0 + (int64_t)it * kThreads < quads) s[it].add(v[it][i]);
            }
        }
    }
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        const int64_t q = q0 + (int64_t)it * kThreads;
        if (q < quads) {
            store_mean4<WIDE>(mean + 4 * q,
                              ((double)s[it].hi.x + (double)s[it].lo.x) * inv_n, ((double)s[it].hi.y + (double)s[it].lo.y) * inv_n,
                              ((double)s[it].hi.z + (double)s[it].lo.z) * inv_n, ((double)s[it].hi.w + (double)s[it].lo.w) * inv_n);
        }
    }
}

// The same for few columns, whose CTAs would not fill the chip and whose threads would walk the members in many latencies:
// the CTA's threads bring the members of 4 QUADS columns to shared memory, three stages of 8 KB ahead, and a thread per column adds
// them in the order of the kernel above, so that no bit depends on the number of columns.  Bound by latency up to about a
// hundred members, then by the additions, whose chain is 4 cycles and whose 7 instructions a member has in each column's thread
// alone.  (Groups of threads that share out the members and join their sums in a tree took 124 us at (1024, 37 888) and gave other
// bits than a thread per quad; rows brought through registers, one stage of 16 KB ahead, 189.)
//
// It lets its successor start early for small states only: else the step that follows would find the SMs set up for this kernel's
// shared memory and keep them so, with little L1 left for its loads in flight.  us of prepare and prepared step, early / not, n = W:
// (1024, 24 415) 192 / 154, (64, 300 000) 118 / 95, (96, 66 666) 36.9 / 31.1, (256, 6251) 18.8 / 19.1, (1024, 1563) 31.0 / 32.9.
constexpr int kMeanStages = 4, kMeanStageQuads = 2 * kThreads;

template <int QUADS>
__global__ void __launch_bounds__(kThreads)
staged_mean_kernel(const float* phi, const int32_t* perm, int n, int64_t stride, int64_t P, double* __restrict__ mean,
                   int64_t mean_stride, double inv_n, bool early) {
    constexpr int COLS = 4 * QUADS, ROWS = kMeanStageQuads / QUADS, HALF = ROWS / 2;
    __shared__ float4 staged[kMeanStages][ROWS][QUADS];
    wait_for_predecessors();
    if (early) let_successor_start();
    const int g = blockIdx.y;
    const int32_t* members = perm + (int64_t)g * n;
    mean += (int64_t)g * mean_stride;
    const int tail = (P & 3) != 0;
    if (tail && blockIdx.x == 0) return mean_tail(phi, members, n, stride, P, mean, inv_n);
    const int ql = threadIdx.x % QUADS, row = threadIdx.x / QUADS;
    const int64_t first = (int64_t)(blockIdx.x - tail) * QUADS, quads = P >> 2;
    const bool ok = first + ql < quads;
    phi += 4 * (first + ql);
    int m0[kMeanStages - 1], m1[kMeanStages - 1];              // this thread's members of the stages ahead
#pragma unroll
    for (int u = 0; u < kMeanStages - 1; ++u) {
        const int j = u * ROWS + row;
        if (j < n) m0[u] = load_written(members + j);
        if (j + HALF < n) m1[u] = load_written(members + j + HALF);
    }
    auto ahead = [&](int j0, int slot, int a, int b) {
        if (ok && j0 + row < n) copy_ahead16(&staged[slot][row][ql], phi + (int64_t)a * stride);
        if (ok && j0 + row + HALF < n) copy_ahead16(&staged[slot][row + HALF][ql], phi + (int64_t)b * stride);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int u = 0; u < kMeanStages - 1; ++u) ahead(u * ROWS, u, m0[u], m1[u]);
    float hi = 0.f, lo = 0.f;
    int slot = 0;
    for (int j0 = 0; j0 < n; j0 += ROWS) {
        const int next = j0 + (kMeanStages - 1) * ROWS;
        int a = 0, b = 0;
        if (next + row < n) a = load_written(members + next + row);
        if (next + row + HALF < n) b = load_written(members + next + row + HALF);
        asm volatile("cp.async.wait_group %0;" ::"n"(kMeanStages - 2) : "memory");
        __syncthreads();
        ahead(next, (slot + kMeanStages - 1) % kMeanStages, a, b);      // where the stage before this one was
        if (threadIdx.x < COLS) {
            const float* x = reinterpret_cast<const float*>(staged[slot]) + threadIdx.x;
            const int count = n - j0 < ROWS ? n - j0 : ROWS;
#pragma unroll 8
            for (int j = 0; j < count; ++j) two_sum(hi, lo, x[j * COLS]);
        }
        slot = (slot + 1) % kMeanStages;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    const int64_t c = 4 * first + threadIdx.x;
    if (threadIdx.x < COLS && c < 4 * quads) mean[c] = ((double)hi + (double)lo) * inv_n;
}

// ---- launches ---------------------------------------------------------------------------

// Tiles of `cols_per_cta` columns (whole vectors of `vec` columns per thread), and one more CTA for
// the columns that are left over.
bool tile_grid(KArgs& k, int vec, int64_t cols_per_cta, int groups, dim3* grid) {
    k.tail = k.P % vec != 0;
    const int64_t tiles = (k.P - k.P % vec + cols_per_cta - 1) / cols_per_cta + k.tail;
    if (tiles > 0x7fffffffll) return false;
    *grid = dim3((unsigned)tiles, (unsigned)groups);
    return true;
}

bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

template <int N, typename ThetaT, int THREADS, bool WIDE, bool DRAW>
cudaError_t launch_reg_shape(KArgs& k, int groups, cudaStream_t stream) {
    dim3 grid;
    if (!tile_grid(k, 8, (int64_t)THREADS * 8, groups, &grid)) return cudaErrorInvalidConfiguration;
    return launch_overlapped(k.mean_phi ? outer_step_reg_kernel<N, ThetaT, THREADS, true, WIDE, DRAW>
                                        : outer_step_reg_kernel<N, ThetaT, THREADS, false, WIDE, DRAW>,
                             grid, THREADS, 0, stream, k);
}

// CTA sizes.  Larger CTAs stream longer pieces of a row, but the ends of the grid weigh more: 64 threads below 2^19
// octs (W = 4, P = 2^20, n = 2 16.4 us, with 256 threads 16.8) and where a thread has more than 4 members, for the
// registers that leaves it; else 256, or what fits the registers better: 192 with 4 members (1878 us with 256 threads 1888,
// W = 16, P = 2^25, float32; bfloat16 1580 / 1613), 320 for pairs with bfloat16 theta (1561 / 1567; smaller states lose
// up to 2 %, 101.1 / 99.1 at P = 2^21).
constexpr int64_t kRegManyOcts = 1 << 19;
template <int N, typename ThetaT>
constexpr int kRegThreads = N == 4 ? 192 : (N == 2 && sizeof(ThetaT) == 2) ? 320 : 256;

template <int N, typename ThetaT>
cudaError_t launch_reg(KArgs& k, bool draw, int groups, cudaStream_t stream) {
    // the strides are multiples of 32 bytes (of 16 for bfloat16 theta, which is read 16 bytes at a time)
    const bool wide = aligned32(k.phi) && aligned32(k.delta) && (sizeof(ThetaT) == 2 || aligned32(k.theta)) &&
                      aligned32(k.mean_phi);
    if (!wide) return draw ? launch_reg_shape<N, ThetaT, 64, false, true>(k, groups, stream)
                           : launch_reg_shape<N, ThetaT, 64, false, false>(k, groups, stream);
    if constexpr (N <= 4) {
        if (k.P / 8 * groups >= kRegManyOcts)
            return draw ? launch_reg_shape<N, ThetaT, kRegThreads<N, ThetaT>, true, true>(k, groups, stream)
                        : launch_reg_shape<N, ThetaT, kRegThreads<N, ThetaT>, true, false>(k, groups, stream);
    }
    return draw ? launch_reg_shape<N, ThetaT, 64, true, true>(k, groups, stream)
                : launch_reg_shape<N, ThetaT, 64, true, false>(k, groups, stream);
}

// CTAs up to which all rows are taken at once: with 8 quads each (n <= 128) about what runs at a time, with 4 quads (n <= 1024,
// 512 threads) two turns.  us in a train, two passes / staged, float32: 521 CTAs (96, 96, 16 667) 13.1 / 9.8, 391 (32, 32, 12 501) 5.6 /
// 3.9, 1042 (24, 12, 16 667) 5.8 / 6.1; of 4 quads 196 (512, 512, 3125) 19.3 / 16.5, 392 (1024, 256, 1563) 13.9 / 19.0.
constexpr int64_t kStagedCtas = 148 * 4, kStagedCtasWide = 148 * 2;

template <typename ThetaT, int THREADS, int ROWQ, int ROWS, bool DRAW>
cudaError_t launch_staged(KArgs& k, int slots, int groups, cudaStream_t stream) {
    dim3 grid;
    if (!tile_grid(k, 4, (int64_t)ROWQ * 4, groups, &grid)) return cudaErrorInvalidConfiguration;
    const size_t smem = (size_t)k.n * ROWQ * 2 * sizeof(float4);
    auto kernel = outer_step_staged_kernel<ThetaT, THREADS, ROWQ, ROWS, DRAW>;
    // the most that any subgroup needs, so that calls of different sizes from several threads do not undo each other's
    constexpr int kMost = ROWS * THREADS * 2 * (int)sizeof(float4);
    if constexpr (kMost > 32768) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost);
        if (e != cudaSuccess) return e;
    }
    return launch_overlapped(kernel, grid, THREADS, smem, stream, k, slots);
}

template <typename ThetaT, int THREADS, int ROWQ, int U, int MINB>
cudaError_t launch_twopass(KArgs& k, bool draw, int groups, cudaStream_t stream) {
    constexpr int SLOTS = THREADS / ROWQ;
    static_assert(SLOTS <= kMostSlots && (SLOTS >= 16) == (ROWQ == 16), "the staged kernel adds the slots in the same order");
    if (k.n <= 128 && (k.P + 31) / 32 * groups <= kStagedCtas) {
        if (k.n <= 32) return draw ? launch_staged<ThetaT, 256, 8, 1, true>(k, SLOTS, groups, stream)
                                   : launch_staged<ThetaT, 256, 8, 1, false>(k, SLOTS, groups, stream);
        if (!draw) return launch_staged<ThetaT, 256, 8, 4, false>(k, SLOTS, groups, stream);
    }
    if (k.n > 128 && k.n <= 1024 && !draw && (k.P + 15) / 16 * groups <= kStagedCtasWide)
        return launch_staged<ThetaT, 512, 4, 8, false>(k, SLOTS, groups, stream);
    dim3 grid;
    if (!tile_grid(k, 4, (int64_t)ROWQ * 4, groups, &grid)) return cudaErrorInvalidConfiguration;
    if constexpr (ROWQ >= 64 && U * THREADS / ROWQ <= 16) {       // the shapes of up to 32 members
        if (draw)
            return launch_overlapped(outer_step_twopass_kernel<ThetaT, THREADS, ROWQ, U, MINB, true>, grid, THREADS, 0,
                                     stream, k);
    }
    if (draw) return cudaErrorInvalidValue;
    return launch_overlapped(outer_step_twopass_kernel<ThetaT, THREADS, ROWQ, U, MINB, false>, grid, THREADS, 0, stream, k);
}

// Subgroup sizes up to which each two-pass shape is used (by measurement, see the kernel's comment):
// threads x quads per row piece x rows in flight per slot, CTAs per SM.
constexpr int kTwoPassMaxN1Slot = 12;     // 128 x 128 x 4, 6 CTAs: one slot, no barrier
constexpr int kTwoPassMaxN2Slots = 24;    // 128 x 64 x 8, 4 CTAs
constexpr int kTwoPassMaxN64Quads4 = 64;  // 256 x 64 x 4, 3 CTAs
constexpr int kTwoPassMaxN64Quads8 = 96;  // 256 x 64 x 8, 2 CTAs
constexpr int kTwoPassMaxN4Rows = 128;    // 256 x 32 x 4, 3 CTAs
constexpr int kTwoPassMaxN32Quads = 224;  // 256 x 32 x 8, 2 CTAs
constexpr int kTwoPassMaxN8Warps = 640;   // 256 x 16 x 8, 2 CTAs; above: 512 x 16 x 8, 1 CTA

template <typename ThetaT>
cudaError_t dispatch(KArgs& k, bool draw, int groups, cudaStream_t stream) {
    switch (k.n) {
        case 1:  return launch_reg<1, ThetaT>(k, draw, groups, stream);
        case 2:  return launch_reg<2, ThetaT>(k, draw, groups, stream);
        case 3:  return launch_reg<3, ThetaT>(k, draw, groups, stream);
        case 4:  return launch_reg<4, ThetaT>(k, draw, groups, stream);
        case 5:  return launch_reg<5, ThetaT>(k, draw, groups, stream);
        case 6:  return launch_reg<6, ThetaT>(k, draw, groups, stream);
        case 7:  return launch_reg<7, ThetaT>(k, draw, groups, stream);
        case 8:  return launch_reg<8, ThetaT>(k, draw, groups, stream);
        default: break;
    }
    if (k.n <= kTwoPassMaxN1Slot) return launch_twopass<ThetaT, 128, 128, 4, 6>(k, draw, groups, stream);
    if (k.n <= kTwoPassMaxN2Slots) return launch_twopass<ThetaT, 128, 64, 8, 4>(k, draw, groups, stream);
    if (k.n <= kTwoPassMaxN64Quads4) return launch_twopass<ThetaT, 256, 64, 4, 3>(k, draw, groups, stream);
    if (k.n <= kTwoPassMaxN64Quads8) return launch_twopass<ThetaT, 256, 64, 8, 2>(k, draw, groups, stream);
    if (k.n <= kTwoPassMaxN4Rows) return launch_twopass<ThetaT, 256, 32, 4, 3>(k, draw, groups, stream);
    if (k.n <= kTwoPassMaxN32Quads) return launch_twopass<ThetaT, 256, 32, 8, 2>(k, draw, groups, stream);
    if (k.n <= kTwoPassMaxN8Warps) return launch_twopass<ThetaT, 256, 16, 8, 2>(k, draw, groups, stream);
    return launch_twopass<ThetaT, 512, 16, 8, 1>(k, draw, groups, stream);
}

}  // namespace

// Few columns: up to two CTAs of 256 quads per SM, three quarters of one for fewer than 32 members, which a thread walks in few latencies.
// us of a draw (alone 5.7) and the means, a thread per quad / staged, one subgroup of n, quads: (24, 28 416) 6.8 / 5.7, (20, 37 888) 6.2 / 6.9,
// (32, 37 888) 8.3 / 7.3, (32, 75 776) 12.8 / 11.0, (64, 9472) 13.2 / 5.8, (128, 37 888) 35 / 17, (256, 18 944) 66 / 18, (1024, 37 888) 273 /
// 115.  Row pieces of 128 bytes for the smallest of them, where 512-byte ones leave SMs idle: (128, 4096) 5.9, of 512 bytes 6.5, (256, 4096) 8.2 / 9.5,
// (1024, 4096) 19.8 / 29.4, (64, 9472) 6.3 / 5.8, (256, 9472) 13.0 / 12.2, (1024, 9472) 37 / 41.
constexpr int64_t kMeanFewQuads = 148 * 512, kMeanFewQuadsSmall = 148 * 192, kMeanNarrowQuads = 148 * 32;
constexpr int64_t kMeanEarlyQuads = 1 << 19;       // of all members
constexpr int kMeanDirectMaxN = 16, kMeanSmallMaxN = 31;

cudaError_t launch_group_mean(const float* phi, const int32_t* perm, int W, int n, int64_t stride, int64_t P,
                              double* mean, int64_t mean_stride, cudaStream_t stream) {
    if (P <= 0 || W <= 0) return cudaSuccess;
    const int groups = W / n;
    const int64_t quads = P >> 2;
    if (groups > 65535) return cudaErrorInvalidConfiguration;
    const double inv_n = 1.0 / (double)n;
    // rows of the means are 32-byte aligned when the base is (the stride is a multiple of 64 bytes)
    const bool wide = (reinterpret_cast<uintptr_t>(mean) & 31u) == 0;
    auto launch = [&](auto kernel, int64_t quads_per_cta, auto... more) {
        const int64_t tiles = (quads + quads_per_cta - 1) / quads_per_cta + ((P & 3) != 0);
        if (tiles > 0x7fffffffll) return cudaErrorInvalidConfiguration;
        return launch_overlapped(kernel, dim3((unsigned)tiles, (unsigned)groups), kThreads, 0, stream, phi, perm, n, stride, P, mean,
                                 mean_stride, inv_n, more...);
    };
    if (n <= 4) return launch(wide ? group_mean_kernel<2, true> : group_mean_kernel<2, false>, 2 * kThreads);
    if (n > kMeanDirectMaxN && quads > 0 && quads * groups <= (n <= kMeanSmallMaxN ? kMeanFewQuadsSmall : kMeanFewQuads)) {
        const bool early = quads * W <= kMeanEarlyQuads;
        return quads * groups <= kMeanNarrowQuads ? launch(staged_mean_kernel<8>, 8, early) : launch(staged_mean_kernel<32>, 32, early);
    }
    return launch(wide ? group_mean_kernel<1, true> : group_mean_kernel<1, false>, kThreads);
}

// Drawing in the kernel saves the launch of the draw and costs every CTA the draw's 0.3 us.  It is the faster, for a call
// alone and for calls that follow each other, as long as the grid is few waves: up to 2^25 worker-parameters for
// n <= 4, whose CTAs are the larger, and up to 2^24 above.  us alone, drawn in the step / by a kernel ahead: n = 2 8.2 / 9.2
// at 2^17, 67.6 / 68.6 at 2^24, 124.9 / 126.0 at 2^25; n = 8 10.2 / 13.3 at 2^20, 61.5 / 62.5 at 2^24; n = 20 75.8 / 77.0 at 2^24.
constexpr int64_t kDrawMaxParams = 1 << 25, kDrawMaxParamsWide = 1 << 24;   // worker-parameters; n <= 4 and above

bool outer_draws(const OuterArgs& a) {
    return a.W <= 32 && a.P * a.W <= (a.n <= 4 ? kDrawMaxParams : kDrawMaxParamsWide);
}

cudaError_t launch_outer(const OuterArgs& a, cudaStream_t stream) {
    if (a.P <= 0 || a.W <= 0) return cudaSuccess;
    KArgs k;
    k.phi = a.phi; k.theta = a.theta; k.delta = a.delta; k.perm = a.perm;
    k.seed = a.seed; k.step = a.step; k.W = a.W;
    k.mean_phi = a.mean_phi; k.mean_stride = a.mean_stride;
    k.stride = a.stride; k.P = a.P; k.n = a.n;
    k.alpha = a.alpha; k.gamma = a.gamma;
    k.beta_over_n = a.beta / (float)a.n;
    k.inv_n = 1.0f / (float)a.n;
    k.n_f = (float)a.n;
    k.inv_n_d = 1.0 / (double)a.n;
    const int groups = a.W / a.n;
    if (groups > 65535) return cudaErrorInvalidConfiguration;
    return a.theta_bf16 ? dispatch<__nv_bfloat16>(k, a.draw, groups, stream) : dispatch<float>(k, a.draw, groups, stream);
}

}  // namespace nolo
