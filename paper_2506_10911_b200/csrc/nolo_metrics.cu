// Replica divergence: how far the W workers' slow weights have drifted apart (the quantity of
// Fig. 3b: the standard deviation of the model weights across the data-parallel replicas).
//
// For every parameter p the population variance of phi[0..W-1][p] across the workers is computed
// with Welford's update in float32 (stable when the replicas are close, as they are), and the
// per-parameter standard deviation and variance are summed over all parameters in float64: first
// inside each CTA, then over the CTAs by the last of them to finish, both in a fixed order, so the result
// is reproducible.  A read-only pass: 4 bytes per worker-parameter.
#include "nolo_internal.h"
#include "nolo_launch.cuh"

namespace nolo {

namespace {

constexpr int kThreads = 256;
// One column's mean and sum of squared deviations over some workers.
struct Moments {
    float mean, m2;
    __device__ __forceinline__ void push(float x, float inv_k) {
        const float d = x - mean;
        mean += d * inv_k;
        m2 += d * (x - mean);
    }
    // this one of n values, o of the m that follow; share = m / (n + m), weight = n * share
    // (Chan, Golub, LeVeque: updating formulae, 1979)
    __device__ __forceinline__ void join(const Moments& o, float share, float weight) {
        const float d = o.mean - mean;
        mean += d * share;
        m2 += o.m2 + d * (weight * d);         // (d * d may overflow where this does not)
    }
    static __device__ __forceinline__ Moments of_pair(float a, float b) {
        const float d = b - a, half = 0.5f * d;
        return {a + half, half * d};
    }
};

// Moments of `rows` (1 to 4) values at once; those that are missing may be anything.  A part joins its workers by fours: a quarter of
// the roundings in a row, whose errors do not cancel, and a quarter of the dependent operations of one worker after the other.  Relative
// error of the returned mean against 64 bits, sixteen parts with single workers / four with fours (with single workers):
// (64, 100 000) -7e-10 / 9e-10 (-8e-9), (32, 50 000) 0 / 4e-10 (-7e-9); at the same number of parts (1000, 100 000) 2e-8 / 4e-9.
struct Quad {
    bool second, third, fourth;
    float share, weight;
    __device__ __forceinline__ explicit Quad(int rows)
        : second(rows > 1), third(rows > 2), fourth(rows > 3), share(fourth ? 0.5f : third ? 1.f / 3.f : 0.f),
          weight(fourth ? 1.f : third ? 2.f / 3.f : 0.f) {}
    __device__ __forceinline__ Moments moments(float a, float b, float c, float d) const {
        Moments m = Moments::of_pair(a, second ? b : a);
        const float x = third ? c : a;
        m.join(Moments::of_pair(x, fourth ? d : x), share, weight);
        return m;
    }
};

__device__ __forceinline__ double2 warp_sum(double2 v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        v.x += __shfl_down_sync(0xffffffffu, v.x, off);
        v.y += __shfl_down_sync(0xffffffffu, v.y, off);
    }
    return v;
}

// The sum over the CTA, in a fixed order, in thread 0.  Contains two barriers.
template <int THREADS>
__device__ __forceinline__ double2 cta_sum(double2 v) {
    __shared__ double2 warp_part[THREADS / 32];
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) warp_part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < THREADS / 32; ++w) { v.x += warp_part[w].x; v.y += warp_part[w].y; }
    return v;
}

// The result from the CTAs' sums, by one CTA in a fixed order.
template <int THREADS>
__device__ __forceinline__ void finish(const double2* partial, int64_t count, int64_t P, double* out) {
    double2 total = make_double2(0.0, 0.0);
#pragma unroll 8
    for (int64_t i = threadIdx.x; i < count; i += THREADS) {
        const double2 v = __ldcg(partial + i);
        total.x += v.x;
        total.y += v.y;
    }
    total = cta_sum<THREADS>(total);
    if (threadIdx.x == 0) {
        out[0] = total.x / (double)P;            // mean over parameters of the across-worker std
        out[1] = sqrt(total.y / (double)P);      // root of the mean across-worker variance
    }
}

// ITEMS quads (4 consecutive columns) per thread; the CTA's threads form PARTS groups that share out the
// workers of the same columns and join their moments in shared memory, for states with few columns, whose
// CTAs would not fill the chip and whose threads would walk the workers one after the other.  FUSED: the
// last CTA to leave its sums adds them up; `arrived` counts them and is zero before and after.
template <int ITEMS, int PARTS, bool FUSED>
__global__ void __launch_bounds__(kThreads, ITEMS == 4 || PARTS > 1 ? 4 : 1)
divergence_kernel(const float* phi, int W, int64_t stride, int64_t P, double2* partial, unsigned* arrived,
                  double* out) {
    constexpr int COLS = kThreads / PARTS;             // threads of one part
    constexpr int ROWS = ITEMS > 1 ? 1 : PARTS > 1 ? 4 : 8;   // rows whose loads are written before the first use
    wait_for_predecessors();
    let_successor_start();
    const int part = threadIdx.x / COLS, lane = threadIdx.x % COLS;
    const int64_t quads = (P + 3) >> 2;                // the last may be partial: rows are padded to multiples of 8
    const int64_t q0 = (int64_t)blockIdx.x * (COLS * ITEMS) + lane;
    const int w0 = (int)((int64_t)W * part / PARTS), w1 = (int)((int64_t)W * (part + 1) / PARTS);

    Moments acc[ITEMS][4];
    bool ok[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
        ok[it] = q0 + it * COLS < quads;
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[it][e] = {0.f, 0.f};
    }
#pragma unroll (ITEMS == 1 ? 1 : 4)
    for (int w = w0; w < w1; w += ROWS) {
        float4 x[ROWS][ITEMS];
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const float4* row = reinterpret_cast<const float4*>(phi + (int64_t)(w + i) * stride);
#pragma unroll
            for (int it = 0; it < ITEMS; ++it)
                if (ok[it] && w + i < w1) x[i][it] = __ldcs(row + q0 + it * COLS);
        }
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            if constexpr (PARTS > 1) {
                static_assert(PARTS == 1 || ROWS == 4, "four rows at once");
                if (i > 0 || !ok[0]) break;
                const int n = w - w0, rows = w1 - w < 4 ? w1 - w : 4;
                const Quad quad(rows);
                const float share = (float)rows * __frcp_rn((float)(n + rows)), weight = (float)n * share;
                acc[0][0].join(quad.moments(x[0][0].x, x[1][0].x, x[2][0].x, x[3][0].x), share, weight);
                acc[0][1].join(quad.moments(x[0][0].y, x[1][0].y, x[2][0].y, x[3][0].y), share, weight);
                acc[0][2].join(quad.moments(x[0][0].z, x[1][0].z, x[2][0].z, x[3][0].z), share, weight);
                acc[0][3].join(quad.moments(x[0][0].w, x[1][0].w, x[2][0].w, x[3][0].w), share, weight);
            } else {
                const float inv_k = __frcp_rn((float)(w + i - w0 + 1));
#pragma unroll
                for (int it = 0; it < ITEMS; ++it) {
                    if (ok[it] && w + i < w1) {
                        acc[it][0].push(x[i][it].x, inv_k); acc[it][1].push(x[i][it].y, inv_k);
                        acc[it][2].push(x[i][it].z, inv_k); acc[it][3].push(x[i][it].w, inv_k);
                    }
                }
            }
        }
    }
    if constexpr (PARTS > 1) {
        static_assert(ITEMS == 1, "parts share one quad per thread");
        __shared__ Moments shared[kThreads][4];
        for (int half = PARTS / 2; half >= 1; half /= 2) {     // part p takes over the workers of part p + half
            __syncthreads();
#pragma unroll
            for (int e = 0; e < 4; ++e) shared[threadIdx.x][e] = acc[0][e];
            __syncthreads();
            if (part < half) {
                // workers held by parts p, p + 2 half, p + 4 half, ... and by p + half, p + 3 half, ...
                int n = 0, m = 0;
                for (int p = part; p < PARTS; p += 2 * half) {
                    n += (int)((int64_t)W * (p + 1) / PARTS) - (int)((int64_t)W * p / PARTS);
                    m += (int)((int64_t)W * (p + half + 1) / PARTS) - (int)((int64_t)W * (p + half) / PARTS);
                }
                const float share = (float)m / (float)(n + m), weight = (float)n * share;
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[0][e].join(shared[threadIdx.x + half * COLS][e], share, weight);
            }
        }
    }
    double2 sum = make_double2(0.0, 0.0);              // of the standard deviations, of the variances
    if (part == 0) {
        const float inv_W = 1.0f / (float)W;
        auto variance = [&](const Moments& m) { return PARTS > 1 ? m.m2 / (float)W : m.m2 * inv_W; };
        const int64_t full = P >> 2;
        const int ragged = (int)(P & 3);
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) {
            if (!ok[it]) continue;
            float4 v = make_float4(variance(acc[it][0]), variance(acc[it][1]), variance(acc[it][2]), variance(acc[it][3]));
            const int64_t q = q0 + it * COLS;
            if (q == full) {                           // the partial quad
                if (ragged < 2) v.y = 0.f;
                if (ragged < 3) v.z = 0.f;
                v.w = 0.f;
            }
            sum.y += (double)v.x + (double)v.y + (double)v.z + (double)v.w;
            sum.x += (double)sqrtf(v.x) + (double)sqrtf(v.y) + (double)sqrtf(v.z) + (double)sqrtf(v.w);
        }
    }
    sum = cta_sum<kThreads>(sum);
    if (threadIdx.x == 0) partial[blockIdx.x] = sum;
    if constexpr (FUSED) {
        __shared__ bool last;
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(arrived, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        finish<kThreads>(partial, gridDim.x, P, out);
        if (threadIdx.x == 0) *arrived = 0;
    }
}

__global__ void __launch_bounds__(1024)
divergence_finish_kernel(const double2* partial, int64_t count, int64_t P, double* out) {
    wait_for_predecessors();
    let_successor_start();
    finish<1024>(partial, count, P, out);
}

struct Shape {
    int items, parts;
    int64_t ctas(int64_t P) const {
        const int64_t quads = (P + 3) >> 2, per_cta = (int64_t)(kThreads / parts) * items;
        return (quads + per_cta - 1) / per_cta;
    }
};

// Four quads per thread and a second kernel for the sums where that leaves enough CTAs, else one quad and one
// kernel, in parts while there are few CTAs and every part keeps a worker.  Enough are eight per
// SM, so that the last, part-filled wave of four weighs little ((128, 3e6) 247 us with one quad, 301 with four, which
// are 1.2 waves); with few workers a CTA is soon done and their number weighs more, the one counter that they all
// add to included: three per SM ((1, 2^22) 45 us with one quad, 29 with four, (12, 3e6) 57 / 53, (16, 3e6) 58 / 62).
// Few are less than four per SM; for further parts than four less than one, unless a part has 64 workers and more to walk, for the
// counter makes more of them dearer again.  us, with four per SM for few throughout / now: (16, 100 000) 26.2 / 15.3,
// (64, 100 000) 29.4 / 18.9, (32, 50 000) 20.3 / 15.8, (40, 60 000) 21.7 / 15.7, (1024, 24 414) 41.8 / 39.6; unparted (1024, 1000) 331, now 21.
// Four quads want four CTAs of 64 registers per SM: at 66
// registers, three CTAs, (16, 2^26) measured 675 us instead of 622.  (Sums of each thread in float32 pairs instead of float64,
// to save its conversions, measured slower: (2, 2e8) 330 -> 360.)
constexpr int64_t kManyCtas = 148 * 8, kManyShortCtas = 148 * 3, kFewCtas = 148 * 4;
constexpr int kShortMaxW = 12;
Shape shape_for(int W, int64_t P) {
    Shape s = {4, 1};
    if (s.ctas(P) >= (W <= kShortMaxW ? kManyShortCtas : kManyCtas)) return s;
    s.items = 1;
    while (s.parts < 32 && W >= 4 * s.parts && s.ctas(P) < (s.parts == 1 || W >= 64 * s.parts ? kFewCtas : kFewCtas / 4))
        s.parts *= s.parts == 16 ? 2 : 4;
    return s;
}

}  // namespace

int64_t divergence_partials(int W, int64_t P) { return shape_for(W, P).ctas(P); }

cudaError_t launch_divergence(const float* phi, int W, int64_t stride, int64_t P, void* partials, unsigned* arrived,
                              double* out2, cudaStream_t stream, int* launches) {
    const Shape s = shape_for(W, P);
    const int64_t ctas = s.ctas(P);
    if (ctas > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    double2* partial = static_cast<double2*>(partials);
    auto launch = [&](auto kernel) {
        return launch_overlapped(kernel, dim3((unsigned)ctas), kThreads, 0, stream, phi, W, stride, P, partial, arrived, out2);
    };
    *launches = s.items == 4 ? 2 : 1;
    if (s.items == 4) {
        const cudaError_t e = launch(divergence_kernel<4, 1, false>);
        if (e != cudaSuccess) return e;
        return launch_overlapped(divergence_finish_kernel, dim3(1), 1024, 0, stream, static_cast<const double2*>(partial), ctas,
                                 P, out2);
    }
    switch (s.parts) {
        case 1: return launch(divergence_kernel<1, 1, true>);
        case 4: return launch(divergence_kernel<1, 4, true>);
        case 16: return launch(divergence_kernel<1, 16, true>);
        default: return launch(divergence_kernel<1, 32, true>);
    }
}

}  // namespace nolo
