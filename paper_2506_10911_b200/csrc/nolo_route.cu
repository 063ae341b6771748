// Random pipeline routing (Section 3.1, Algorithm 1) as a permutation gather of micro-batch
// activations between the replicas of consecutive stages.  A pure copy: every byte is read once
// and written once, 128 or 256 bits per access, streaming cache policy.
//
//   forward :  out[b][r][k][:] = in[b][table[b][k][r]][k][:]
//   backward:  out[b][table[b][k][r]][k][:] = in[b][r][k][:]     (same path, reversed)
//
// Bound by DRAM for all but the smallest calls, which are bound by latency: kernels are launched while
// their predecessor runs, and up to 32 replicas draw their permutation inside the copy.
#include "nolo_draw.cuh"
#include "nolo_internal.h"
#include "nolo_launch.cuh"
#include "nolo_shifted.h"

namespace nolo {

namespace {

struct CopyArgs {
    const unsigned char* in;
    unsigned char* out;
    int32_t* table;           // [B][K][R]
    int B, R, K;
    int64_t bytes;            // of one block, or of the part of it that is copied
    int64_t stride;           // bytes between blocks
    const unsigned char* in_end;
    int backward;
    // kernels that draw the table themselves (DRAW)
    uint64_t seed, step;
    int first_boundary, per_microbatch;
};

// Asks for the whole 16-byte vectors of this CTA's tile of an input block.
template <int TILE>
__device__ __forceinline__ void prefetch_tile(const CopyArgs& a, int64_t block) {
    const int64_t first = (int64_t)blockIdx.x * TILE, left = a.bytes - first;
    const uintptr_t from = reinterpret_cast<uintptr_t>(a.in + block * a.stride + first);
    const uintptr_t lo = (from + 15) & ~uintptr_t(15), hi = (from + (left < TILE ? left : TILE)) & ~uintptr_t(15);
    prefetch_to_l2(reinterpret_cast<const void*>(lo), (int64_t)(hi - lo));
}

// The replica of the other side for slot k of replica r at boundary b.  DRAW: drawn by the first warp
// before the kernels ahead are waited for; one CTA per permutation writes the table.  The lane that finds the
// replica has the tile brought to L2 while the kernels ahead end (a forward and a backward call of 67 MB 39.8 us, 43.5
// without).
template <bool DRAW, int TILE>
__device__ __forceinline__ int peer_of(const CopyArgs& a, int b, int r, int k) {
    int32_t* row = a.table + ((int64_t)b * a.K + k) * a.R;
    if constexpr (!DRAW) {
        return load_written(row + r);
    } else {
        __shared__ int peer;
        int rank = 0;
        if (threadIdx.x < 32) {
            rank = rank_by_warp(a.R, a.first_boundary + b, a.per_microbatch ? k : 0, kDomainRoute, a.seed, a.step);
            if (rank == r) {
                peer = threadIdx.x;
                prefetch_tile<TILE>(a, ((int64_t)b * a.R + (a.backward ? r : (int)threadIdx.x)) * a.K + k);
            }
        }
        wait_for_predecessors();
        let_successor_start();      // not before: it may count on all that went before this kernel
        if (r == 0 && blockIdx.x == 0 && (int)threadIdx.x < a.R) row[rank] = threadIdx.x;
        __syncthreads();
        const int p = peer;
        __syncthreads();      // before the next draw of this CTA
        return p;
    }
}

// A 256-bit vector, moved by one access.
struct __align__(32) Wide { uint4 a, b; };
__device__ __forceinline__ Wide load_stream(const Wide* p) {
    Wide v;
    asm volatile("ld.global.cs.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v.a.x), "=r"(v.a.y), "=r"(v.a.z), "=r"(v.a.w), "=r"(v.b.x), "=r"(v.b.y), "=r"(v.b.z), "=r"(v.b.w)
                 : "l"(p));
    return v;
}
__device__ __forceinline__ void store_stream(Wide* p, const Wide& v) {
    asm volatile("st.global.cs.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"r"(v.a.x), "r"(v.a.y), "r"(v.a.z), "r"(v.a.w),
                 "r"(v.b.x), "r"(v.b.y), "r"(v.b.z), "r"(v.b.w), "l"(p)
                 : "memory");
}
__device__ __forceinline__ uint4 load_stream(const uint4* p) { return __ldcs(p); }
__device__ __forceinline__ void store_stream(uint4* p, const uint4& v) { __stcs(p, v); }

// A tile of THREADS x N vectors V of one block, block and vectors aligned to V.
template <typename V, int THREADS, int N>
__device__ __forceinline__ void copy_tile(const unsigned char* src, unsigned char* dst, int64_t bytes) {
    const int64_t vecs = bytes / sizeof(V), v0 = (int64_t)blockIdx.x * (THREADS * N) + threadIdx.x;
    V v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int64_t x = v0 + (int64_t)i * THREADS;
        if (x < vecs) v[i] = load_stream(reinterpret_cast<const V*>(src) + x);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const int64_t x = v0 + (int64_t)i * THREADS;
        if (x < vecs) store_stream(reinterpret_cast<V*>(dst) + x, v[i]);
    }
}

// Bytes s .. s+15 of two neighbouring 16-byte vectors.
__device__ __forceinline__ uint4 shifted(const uint4& x, const uint4& y, int s) {
    const uint32_t w[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    const int words = s >> 2, bits = (s & 3) * 8;
    uint32_t v[5];
#pragma unroll
    for (int i = 0; i < 5; ++i)
        v[i] = words == 0 ? w[i] : words == 1 ? w[i + 1] : words == 2 ? w[i + 2] : w[i + 3];
    return make_uint4(__funnelshift_r(v[0], v[1], bits), __funnelshift_r(v[1], v[2], bits), __funnelshift_r(v[2], v[3], bits),
                      __funnelshift_r(v[3], v[4], bits));
}

// The same for blocks of elements T that begin anywhere (at a multiple of sizeof(T)), the source at
// another offset from a 16-byte boundary than the destination: each 16-byte vector of the destination is put
// together from the two aligned source vectors it straddles (see ShiftedSpan).  A warp has N x 32 consecutive vectors,
// so that the second one comes from the next lane by shuffle (holding both in registers measured 10-20 % slower:
// fewer bytes in flight).
template <typename T, int THREADS, int N>
__device__ __forceinline__ void copy_tile_shifted(const unsigned char* src, unsigned char* dst, int64_t bytes,
                                                  const unsigned char* in_end) {
    static_assert(THREADS * sizeof(T) >= kLine + 32, "one element per thread at the ends");
    const ShiftedSpan p = shifted_span(src, dst, bytes, in_end);
    const uint4* from = reinterpret_cast<const uint4*>(p.from);
    const int lane = threadIdx.x & 31;
    const int64_t v0 = ((int64_t)blockIdx.x * (THREADS / 32) + (threadIdx.x >> 5)) * (32 * N) + lane;
    uint4 v[N + 1];
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (v0 + 32 * i < p.loads) v[i] = __ldcs(from + v0 + 32 * i);
    if (lane == 0 && v0 + 32 * N < p.loads) v[N] = __ldcs(from + v0 + 32 * N);
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const uint4 give = lane == 0 ? v[i + 1] : v[i];
        uint4 next;
        next.x = __shfl_sync(0xffffffffu, give.x, (lane + 1) & 31);
        next.y = __shfl_sync(0xffffffffu, give.y, (lane + 1) & 31);
        next.z = __shfl_sync(0xffffffffu, give.z, (lane + 1) & 31);
        next.w = __shfl_sync(0xffffffffu, give.w, (lane + 1) & 31);
        if (v0 + 32 * i < p.vecs) __stcs(reinterpret_cast<uint4*>(dst + p.head) + v0 + 32 * i, shifted(v[i], next, p.shift));
    }
    if (blockIdx.x == 0 && threadIdx.x < (kLine + 32) / sizeof(T)) {
        const int e = threadIdx.x * sizeof(T);
        const int64_t at = e < kLine ? e : p.head + 16 * p.vecs + (e - kLine);
        if (e < kLine ? at < p.head : at < bytes) *reinterpret_cast<T*>(dst + at) = *reinterpret_cast<const T*>(src + at);
    }
}

// One tile of one block per CTA.  V: Wide or uint4 for blocks that are a multiple of it, else the element.
template <typename V, int THREADS, int N, bool DRAW>
__global__ void __launch_bounds__(THREADS)
route_copy_kernel(const CopyArgs a) {
    if constexpr (!DRAW) {
        wait_for_predecessors();
        let_successor_start();
    }
    constexpr int TILE = THREADS * N * (sizeof(V) < 16 ? 16 : (int)sizeof(V));
    for (int b = blockIdx.z; b < a.B; b += gridDim.z) {
        for (int rk = blockIdx.y; rk < a.R * a.K; rk += gridDim.y) {
            const int r = rk / a.K, k = rk - r * a.K;
            const int peer = peer_of<DRAW, TILE>(a, b, r, k);
            const int64_t here = ((int64_t)b * a.R + r) * a.K + k, there = ((int64_t)b * a.R + peer) * a.K + k;
            const unsigned char* src = a.in + (a.backward ? here : there) * a.stride;
            unsigned char* dst = a.out + (a.backward ? there : here) * a.stride;
            if constexpr (sizeof(V) >= 16)
                copy_tile<V, THREADS, N>(src, dst, a.bytes);
            else
                copy_tile_shifted<V, THREADS, N>(src, dst, a.bytes, a.in_end);
        }
    }
}

// Plain device-to-device copy, a one-shot grid of 128-bit streaming loads and stores like the
// routing copy: the yardstick the other kernels are compared with.  Two vectors per thread is the
// fastest plain copy found on B200 (6.97 TB/s against 6.90 with four and 6.87 with eight; 256-bit
// loads and stores gave the same 6.9-7.0).
constexpr int kProbeThreads = 256;
constexpr int kProbeVecPerThread = 2;
constexpr int kProbeTileVecs = kProbeThreads * kProbeVecPerThread;

__global__ void __launch_bounds__(kProbeThreads)
copy_probe_kernel(const uint4* in, uint4* out, int64_t vecs) {
    const int64_t v0 = (int64_t)blockIdx.x * kProbeTileVecs + threadIdx.x;
    uint4 v[kProbeVecPerThread];
#pragma unroll
    for (int i = 0; i < kProbeVecPerThread; ++i) {
        const int64_t x = v0 + (int64_t)i * kProbeThreads;
        if (x < vecs) v[i] = __ldcs(in + x);
    }
#pragma unroll
    for (int i = 0; i < kProbeVecPerThread; ++i) {
        const int64_t x = v0 + (int64_t)i * kProbeThreads;
        if (x < vecs) __stcs(out + x, v[i]);
    }
}

}  // namespace

cudaError_t launch_copy_probe(const void* in, void* out, int64_t bytes, cudaStream_t stream) {
    const int64_t vecs = bytes / 16;
    const int64_t tiles = (vecs + kProbeTileVecs - 1) / kProbeTileVecs;
    if (tiles <= 0) return cudaSuccess;
    if (tiles > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    copy_probe_kernel<<<(unsigned)tiles, kProbeThreads, 0, stream>>>(static_cast<const uint4*>(in),
                                                                static_cast<uint4*>(out), vecs);
    return cudaGetLastError();
}

// Drawing in the copy saves the launch of the draw, lets the copy ask for its data ahead of its wait, and costs every
// CTA the draw, 0.3 us and the more the more replicas there are.  It is the faster, for a call alone and for calls that follow
// each other, as long as the grid is few waves, and for few replicas long after if the CTAs' tiles are filled to four fifths.  us alone,
// drawn in the copy / by a kernel ahead:
// 6 MB 10.2 / 11.3, 134 MB (multiples of 32 bytes) 47.1 / 48.1, 67 MB of other blocks 28.7 / 29.7.  There and back, 8 replicas:
// 140 MB a way 85.8 / 90.5, 420 MB 240 / 245, 944 MB 536 / 543, at odd offsets 73 MB 46.2 / 50.3, 94 MB 59.2 / 62.5, 126 MB 79.1 /
// 80.4; 32 replicas: 420 MB 255 / 245, at odd offsets 84 MB 58.9 / 56.8.  300 MB in blocks of 2 KB 611 / 246, 8 KB (half a tile) 220 /
// 189, 16 KB 175 / 184, 18 KB (two tiles) 199 / 184, 24 KB 180 / 183, 32 KB 175 / 182; 97 MB at odd offsets, 8 KB 87.9 / 80.6, 12 KB 71.4 / 70.4,
// 16 KB 64.4 / 67.1, 33 KB (three tiles) 69.9 / 67.6, 66 KB (five) 64.4 / 65.3.  The lines of 1 GB and 100 MB are where it was measured
// to; the gain beyond is a percent.
constexpr int kFewReplicas = 8;
constexpr int64_t kDrawMaxBytes = 64ll << 20, kDrawMaxBytesFew = 100ll << 20;
constexpr int64_t kDrawMaxBytesWide = 128ll << 20, kDrawMaxBytesWideFew = 1024ll << 20;   // for multiples of 32 bytes
constexpr int64_t kDrawTile = 16 << 10;           // bytes per CTA of every copy that draws

bool route_draws(const RouteArgs& a) {
    const int64_t block = a.E * a.elem_size, bytes = (int64_t)a.B * a.R * a.K * block;
    const int64_t tiles = (block + kDrawTile - 1) / kDrawTile;
    const bool wide = block % 32 == 0, few = a.R <= kFewReplicas && 5 * block >= 4 * tiles * kDrawTile;
    const int64_t most = wide ? (few ? kDrawMaxBytesWideFew : kDrawMaxBytesWide) : (few ? kDrawMaxBytesFew : kDrawMaxBytes);
    return a.R <= 32 && bytes <= most;
}

template <typename V, int THREADS, int N>
cudaError_t launch_shape(const CopyArgs& c, bool draw, cudaStream_t stream) {
    constexpr int64_t tile = (int64_t)THREADS * N * (sizeof(V) < 16 ? 16 : sizeof(V));
    const int64_t tiles = (c.bytes + tile - 1) / tile, rk = (int64_t)c.R * c.K;
    if (tiles > 0x7fffffffll) return cudaErrorInvalidConfiguration;
    if (draw && tile != kDrawTile) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)tiles, (unsigned)(rk < 65535 ? rk : 65535), (unsigned)(c.B < 65535 ? c.B : 65535));
    return launch_overlapped(draw ? route_copy_kernel<V, THREADS, N, true> : route_copy_kernel<V, THREADS, N, false>, grid,
                             THREADS, 0, stream, c);
}

// One CTA per tile: a one-shot grid streams through memory in address order, about 10 % faster on B200 than a resident
// grid striding over the tiles (the kernel loops only where a grid dimension ends).  CTA shapes: the largest that keeps
// its rate on a device under its power cap too, where shapes of 512 and more threads lost 2-3 % (96 blocks of
// 64 MB there and back: 384 threads x 1 vector of 32 bytes 3676 us, 256 x 4 of 16 bytes 3724); copies that draw want few
// CTAs; blocks at any offset many vectors per thread, because what a CTA does before its loads is a chain of several
// hundred cycles (96 blocks of 4 MB, bfloat16: 128 x 8 6780 GB/s, 256 x 1 2910, one element per access 2180).
cudaError_t launch_route(const RouteArgs& a, cudaStream_t stream) {
    CopyArgs c;
    const int64_t skip = a.first_element * a.elem_size;
    c.in = static_cast<const unsigned char*>(a.in) + skip;
    c.out = static_cast<unsigned char*>(a.out) + skip;
    c.table = a.table;
    c.B = a.B; c.R = a.R; c.K = a.K;
    c.bytes = (a.elements > 0 ? a.elements : a.E) * a.elem_size;
    c.stride = a.E * a.elem_size;
    c.in_end = static_cast<const unsigned char*>(a.in) + (int64_t)a.B * a.R * a.K * c.stride;
    c.backward = a.backward;
    c.seed = a.seed; c.step = a.step;
    c.first_boundary = a.first_boundary; c.per_microbatch = a.per_microbatch;
    if (a.B <= 0 || a.R <= 0 || a.K <= 0 || c.bytes <= 0) return cudaSuccess;
    const int64_t aligned = c.bytes | c.stride | (int64_t)reinterpret_cast<uintptr_t>(c.in) | (int64_t)reinterpret_cast<uintptr_t>(c.out);
    const bool wide = aligned % 32 == 0;
    if (wide) return a.draw ? launch_shape<Wide, 256, 2>(c, true, stream) : launch_shape<Wide, 384, 1>(c, false, stream);
    if (aligned % 16 == 0) return a.draw ? launch_shape<uint4, 256, 4>(c, true, stream) : launch_shape<uint4, 256, 2>(c, false, stream);
    return a.elem_size == 4 ? launch_shape<uint32_t, 128, 8>(c, a.draw, stream) : launch_shape<uint16_t, 128, 8>(c, a.draw, stream);
}

}  // namespace nolo
