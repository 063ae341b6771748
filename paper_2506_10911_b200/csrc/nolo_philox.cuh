// Philox-4x64-10 counter-based generator (Salmon, Moraes, Dror, Shaw: "Parallel random numbers: as
// easy as 1, 2, 3", SC'11) for device code.  Integer arithmetic only.
#pragma once

#include <stdint.h>

namespace nolo {

struct Philox4 {
    uint64_t w0, w1, w2, w3;
};

// Published Philox4x64 multipliers and Weyl key increments.
constexpr uint64_t kPhiloxM0 = 0xD2E7470EE14C6C93ull;
constexpr uint64_t kPhiloxM1 = 0xCA5A826395121157ull;
constexpr uint64_t kPhiloxW0 = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kPhiloxW1 = 0xBB67AE8584CAA73Bull;

// The 128-bit product of two 64-bit numbers from four 32 x 32 -> 64-bit ones, none of whose sums overflows.
// (__umul64hi and a product for the low half together cost about half as many instructions more.)
__device__ __forceinline__ void multiply(uint64_t a, uint64_t m, uint64_t& hi, uint64_t& lo) {
    const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), m0 = (uint32_t)m, m1 = (uint32_t)(m >> 32);
    const uint64_t p0 = (uint64_t)a0 * m0;
    const uint64_t p1 = (uint64_t)a0 * m1 + (p0 >> 32);
    const uint64_t p2 = (uint64_t)a1 * m0 + (uint32_t)p1;
    hi = (uint64_t)a1 * m1 + (p1 >> 32) + (p2 >> 32);
    lo = (p2 << 32) | (uint32_t)p0;
}

__device__ __forceinline__ Philox4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                                 uint64_t k0, uint64_t k1) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t hi0, lo0, hi1, lo1;
        multiply(c0, kPhiloxM0, hi0, lo0);
        multiply(c2, kPhiloxM1, hi1, lo1);
        const uint64_t n0 = hi1 ^ c1 ^ k0;
        const uint64_t n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += kPhiloxW0; k1 += kPhiloxW1;
    }
    Philox4 o;
    o.w0 = c0; o.w1 = c1; o.w2 = c2; o.w3 = c3;
    return o;
}

// Sort key of element i of a permutation draw: counter (i, boundary, slot, domain), key (seed, step).
__device__ __forceinline__ uint64_t draw_key(uint64_t i, uint64_t boundary, uint64_t slot, uint64_t domain,
                                             uint64_t seed, uint64_t step) {
    return philox4x64_10(i, boundary, slot, domain, seed, step).w0;
}

}  // namespace nolo
