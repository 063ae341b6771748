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

// Rounds FROM .. 9 on the counter c, with the key of round 0.
template <int FROM>
__device__ __forceinline__ Philox4 philox_rounds(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3, uint64_t k0, uint64_t k1) {
    k0 += FROM * kPhiloxW0;
    k1 += FROM * kPhiloxW1;
#pragma unroll
    for (int r = FROM; r < 10; ++r) {
        // (the products spelled out in 32-bit ones, in carry chains or in 64-bit sums, measured 10-20 % slower)
        const uint64_t hi0 = __umul64hi(kPhiloxM0, c0), lo0 = kPhiloxM0 * c0;
        const uint64_t hi1 = __umul64hi(kPhiloxM1, c2), lo1 = kPhiloxM1 * c2;
        const uint64_t n0 = hi1 ^ c1 ^ k0;
        const uint64_t n2 = hi0 ^ c3 ^ k1;
        c0 = n0; c1 = lo1; c2 = n2; c3 = lo0;
        k0 += kPhiloxW0; k1 += kPhiloxW1;
    }
    Philox4 o;
    o.w0 = c0; o.w1 = c1; o.w2 = c2; o.w3 = c3;
    return o;
}

__device__ __forceinline__ Philox4 philox4x64_10(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                                 uint64_t k0, uint64_t k1) {
    return philox_rounds<0>(c0, c1, c2, c3, k0, k1);
}

// The first three rounds for many counters (c0, c1, c2, c3) that share c2 and c3: five of their six products
// depend on only one of c0 and c1.  A block from its two parts takes 15 products instead of 20.
struct PhiloxOfC0 { uint64_t a, b, c, d; };
struct PhiloxOfC1 { uint64_t hi, lo; };

__device__ __forceinline__ PhiloxOfC0 philox_of_c0(uint64_t c0, uint64_t c2, uint64_t c3, uint64_t k0, uint64_t k1) {
    const uint64_t x1 = kPhiloxM1 * c2;
    const uint64_t x2 = __umul64hi(kPhiloxM0, c0) ^ c3 ^ k1, x3 = kPhiloxM0 * c0;
    const uint64_t y0 = __umul64hi(kPhiloxM1, x2) ^ x1 ^ (k0 + kPhiloxW0), y1 = kPhiloxM1 * x2;
    PhiloxOfC0 p;
    p.a = x3 ^ (k1 + kPhiloxW1);
    p.b = y1 ^ (k0 + 2 * kPhiloxW0);
    p.c = __umul64hi(kPhiloxM0, y0) ^ (k1 + 2 * kPhiloxW1);
    p.d = kPhiloxM0 * y0;
    return p;
}
__device__ __forceinline__ PhiloxOfC1 philox_of_c1(uint64_t c1, uint64_t c2, uint64_t k0) {
    const uint64_t x0 = __umul64hi(kPhiloxM1, c2) ^ c1 ^ k0;
    PhiloxOfC1 p;
    p.hi = __umul64hi(kPhiloxM0, x0);
    p.lo = kPhiloxM0 * x0;
    return p;
}
__device__ __forceinline__ Philox4 philox_join(const PhiloxOfC0& p, const PhiloxOfC1& q, uint64_t k0, uint64_t k1) {
    const uint64_t y2 = q.hi ^ p.a;
    return philox_rounds<3>(__umul64hi(kPhiloxM1, y2) ^ p.b, kPhiloxM1 * y2, p.c ^ q.lo, p.d, k0, k1);
}

// Sort key of element i of a permutation draw: counter (i, boundary, slot, domain), key (seed, step).
__device__ __forceinline__ uint64_t draw_key(uint64_t i, uint64_t boundary, uint64_t slot, uint64_t domain,
                                             uint64_t seed, uint64_t step) {
    return philox4x64_10(i, boundary, slot, domain, seed, step).w0;
}

}  // namespace nolo
