// Log-normal times from Philox blocks in float64, the inner loop of the latency simulations.
//
// Words -> u = ((x >> 11) + 0.5) 2^-53; Box-Muller on the word pairs (0,1) and (2,3), r = sqrt(-2 ln u_a),
// gives the normals [r01 cos, r01 sin, r23 cos, r23 sin] of the angle 2 pi u_b; t = exp(mu + sigma z).
//
// The logarithm, sine and cosine and exponential are table-driven in the manner of P. T. P. Tang (ACM TOMS 15, 1989,
// "Table-driven implementation of the exponential function in IEEE floating-point arithmetic", and TOMS 16, 1990, for the
// logarithm): a table in shared memory takes the leading bits, a short polynomial the rest.  Two arrangements are those of
// the log and exp of Arm's optimized-routines: the logarithm's intervals of equal high word from 0.6875 on, found and reduced by
// subtraction of integers, with a reciprocal of 1 next to 1; and powers stored with their index taken off the high word, so that one
// addition of the shifted exponent puts either right.  The tables' values are computed from their definitions.  The arguments are confined
// (u in (0, 1], angles as integers, exponents checked once on the host), so no special case is left in the loop, the
// angle is reduced in integers and the factors 2, pi, sigma, e^mu and 2048 / ln 2 are folded into tables and constants.
//
// Bound by the dispatch of 32- and 64-bit operands, to which the float64 operations (19 to 20 per time) and Philox's
// products contribute alike: an instruction less of any kind shows.  Intervals of 2^-9 (logarithm), entries of 2 pi / 512 and
// 2^(1 / 2048) (33 KB in all) need 39 float64 operations per pair of times, those of 128, 256 and 256 entries (9 KB) needed
// 48: 380 -> 317 thread-instructions per four times in the straggler simulation, and errors no larger (root mean square
// 1.28e-16 -> 1.18e-16 at sigma = 1, 4.9e-16 -> 2.6e-16 at mu = -3, sigma = 2.5).
#pragma once

#include <stdint.h>

#include "nolo_philox.cuh"

namespace nolo {

namespace {

// c near the reciprocal of the middle of group i of the logarithm's intervals, and ln c in two parts
__device__ const double kLogGroup[16][3] = {
    {0x1.6c00000000000p+0, 0x1.686c81e9b14afp-2, -0x1.ddea0f7f58e3dp-57},
    {0x1.5d00000000000p+0, 0x1.3d54fa5c1f710p-2, -0x1.e3265c6a1c98dp-56},
    {0x1.4e00000000000p+0, 0x1.1058bf9ae4ad5p-2, 0x1.89fa0ab4cb31dp-58},
    {0x1.4100000000000p+0, 0x1.cf6354e09c5dcp-3, 0x1.239a07d55b695p-57},
    {0x1.3500000000000p+0, 0x1.815c0a14357ebp-3, -0x1.4be48073a0564p-58},
    {0x1.2a00000000000p+0, 0x1.371fc201e8f74p-3, 0x1.de6cb62af18a0p-58},
    {0x1.1f00000000000p+0, 0x1.d4313d66cb35dp-4, 0x1.790dd951d90fap-58},
    {0x1.1600000000000p+0, 0x1.51b073f06183fp-4, 0x1.a49e39a1a8be4p-58},
    {0x1.0d00000000000p+0, 0x1.95c830ec8e3ebp-5, 0x1.f5a0e80520bf2p-59},
    {0x1.0400000000000p+0, 0x1.fc0a8b0fc03e4p-7, -0x1.83092c59642a1p-62},
    {0x1.f000000000000p-1, -0x1.0415d89e74444p-5, -0x1.c05cf1d753622p-59},
    {0x1.d400000000000p-1, -0x1.700d30aeac0e1p-4, 0x1.72566212cdd05p-61},
    {0x1.ba00000000000p-1, -0x1.2d1610c86813ap-3, 0x1.499a3f25af95fp-58},
    {0x1.a400000000000p-1, -0x1.95a5adcf7017fp-3, -0x1.142c507fb7a3dp-58},
    {0x1.9000000000000p-1, -0x1.f991c6cb3b379p-3, -0x1.f665066f980a2p-57},
    {0x1.7e00000000000p-1, -0x1.2bef07cdc9354p-2, 0x1.82dad7fd86088p-56},
};
// 2^(i / 32) in two parts
__device__ const double2 kExpCoarse[32] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54},
};
// 2^(i / 2048) in two parts
__device__ const double2 kExpFine[64] = {
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.00162f3904052p+0, -0x1.7b5d0d58ea8f4p-58},
    {0x1.002c605e2e8cfp+0, -0x1.d7c96f201bb2fp-55}, {0x1.0042936faa3d8p+0, -0x1.0484245243777p-55},
    {0x1.0058c86da1c0ap+0, -0x1.5e00e62d6b30dp-56}, {0x1.006eff583fc3dp+0, -0x1.4acf197a00142p-54},
    {0x1.0085382faef83p+0, 0x1.da93f90835f75p-56}, {0x1.009b72f41a12bp+0, 0x1.86364f8fbe8f8p-54},
    {0x1.00b1afa5abcbfp+0, -0x1.4f6b2a7609f71p-55}, {0x1.00c7ee448ee02p+0, 0x1.4362ca5bc26f1p-56},
    {0x1.00de2ed0ee0f5p+0, -0x1.406ac4e81a645p-57}, {0x1.00f4714af41d3p+0, -0x1.91b2060859321p-54},
    {0x1.010ab5b2cbd11p+0, 0x1.c1d0660524e08p-54}, {0x1.0120fc089ff63p+0, 0x1.843aa8b9cbbc6p-55},
    {0x1.0137444c9b5b5p+0, -0x1.2b6aeb6176892p-56}, {0x1.014d8e7ee8d2fp+0, 0x1.2edc08e5da99ap-56},
    {0x1.0163da9fb3335p+0, 0x1.b61299ab8cdb7p-54}, {0x1.017a28af25567p+0, 0x1.70fc41c5c2d53p-55},
    {0x1.019078ad6a19fp+0, -0x1.008eff5142bf9p-56}, {0x1.01a6ca9aac5f3p+0, -0x1.09bb78eeead0ap-54},
    {0x1.01bd1e77170b4p+0, 0x1.5e7626621eb5bp-56}, {0x1.01d37442d5070p+0, -0x1.ce39cbbab8bbep-57},
    {0x1.01e9cbfe113efp+0, -0x1.c11f5239bf535p-55}, {0x1.020025a8f6a35p+0, -0x1.afb99946ee3f0p-54},
    {0x1.02168143b0281p+0, -0x1.2bf310fc54eb6p-55}, {0x1.022cdece68c4fp+0, -0x1.491793e46834dp-54},
    {0x1.02433e494b755p+0, -0x1.314aa16278aa3p-54}, {0x1.02599fb483385p+0, 0x1.56dc8046821f4p-55},
    {0x1.027003103b10ep+0, -0x1.082ef51b61d7ep-56}, {0x1.0286685c9e059p+0, -0x1.fd4cf26ea5d0fp-54},
    {0x1.029ccf99d720ap+0, 0x1.64cbba902ca27p-58}, {0x1.02b338c811703p+0, 0x1.4a47a505b3a47p-54},
    {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56}, {0x1.02e010f835f7bp+0, 0x1.783bf6946c8aap-56},
    {0x1.02f67ffa765e6p+0, -0x1.b8db0e9dbd87ep-55}, {0x1.030cf0ee64571p+0, -0x1.01b29a4bf66cap-54},
    {0x1.032363d42b027p+0, 0x1.fea8d61ed6016p-54}, {0x1.0339d8abf5851p+0, 0x1.662a7706efdccp-54},
    {0x1.03504f75ef071p+0, 0x1.bc2ee8e5799acp-54}, {0x1.0366c83242b47p+0, -0x1.1d5a1cd30131fp-54},
    {0x1.037d42e11bbccp+0, 0x1.56811eeade11ap-57}, {0x1.0393bf82a5538p+0, 0x1.a7fcacf6e59bep-56},
    {0x1.03aa3e170aafep+0, -0x1.f1a93c1b824d3p-54}, {0x1.03c0be9e770cbp+0, -0x1.98df5195d7cfep-55},
    {0x1.03d7411915a8ap+0, 0x1.b7c00e7b751dap-54}, {0x1.03edc58711c63p+0, -0x1.5fc87e6550bd1p-55},
    {0x1.04044be896ab6p+0, 0x1.9dc3add8f9c02p-54}, {0x1.041ad43dcfa24p+0, -0x1.bd72fa368d2d9p-54},
    {0x1.04315e86e7f85p+0, -0x1.0a31c1977c96ep-54}, {0x1.0447eac40aff0p+0, 0x1.992d35a5dba43p-54},
    {0x1.045e78f5640b9p+0, 0x1.35bc86af4ee9ap-56}, {0x1.0475091b1e76dp+0, 0x1.874a4ea995fc6p-54},
    {0x1.048b9b35659d8p+0, 0x1.21cd53d5e8b66p-57}, {0x1.04a22f4464e00p+0, -0x1.015bc35726658p-55},
    {0x1.04b8c54847a28p+0, -0x1.e7992580447b0p-56}, {0x1.04cf5d41394cfp+0, 0x1.9ac13255c29e3p-55},
    {0x1.04e5f72f654b1p+0, 0x1.4c3793aa0d08dp-55}, {0x1.04fc9312f70c5p+0, 0x1.3241bde3cbac0p-54},
    {0x1.051330ec1a03fp+0, 0x1.79a8be239ca45p-54}, {0x1.0529d0baf9a8fp+0, 0x1.7ee717ff20af2p-54},
    {0x1.0540727fc1762p+0, -0x1.abcae24b819dfp-54}, {0x1.0557163a9ce9fp+0, -0x1.cfaf0a2f3724bp-54},
    {0x1.056dbbebb786bp+0, 0x1.06c87433776c9p-55}, {0x1.058463933cd29p+0, -0x1.f41499f211486p-54},
};
// sin(pi (2j + 1) / 512)
__device__ const double kSinTable[128] = {
    0x1.921f0fe670071p-8, 0x1.2d936bbe30efdp-6, 0x1.f693731d1cf01p-6, 0x1.5fc00d290cd43p-5,
    0x1.c428d12c0d7e3p-5, 0x1.1440134d709b3p-4, 0x1.4661179272096p-4, 0x1.787586a5d5b21p-4,
    0x1.aa7b724495c03p-4, 0x1.dc70ecbae9fc9p-4, 0x1.072a047ba831dp-3, 0x1.20116d4ec7bcfp-3,
    0x1.38edbb0cd8d14p-3, 0x1.51bdf8597c5f2p-3, 0x1.6a81304f64ab2p-3, 0x1.83366e89c64c6p-3,
    0x1.9bdcbf2dc4366p-3, 0x1.b4732ef3d6722p-3, 0x1.ccf8cb312b286p-3, 0x1.e56ca1e101a1bp-3,
    0x1.fdcdc1adfedf9p-3, 0x1.0b0d9cfdbdb90p-2, 0x1.172a0d7765177p-2, 0x1.233bbabc3bb71p-2,
    0x1.2f422daec0387p-2, 0x1.3b3cefa0414b7p-2, 0x1.472b8a5571054p-2, 0x1.530d880af3c24p-2,
    0x1.5ee27379ea693p-2, 0x1.6aa9d7dc77e17p-2, 0x1.766340f2418f6p-2, 0x1.820e3b04eaac4p-2,
    0x1.8daa52ec8a4b0p-2, 0x1.993716141bdffp-2, 0x1.a4b4127dea1e5p-2, 0x1.b020d6c7f4009p-2,
    0x1.bb7cf2304bd01p-2, 0x1.c6c7f4997000bp-2, 0x1.d2016e8e9db5bp-2, 0x1.dd28f1481cc58p-2,
    0x1.e83e0eaf85114p-2, 0x1.f3405963fd067p-2, 0x1.fe2f64be71210p-2, 0x1.0485626ae221ap-1,
    0x1.09e907417c5e1p-1, 0x1.0f426bb2a8e7ep-1, 0x1.14915af336cebp-1, 0x1.19d5a09f2b9b8p-1,
    0x1.1f0f08bbc861bp-1, 0x1.243d5fb98ac1fp-1, 0x1.2960727629ca8p-1, 0x1.2e780e3e8ea17p-1,
    0x1.338400d0c8e57p-1, 0x1.3884185dfeb22p-1, 0x1.3d78238c58344p-1, 0x1.425ff178e6bb1p-1,
    0x1.473b51b987347p-1, 0x1.4c0a145ec0004p-1, 0x1.50cc09f59a09bp-1, 0x1.5581038975137p-1,
    0x1.5a28d2a5d7250p-1, 0x1.5ec3495837074p-1, 0x1.63503a31c1be9p-1, 0x1.67cf78491af10p-1,
    0x1.6c40d73c18275p-1, 0x1.70a42b3176d7ap-1, 0x1.74f948da8d28dp-1, 0x1.79400574f55e5p-1,
    0x1.7d7836cc33db2p-1, 0x1.81a1b33b57accp-1, 0x1.85bc51ae958ccp-1, 0x1.89c7e9a4dd4aap-1,
    0x1.8dc45331698ccp-1, 0x1.91b166fd49da2p-1, 0x1.958efe48e6dd7p-1, 0x1.995cf2ed80d22p-1,
    0x1.9d1b1f5ea80d5p-1, 0x1.a0c95eabaf937p-1, 0x1.a4678c8119ac8p-1, 0x1.a7f58529fe69dp-1,
    0x1.ab7325916c0d4p-1, 0x1.aee04b43c1474p-1, 0x1.b23cd470013b4p-1, 0x1.b5889fe921405p-1,
    0x1.b8c38d27504e9p-1, 0x1.bbed7c49380eap-1, 0x1.bf064e15377ddp-1, 0x1.c20de3fa971b0p-1,
    0x1.c5042012b6907p-1, 0x1.c7e8e52233cf3p-1, 0x1.cabc169a0b900p-1, 0x1.cd7d9898b32f6p-1,
    0x1.d02d4feb2bd92p-1, 0x1.d2cb220e0ef9fp-1, 0x1.d556f52e93eb1p-1, 0x1.d7d0b02b8ecf9p-1,
    0x1.da383a9668988p-1, 0x1.dc8d7cb410260p-1, 0x1.ded05f7de47dap-1, 0x1.e100cca2980acp-1,
    0x1.e31eae870ce25p-1, 0x1.e529f04729ffcp-1, 0x1.e7227db6a9744p-1, 0x1.e9084361df7f2p-1,
    0x1.eadb2e8e7a88ep-1, 0x1.ec9b2d3c3bf84p-1, 0x1.ee482e25a9dbcp-1, 0x1.efe220c0b95ecp-1,
    0x1.f168f53f7205dp-1, 0x1.f2dc9c9089a9dp-1, 0x1.f43d085ff92ddp-1, 0x1.f58a2b1789e84p-1,
    0x1.f6c3f7df5bbb7p-1, 0x1.f7ea629e63d6ep-1, 0x1.f8fd5ffae41dbp-1, 0x1.f9fce55adb2c8p-1,
    0x1.fae8e8e46cfbbp-1, 0x1.fbc1617e44186p-1, 0x1.fc8646cfeb721p-1, 0x1.fd37914220b84p-1,
    0x1.fdd539ff1f456p-1, 0x1.fe5f3af2e3940p-1, 0x1.fed58ecb673c4p-1, 0x1.ff3830f8d575cp-1,
    0x1.ff871dadb81dfp-1, 0x1.ffc251df1d3f8p-1, 0x1.ffe9cb44b51a1p-1, 0x1.fffd8858e8a92p-1,
};

constexpr int kLogIntervals = 512, kLogOne = 320;   // interval kLogOne begins at 1
constexpr int kSinCosEntries = 512;
constexpr int kExpEntries = 2048;

// exp(mu + sigma z) = e^mu 2^(sigma' z / 2048)
struct LogNormal {
    double mu, sigma;            // as given
    double exp_mu, exp_mu_rest;  // e^mu in two parts
    double square;               // sigma'^2, a factor of everything that makes up sigma'^2 (-2 ln u)
    double log_poly[5];          // of r^1 .. r^5, times it

    __host__ static LogNormal make(double mu, double sigma) {
        constexpr double k2048_over_ln2 = 0x1.71547652b82fep+11;
        // (a sigma of 0 as one that changes no time but leaves the square root a positive argument)
        const double scaled = (sigma > 1e-100 ? sigma : 1e-100) * k2048_over_ln2, square = scaled * scaled;
        const long double power = expl((long double)mu);
        // -2 ln(1 + r) to r^5, interpolated at Chebyshev nodes of |r| <= 2^-9: within 2.4e-18
        return {mu, sigma, (double)power, (double)(power - (long double)(double)power), square,
                {-2.0 * square, 0.99999999999939366846 * square, -0.66666666666614695386 * square, 0.50000127156893844812 * square,
                 -0.40000108991633401330 * square}};
    }
    // |z| < 8.7, so exp stays within the normal numbers and the table-driven form applies.
    __host__ static bool tame(double mu, double sigma) { return fabs(mu) + 8.7 * sigma < 700.0; }
};

struct LogNormalTables {
    double2 log[kLogIntervals];            // c_i, 2 ln c_i sigma'^2
    double2 sin_cos[kSinCosEntries];       // of 2 pi (j + 1/2) / 512
    double exp2[kExpEntries];              // e^mu 2^(j / 2048), j taken off its high word 9 bits up
    double exponent[56];                   // 2 ln 2 (54 - j) sigma'^2
};

// Filled by the whole CTA; a barrier has to follow.
__device__ __forceinline__ void fill_tables(LogNormalTables& t, const LogNormal& q) {
    for (int i = threadIdx.x; i < kLogIntervals; i += blockDim.x) {
        // c the reciprocal of the middle m of the interval, ln c = ln c_g + 2 artanh((c - c_g) / (c + c_g)) with c_g of its
        // group; 1 on both sides of 1, and 2^-120 for its logarithm
        double c = __drcp_rn(__hiloint2double(0x3FE60000 + (i << 11) + (1 << 10), 0));
        const double* group = kLogGroup[i >> 5];
        const double s = __ddiv_rn(c - group[0], c + group[0]), s2 = s * s;
        const double odd = fma(s2, fma(s2, fma(s2, fma(s2, 1.0 / 9.0, 1.0 / 7.0), 1.0 / 5.0), 1.0 / 3.0), 0.0) * s;
        double twice_ln = 2.0 * (group[1] + (group[2] + 2.0 * (s + odd)));
        if (i == kLogOne - 1 || i == kLogOne) {
            c = 1.0;
            twice_ln = 0x1.0p-120;
        }
        t.log[i] = make_double2(c, twice_ln * q.square);
    }
    for (int j = threadIdx.x; j < kExpEntries; j += blockDim.x) {
        const double2 a = kExpCoarse[j >> 6], b = kExpFine[j & 63];
        const double ab = a.x * b.x, ab_rest = fma(a.x, b.x, -ab) + fma(a.x, b.y, a.y * b.x);
        const double v = ab * q.exp_mu, e = v + (fma(ab, q.exp_mu, -v) + fma(ab, q.exp_mu_rest, ab_rest * q.exp_mu));
        t.exp2[j] = __hiloint2double(__double2hiint(e) - (j << 9), __double2loint(e));
    }
    for (int i = threadIdx.x; i < kSinCosEntries; i += blockDim.x) {
        const double a = kSinTable[i & 127], b = kSinTable[127 - (i & 127)];
        const double s = i & 128 ? b : a, c = i & 128 ? -a : b;            // second quadrant: cos, -sin
        t.sin_cos[i] = i & 256 ? make_double2(-s, -c) : make_double2(s, c);
    }
    for (int i = threadIdx.x; i < 55; i += blockDim.x) t.exponent[i] = (54 - i) * 0x1.62e42fefa39efp+0 * q.square;
}

// e^mu 2^(radius x / 2048), radius x = k + f, |f| <= 1/2, k by adding 1.5 * 2^52.
__device__ __forceinline__ double exp2_2048(const LogNormalTables& t, double radius, double x) {
    const double shifted = fma(radius, x, 0x1.8p52);
    const int k = __double2loint(shifted);
    const double f = fma(radius, x, 0x1.8p52 - shifted);
    // e^y - 1, y = f ln2 / 2048, to y^3, interpolated: within 5.9e-18
    constexpr double kY = 0x1.62e42fefa39efp-12;                         // ln2 / 2048
    double p = fma(f, kY * kY * kY * 0.16666666686436549282, kY * kY * 0.500000000988494131);
    p = fma(p, f, kY) * f;
    const double power = t.exp2[k & (kExpEntries - 1)];
    const double e = __hiloint2double(__double2hiint(power) + (k << 9), __double2loint(power));
    return fma(e, p, e);
}

// The two times of one word pair: cosine first, sine second.
template <bool TAME>
__device__ __forceinline__ void lognormal2(const LogNormalTables& t, uint64_t wa, uint64_t wb, const LogNormal& q,
                                           double& t_cos, double& t_sin) {
    if constexpr (!TAME) {
        double s, c;
        const double r = sqrt(-2.0 * log(((double)(wa >> 11) + 0.5) * 0x1.0p-53));
        sincospi(2.0 * (((double)(wb >> 11) + 0.5) * 0x1.0p-53), &s, &c);
        t_cos = exp(q.mu + q.sigma * (r * c));
        t_sin = exp(q.mu + q.sigma * (r * s));
        return;
    }
    // sigma'^2 (-2 ln u), u = v 2^-64 = m 2^(e - 64) with m in [0.6875, 1.375), m c_i = 1 + r, |r| <= 2^-9.  Near u = 1
    // both 64 - e and ln c_i vanish and nothing cancels; the 2^-120 kept in their place makes the result positive at u = 1.
    const double v = __ull2double_rn((wa & ~0x7FFull) | 0x400);           // 2^11 times (wa >> 11) + 1/2, rounded as that is
    const int above = __double2hiint(v) - 0x3FE60000;
    const int e = above >> 20;                                            // 10 .. 64
    const double m = __hiloint2double(__double2hiint(v) - (e << 20), __double2loint(v));
    const double2 cl = t.log[(above >> 11) & (kLogIntervals - 1)];
    const double r = fma(m, cl.x, -1.0);
    double p = fma(r, q.log_poly[4], q.log_poly[3]);
    p = fma(p, r, q.log_poly[2]);
    p = fma(p, r, q.log_poly[1]);
    p = fma(p, r, q.log_poly[0]);
    const double x = fma(p, r, t.exponent[e - 10] + cl.y);
    // sqrt(x): y = x^-1/2 (1 + O(2^-20)), one step of third order
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = x * y, d = fma(-h, y, 1.0);
    const double radius = fma(h * d, fma(d, 0.375, 0.5), h);
    // angle: the table entry of the leading 9 bits, turned by the rest, a = pi 2^-53 i (|a| <= pi / 512)
    const uint32_t hi = (uint32_t)(wb >> 32), lo = (uint32_t)wb;
    const double i = __hiloint2double(0x43300000 | ((hi >> 10) & 0x1FFF), __funnelshift_r(lo, hi, 10) | 1) -
                     (0x1.0p52 + 0x1.0p44);
    constexpr double k = 0x1.921fb54442d18p-52;   // pi 2^-53
    const double2 sc = t.sin_cos[hi >> 23];
    const double i2 = i * i;
    const double sa = fma(i2, fma(i2, k * k * k * k * k / 120.0, -k * k * k / 6.0), k) * i;
    const double ca = fma(i2, k * k * k * k * 0.041666614375651651347, k * k * -0.49999999999975390835) * i2;   // cos a - 1, within 1e-17
    const double s = fma(sc.y, sa, fma(sc.x, ca, sc.x));
    const double c = fma(-sc.x, sa, fma(sc.y, ca, sc.y));
    t_cos = exp2_2048(t, radius, c);
    t_sin = exp2_2048(t, radius, s);
}

// The four times of one block.
template <bool TAME>
__device__ __forceinline__ void lognormal4(const LogNormalTables& t, const Philox4& b, const LogNormal& q, double (&out)[4]) {
    lognormal2<TAME>(t, b.w0, b.w1, q, out[0], out[1]);
    lognormal2<TAME>(t, b.w2, b.w3, q, out[2], out[3]);
}

}  // namespace

}  // namespace nolo
