// Log-normal times from Philox blocks in float64, the inner loop of the latency simulations.
//
// Words -> u = ((x >> 11) + 0.5) 2^-53; Box-Muller on the word pairs (0,1) and (2,3), r = sqrt(-2 ln u_a),
// gives the normals [r01 cos, r01 sin, r23 cos, r23 sin] of the angle 2 pi u_b; t = exp(mu + sigma z).
//
// Bound by the pipes of the float64 operations and of Philox's products.  The logarithm, sine and cosine and
// exponential are table-driven in the manner of P. T. P. Tang (ACM TOMS 15, 1989, "Table-driven implementation of
// the exponential function in IEEE floating-point arithmetic", and TOMS 16, 1990, for the logarithm): a table in
// shared memory takes the leading bits, a Taylor polynomial the rest.  The logarithm's intervals (128 of equal high
// word, from 0.6875 on, with a reciprocal of 1 next to 1) are laid out as in the log of Arm's optimized-routines; the
// tables' values are computed from their definitions.  The arguments are confined (u in (0, 1],
// angles as integers, exponents checked once on the host), so no special case is left in the loop, the angle
// is reduced in integers and the factors 2, pi, sigma and 256 / ln 2 are folded into constants.  About 24 float64
// operations per time; each step is good to one or two units in the last place.
#pragma once

#include <stdint.h>

#include "nolo_philox.cuh"

namespace nolo {

namespace {

// reciprocal c_i of the centre of interval i (1 next to 1), 2 ln c_i (2^-120 for c_i = 1)
__device__ const double2 kLogTable[128] = {
    {0x1.734f0c541fe8dp+0, 0x1.7cc7f7db46a0ep-1}, {0x1.713786d9c7c09p+0, 0x1.76feecb947176p-1},
    {0x1.6f26016f26017p+0, 0x1.713e33a46a17cp-1}, {0x1.6d1a62681c861p+0, 0x1.6b85b4cffa3fdp-1},
    {0x1.6b1490aa31a3dp+0, 0x1.65d558d4ce00bp-1}, {0x1.691473a88d0c0p+0, 0x1.602d08af091ecp-1},
    {0x1.6719f3601671ap+0, 0x1.5a8cadbbedfa1p-1}, {0x1.6524f853b4aa3p+0, 0x1.54f431b7be1a8p-1},
    {0x1.63356b88ac0dep+0, 0x1.4f637ebba9810p-1}, {0x1.614b36831ae94p+0, 0x1.49da7f3bcc420p-1},
    {0x1.5f66434292dfcp+0, 0x1.44591e0539f49p-1}, {0x1.5d867c3ece2a5p+0, 0x1.3edf463c1683ep-1},
    {0x1.5babcc647fa91p+0, 0x1.396ce359bbf53p-1}, {0x1.59d61f123ccaap+0, 0x1.3401e12aecba0p-1},
    {0x1.5805601580560p+0, 0x1.2e9e2bce12286p-1}, {0x1.56397ba7c52e2p+0, 0x1.2941afb186b7cp-1},
    {0x1.54725e6bb82fep+0, 0x1.23ec5991eba49p-1}, {0x1.52aff56a8054bp+0, 0x1.1e9e1678899f5p-1},
    {0x1.50f22e111c4c5p+0, 0x1.1956d3b9bc2f9p-1}, {0x1.4f38f62dd4c9bp+0, 0x1.14167ef367784p-1},
    {0x1.4d843bedc2c4cp+0, 0x1.0edd060b78082p-1}, {0x1.4bd3edda68fe1p+0, 0x1.09aa572e6c6d4p-1},
    {0x1.4a27fad76014ap+0, 0x1.047e60cde83b7p-1}, {0x1.4880522014880p+0, 0x1.feb2233ea07cbp-2},
    {0x1.46dce34596066p+0, 0x1.f474b134df228p-2}, {0x1.453d9e2c776cap+0, 0x1.ea4449f04aaf5p-2},
    {0x1.43a2730abee4dp+0, 0x1.e020cc6235ab5p-2}, {0x1.420b5265e5951p+0, 0x1.d60a17f903514p-2},
    {0x1.40782d10e6566p+0, 0x1.cc000c9db3c52p-2}, {0x1.3ee8f42a5af07p+0, 0x1.c2028ab17f9b5p-2},
    {0x1.3d5d991aa75c6p+0, 0x1.b811730b823d4p-2}, {0x1.3bd60d9232955p+0, 0x1.ae2ca6f672bd8p-2},
    {0x1.3a524387ac822p+0, 0x1.a454082e6ab03p-2}, {0x1.38d22d366088ep+0, 0x1.9a8778debaa3ap-2},
    {0x1.3755bd1c945eep+0, 0x1.90c6db9fcbcdbp-2}, {0x1.35dce5f9f2af8p+0, 0x1.871213750e994p-2},
    {0x1.34679ace01346p+0, 0x1.7d6903caf5acdp-2}, {0x1.32f5ced6a1dfap+0, 0x1.73cb9074fd14dp-2},
    {0x1.3187758e9ebb6p+0, 0x1.6a399dabbd383p-2}, {0x1.301c82ac40260p+0, 0x1.60b3100b09474p-2},
    {0x1.2eb4ea1fed14bp+0, 0x1.5737cc9018cddp-2}, {0x1.2d50a012d50a0p+0, 0x1.4dc7b897bc1c7p-2},
    {0x1.2bef98e5a3711p+0, 0x1.4462b9dc9b3dcp-2}, {0x1.2a91c92f3c105p+0, 0x1.3b08b6757f2a7p-2},
    {0x1.293725bb804a5p+0, 0x1.31b994d3a4f86p-2}, {0x1.27dfa38a1ce4dp+0, 0x1.28753bc11aba2p-2},
    {0x1.268b37cd60127p+0, 0x1.1f3b925f25d44p-2}, {0x1.2539d7e9177b2p+0, 0x1.160c8024b27b0p-2},
    {0x1.23eb79717605bp+0, 0x1.0ce7ecdccc28bp-2}, {0x1.22a0122a0122ap+0, 0x1.03cdc0a51ec0dp-2},
    {0x1.21579804855e6p+0, 0x1.f57bc7d9005dbp-3}, {0x1.2012012012012p+0, 0x1.e3707ee30487bp-3},
    {0x1.1ecf43c7fb84cp+0, 0x1.d179788219362p-3}, {0x1.1d8f5672e4abdp+0, 0x1.bf968769fca18p-3},
    {0x1.1c522fc1ce059p+0, 0x1.adc77ee5aea8ep-3}, {0x1.1b17c67f2bae3p+0, 0x1.9c0c32d4d254dp-3},
    {0x1.19e0119e0119ep+0, 0x1.8a6477a91dc29p-3}, {0x1.18ab083902bdbp+0, 0x1.78d02263d82d7p-3},
    {0x1.1778a191bd684p+0, 0x1.674f089365a78p-3}, {0x1.1648d50fc3201p+0, 0x1.55e10050e0382p-3},
    {0x1.151b9a3fdd5c9p+0, 0x1.4485e03dbdfb0p-3}, {0x1.13f0e8d344724p+0, 0x1.333d7f8183f4ap-3},
    {0x1.12c8b89edc0acp+0, 0x1.2207b5c7854a1p-3}, {0x1.11a3019a74826p+0, 0x1.10e45b3cae829p-3},
    {0x1.107fbbe011080p+0, 0x1.ffa6911ab9309p-4}, {0x1.0f5edfab325a2p+0, 0x1.dda8adc67ee59p-4},
    {0x1.0e40655826011p+0, 0x1.bbcebfc68f424p-4}, {0x1.0d24456359e3ap+0, 0x1.9a187b573de81p-4},
    {0x1.0c0a7868b4171p+0, 0x1.788595a3577c8p-4}, {0x1.0af2f722eecb5p+0, 0x1.5715c4c03cee1p-4},
    {0x1.09ddba6af8360p+0, 0x1.35c8bfaa13069p-4}, {0x1.08cabb37565e2p+0, 0x1.149e3e4005a8dp-4},
    {0x1.07b9f29b8eae2p+0, 0x1.e72bf2813ce6ap-5}, {0x1.06ab59c7912fbp+0, 0x1.a55f548c5c427p-5},
    {0x1.059eea0727586p+0, 0x1.63d6178690bbep-5}, {0x1.04949cc1664c5p+0, 0x1.228fb1fea2e0ap-5},
    {0x1.038c6b78247fcp+0, 0x1.c317384c75f0dp-6}, {0x1.02864fc7729e9p+0, 0x1.41929f968330cp-6},
    {0x1.0182436517a37p+0, 0x1.8121214586b02p-7}, {0x1.0000000000000p+0, 0x1.0000000000000p-120},
    {0x1.0000000000000p+0, 0x1.0000000000000p-120}, {0x1.fa11caa01fa12p-1, -0x1.7dc475f810a69p-6},
    {0x1.f6310aca0dbb5p-1, -0x1.3cea44346a584p-5}, {0x1.f25f644230ab5p-1, -0x1.b9fc027af919ap-5},
    {0x1.ee9c7f8458e02p-1, -0x1.1b0d98923d97fp-4}, {0x1.eae807aba01ebp-1, -0x1.58a5bafc8e4d3p-4},
    {0x1.e741aa59750e4p-1, -0x1.95c830ec8e3f2p-4}, {0x1.e3a9179dc1a73p-1, -0x1.d276b8adb0b56p-4},
    {0x1.e01e01e01e01ep-1, -0x1.075983598e471p-3}, {0x1.dca01dca01dcap-1, -0x1.253f62f0a1417p-3},
    {0x1.d92f2231e7f8ap-1, -0x1.42edcbea646eep-3}, {0x1.d5cac807572b2p-1, -0x1.60658a93750c4p-3},
    {0x1.d272ca3fc5b1ap-1, -0x1.7da766d7b12d0p-3}, {0x1.cf26e5c44bfc6p-1, -0x1.9ab42462033aep-3},
    {0x1.cbe6d9601cbe7p-1, -0x1.b78c82bb0eda0p-3}, {0x1.c8b265afb8a42p-1, -0x1.d4313d66cb35dp-3},
    {0x1.c5894d10d4986p-1, -0x1.f0a30c01162a4p-3}, {0x1.c26b5392ea01cp-1, -0x1.0671512ca596fp-2},
    {0x1.bf583ee868d8bp-1, -0x1.14785846742acp-2}, {0x1.bc4fd65883e7bp-1, -0x1.2266f190a5acdp-2},
    {0x1.b951e2b18ff23p-1, -0x1.303d718e47fd5p-2}, {0x1.b65e2e3beee05p-1, -0x1.3dfc2b0ecc62ap-2},
    {0x1.b37484ad806cep-1, -0x1.4ba36f39a55e5p-2}, {0x1.b094b31d922a4p-1, -0x1.59338d9982085p-2},
    {0x1.adbe87f94905ep-1, -0x1.66acd4272ad51p-2}, {0x1.aaf1d2f87ebfdp-1, -0x1.740f8f54037a3p-2},
    {0x1.a82e65130e159p-1, -0x1.815c0a14357e9p-2}, {0x1.a574107688a4ap-1, -0x1.8e928de886d41p-2},
    {0x1.a2c2a87c51ca0p-1, -0x1.9bb362e7dfb85p-2}, {0x1.a01a01a01a01ap-1, -0x1.a8becfc882f19p-2},
    {0x1.9d79f176b682dp-1, -0x1.b5b519e8fb5a6p-2}, {0x1.9ae24ea5510dap-1, -0x1.c2968558c18c2p-2},
    {0x1.9852f0d8ec0ffp-1, -0x1.cf6354e09c5ddp-2}, {0x1.95cbb0be377aep-1, -0x1.dc1bca0abec7bp-2},
    {0x1.934c67f9b2ce6p-1, -0x1.e8c0252aa5a60p-2}, {0x1.90d4f120190d5p-1, -0x1.f550a564b7b37p-2},
    {0x1.8e6527af1373fp-1, -0x1.00e6c45ad501dp-1}, {0x1.8bfce8062ff3ap-1, -0x1.071b85fcd590dp-1},
    {0x1.899c0f601899cp-1, -0x1.0d46b579ab74bp-1}, {0x1.87427bcc092b9p-1, -0x1.136870293a8b0p-1},
    {0x1.84f00c2780614p-1, -0x1.1980d2dd4236fp-1}, {0x1.82a4a0182a4a0p-1, -0x1.1f8ff9e48a2f3p-1},
    {0x1.8060180601806p-1, -0x1.2596010df763ap-1}, {0x1.7e225515a4f1dp-1, -0x1.2b9303ab89d25p-1},
    {0x1.7beb3922e017cp-1, -0x1.31871c9544185p-1}, {0x1.79baa6bb6398bp-1, -0x1.3772662bfd85cp-1},
    {0x1.77908119ac60dp-1, -0x1.3d54fa5c1f710p-1}, {0x1.756cac201756dp-1, -0x1.432ef2a04e813p-1},
};
// 2^(j / 256)
__device__ const double kExpTable[256] = {
    0x1.0000000000000p+0, 0x1.00b1afa5abcbfp+0, 0x1.0163da9fb3335p+0, 0x1.02168143b0281p+0,
    0x1.02c9a3e778061p+0, 0x1.037d42e11bbccp+0, 0x1.04315e86e7f85p+0, 0x1.04e5f72f654b1p+0,
    0x1.059b0d3158574p+0, 0x1.0650a0e3c1f89p+0, 0x1.0706b29ddf6dep+0, 0x1.07bd42b72a836p+0,
    0x1.0874518759bc8p+0, 0x1.092bdf66607e0p+0, 0x1.09e3ecac6f383p+0, 0x1.0a9c79b1f3919p+0,
    0x1.0b5586cf9890fp+0, 0x1.0c0f145e46c85p+0, 0x1.0cc922b7247f7p+0, 0x1.0d83b23395decp+0,
    0x1.0e3ec32d3d1a2p+0, 0x1.0efa55fdfa9c5p+0, 0x1.0fb66affed31bp+0, 0x1.1073028d7233ep+0,
    0x1.11301d0125b51p+0, 0x1.11edbab5e2ab6p+0, 0x1.12abdc06c31ccp+0, 0x1.136a814f204abp+0,
    0x1.1429aaea92de0p+0, 0x1.14e95934f312ep+0, 0x1.15a98c8a58e51p+0, 0x1.166a45471c3c2p+0,
    0x1.172b83c7d517bp+0, 0x1.17ed48695bbc0p+0, 0x1.18af9388c8deap+0, 0x1.1972658375d2fp+0,
    0x1.1a35beb6fcb75p+0, 0x1.1af99f8138a1cp+0, 0x1.1bbe084045cd4p+0, 0x1.1c82f95281c6bp+0,
    0x1.1d4873168b9aap+0, 0x1.1e0e75eb44027p+0, 0x1.1ed5022fcd91dp+0, 0x1.1f9c18438ce4dp+0,
    0x1.2063b88628cd6p+0, 0x1.212be3578a819p+0, 0x1.21f49917ddc96p+0, 0x1.22bdda27912d1p+0,
    0x1.2387a6e756238p+0, 0x1.2451ffb82140ap+0, 0x1.251ce4fb2a63fp+0, 0x1.25e85711ece75p+0,
    0x1.26b4565e27cddp+0, 0x1.2780e341ddf29p+0, 0x1.284dfe1f56381p+0, 0x1.291ba7591bb70p+0,
    0x1.29e9df51fdee1p+0, 0x1.2ab8a66d10f13p+0, 0x1.2b87fd0dad990p+0, 0x1.2c57e39771b2fp+0,
    0x1.2d285a6e4030bp+0, 0x1.2df961f641589p+0, 0x1.2ecafa93e2f56p+0, 0x1.2f9d24abd886bp+0,
    0x1.306fe0a31b715p+0, 0x1.31432edeeb2fdp+0, 0x1.32170fc4cd831p+0, 0x1.32eb83ba8ea32p+0,
    0x1.33c08b26416ffp+0, 0x1.3496266e3fa2dp+0, 0x1.356c55f929ff1p+0, 0x1.36431a2de883bp+0,
    0x1.371a7373aa9cbp+0, 0x1.37f26231e754ap+0, 0x1.38cae6d05d866p+0, 0x1.39a401b7140efp+0,
    0x1.3a7db34e59ff7p+0, 0x1.3b57fbfec6cf4p+0, 0x1.3c32dc313a8e5p+0, 0x1.3d0e544ede173p+0,
    0x1.3dea64c123422p+0, 0x1.3ec70df1c5175p+0, 0x1.3fa4504ac801cp+0, 0x1.40822c367a024p+0,
    0x1.4160a21f72e2ap+0, 0x1.423fb2709468ap+0, 0x1.431f5d950a897p+0, 0x1.43ffa3f84b9d4p+0,
    0x1.44e086061892dp+0, 0x1.45c2042a7d232p+0, 0x1.46a41ed1d0057p+0, 0x1.4786d668b3237p+0,
    0x1.486a2b5c13cd0p+0, 0x1.494e1e192aed2p+0, 0x1.4a32af0d7d3dep+0, 0x1.4b17dea6db7d7p+0,
    0x1.4bfdad5362a27p+0, 0x1.4ce41b817c114p+0, 0x1.4dcb299fddd0dp+0, 0x1.4eb2d81d8abffp+0,
    0x1.4f9b2769d2ca7p+0, 0x1.508417f4531eep+0, 0x1.516daa2cf6642p+0, 0x1.5257de83f4eefp+0,
    0x1.5342b569d4f82p+0, 0x1.542e2f4f6ad27p+0, 0x1.551a4ca5d920fp+0, 0x1.56070dde910d2p+0,
    0x1.56f4736b527dap+0, 0x1.57e27dbe2c4cfp+0, 0x1.58d12d497c7fdp+0, 0x1.59c0827ff07ccp+0,
    0x1.5ab07dd485429p+0, 0x1.5ba11fba87a03p+0, 0x1.5c9268a5946b7p+0, 0x1.5d84590998b93p+0,
    0x1.5e76f15ad2148p+0, 0x1.5f6a320dceb71p+0, 0x1.605e1b976dc09p+0, 0x1.6152ae6cdf6f4p+0,
    0x1.6247eb03a5585p+0, 0x1.633dd1d1929fdp+0, 0x1.6434634ccc320p+0, 0x1.652b9febc8fb7p+0,
    0x1.6623882552225p+0, 0x1.671c1c70833f6p+0, 0x1.68155d44ca973p+0, 0x1.690f4b19e9538p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6b052fa75173ep+0, 0x1.6c012750bdabfp+0, 0x1.6cfdcddd47645p+0,
    0x1.6dfb23c651a2fp+0, 0x1.6ef9298593ae5p+0, 0x1.6ff7df9519484p+0, 0x1.70f7466f42e87p+0,
    0x1.71f75e8ec5f74p+0, 0x1.72f8286ead08ap+0, 0x1.73f9a48a58174p+0, 0x1.74fbd35d7cbfdp+0,
    0x1.75feb564267c9p+0, 0x1.77024b1ab6e09p+0, 0x1.780694fde5d3fp+0, 0x1.790b938ac1cf6p+0,
    0x1.7a11473eb0187p+0, 0x1.7b17b0976cfdbp+0, 0x1.7c1ed0130c132p+0, 0x1.7d26a62ff86f0p+0,
    0x1.7e2f336cf4e62p+0, 0x1.7f3878491c491p+0, 0x1.80427543e1a12p+0, 0x1.814d2add106d9p+0,
    0x1.82589994cce13p+0, 0x1.8364c1eb941f7p+0, 0x1.8471a4623c7adp+0, 0x1.857f4179f5b21p+0,
    0x1.868d99b4492edp+0, 0x1.879cad931a436p+0, 0x1.88ac7d98a6699p+0, 0x1.89bd0a478580fp+0,
    0x1.8ace5422aa0dbp+0, 0x1.8be05bad61778p+0, 0x1.8cf3216b5448cp+0, 0x1.8e06a5e0866d9p+0,
    0x1.8f1ae99157736p+0, 0x1.902fed0282c8ap+0, 0x1.9145b0b91ffc6p+0, 0x1.925c353aa2fe2p+0,
    0x1.93737b0cdc5e5p+0, 0x1.948b82b5f98e5p+0, 0x1.95a44cbc8520fp+0, 0x1.96bdd9a7670b3p+0,
    0x1.97d829fde4e50p+0, 0x1.98f33e47a22a2p+0, 0x1.9a0f170ca07bap+0, 0x1.9b2bb4d53fe0dp+0,
    0x1.9c49182a3f090p+0, 0x1.9d674194bb8d5p+0, 0x1.9e86319e32323p+0, 0x1.9fa5e8d07f29ep+0,
    0x1.a0c667b5de565p+0, 0x1.a1e7aed8eb8bbp+0, 0x1.a309bec4a2d33p+0, 0x1.a42c980460ad8p+0,
    0x1.a5503b23e255dp+0, 0x1.a674a8af46052p+0, 0x1.a799e1330b358p+0, 0x1.a8bfe53c12e59p+0,
    0x1.a9e6b5579fdbfp+0, 0x1.ab0e521356ebap+0, 0x1.ac36bbfd3f37ap+0, 0x1.ad5ff3a3c2774p+0,
    0x1.ae89f995ad3adp+0, 0x1.afb4ce622f2ffp+0, 0x1.b0e07298db666p+0, 0x1.b20ce6c9a8952p+0,
    0x1.b33a2b84f15fbp+0, 0x1.b468415b749b1p+0, 0x1.b59728de5593ap+0, 0x1.b6c6e29f1c52ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.b928cf22749e4p+0, 0x1.ba5b030a1064ap+0, 0x1.bb8e0b79a6f1fp+0,
    0x1.bcc1e904bc1d2p+0, 0x1.bdf69c3f3a207p+0, 0x1.bf2c25bd71e09p+0, 0x1.c06286141b33dp+0,
    0x1.c199bdd85529cp+0, 0x1.c2d1cd9fa652cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c544778fafb22p+0,
    0x1.c67f12e57d14bp+0, 0x1.c7ba88988c933p+0, 0x1.c8f6d9406e7b5p+0, 0x1.ca3405751c4dbp+0,
    0x1.cb720dcef9069p+0, 0x1.ccb0f2e6d1675p+0, 0x1.cdf0b555dc3fap+0, 0x1.cf3155b5bab74p+0,
    0x1.d072d4a07897cp+0, 0x1.d1b532b08c968p+0, 0x1.d2f87080d89f2p+0, 0x1.d43c8eacaa1d6p+0,
    0x1.d5818dcfba487p+0, 0x1.d6c76e862e6d3p+0, 0x1.d80e316c98398p+0, 0x1.d955d71ff6075p+0,
    0x1.da9e603db3285p+0, 0x1.dbe7cd63a8315p+0, 0x1.dd321f301b460p+0, 0x1.de7d5641c0658p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e11676b197d17p+0, 0x1.e264614f5a129p+0, 0x1.e3b333b16ee12p+0,
    0x1.e502ee78b3ff6p+0, 0x1.e653924676d76p+0, 0x1.e7a51fbc74c83p+0, 0x1.e8f7977cdb740p+0,
    0x1.ea4afa2a490dap+0, 0x1.eb9f4867cca6ep+0, 0x1.ecf482d8e67f1p+0, 0x1.ee4aaa2188510p+0,
    0x1.efa1bee615a27p+0, 0x1.f0f9c1cb6412ap+0, 0x1.f252b376bba97p+0, 0x1.f3ac948dd7274p+0,
    0x1.f50765b6e4540p+0, 0x1.f6632798844f8p+0, 0x1.f7bfdad9cbe14p+0, 0x1.f91d802243c89p+0,
    0x1.fa7c1819e90d8p+0, 0x1.fbdba3692d514p+0, 0x1.fd3c22b8f71f1p+0, 0x1.fe9d96b2a23d9p+0,
};
// sin(pi (2j + 1) / 256)
__device__ const double kSinTable[64] = {
    0x1.921d1fcdec784p-7, 0x1.2d865759455cdp-5, 0x1.f656e79f820e0p-5, 0x1.5f6d00a9aa419p-4,
    0x1.c3785c79ec2d5p-4, 0x1.139f0cedaf577p-3, 0x1.45576b1293e5ap-3, 0x1.76dd9de50bf31p-3,
    0x1.a82a025b00451p-3, 0x1.d934fe5454311p-3, 0x1.04fb80e37fdaep-2, 0x1.1d3443f4cdb3ep-2,
    0x1.35410c2e18152p-2, 0x1.4d1e24278e76ap-2, 0x1.64c7ddd3f27c6p-2, 0x1.7c3a9311dcce7p-2,
    0x1.9372a63bc93d7p-2, 0x1.aa6c82b6d3fcap-2, 0x1.c1249d8011ee7p-2, 0x1.d79775b86e389p-2,
    0x1.edc1952ef78d6p-2, 0x1.01cfc874c3eb7p-1, 0x1.0c9704d5d898fp-1, 0x1.1734d63dedb49p-1,
    0x1.21a799933eb59p-1, 0x1.2bedb25faf3eap-1, 0x1.36058b10659f3p-1, 0x1.3fed9534556d4p-1,
    0x1.49a449b9b0939p-1, 0x1.5328292a35596p-1, 0x1.5c77bbe65018cp-1, 0x1.6591925f0783dp-1,
    0x1.6e74454eaa8afp-1, 0x1.771e75f037261p-1, 0x1.7f8ece3571771p-1, 0x1.87c400fba2ebfp-1,
    0x1.8fbcca3ef940dp-1, 0x1.9777ef4c7d742p-1, 0x1.9ef43ef29af94p-1, 0x1.a63091b02fae2p-1,
    0x1.ad2bc9e21d511p-1, 0x1.b3e4d3ef55712p-1, 0x1.ba5aa673590d2p-1, 0x1.c08c426725549p-1,
    0x1.c678b3488739bp-1, 0x1.cc1f0f3fcfc5cp-1, 0x1.d17e7743e35dcp-1, 0x1.d696173c9e68bp-1,
    0x1.db6526238a09bp-1, 0x1.dfeae622dbe2bp-1, 0x1.e426a4b2bc17ep-1, 0x1.e817bab4cd10dp-1,
    0x1.ebbd8c8df0b74p-1, 0x1.ef178a3e473c2p-1, 0x1.f2252f7763adap-1, 0x1.f4e603b0b2f2dp-1,
    0x1.f7599a3a12077p-1, 0x1.f97f924c9099bp-1, 0x1.fb5797195d741p-1, 0x1.fce15fd6da67bp-1,
    0x1.fe1cafcbd5b09p-1, 0x1.ff095658e71adp-1, 0x1.ffa72effef75dp-1, 0x1.fff62169b92dbp-1,
};

constexpr int kSinCosEntries = 256;

// exp(mu + sigma z) = 2^((mu' + sigma' z) / 256)
struct LogNormal {
    double mu, sigma;            // as given
    double mu_scaled;
    double square;               // sigma'^2, a factor of everything that makes up sigma'^2 (-2 ln u)
    double log_poly[7];          // of r^1 .. r^7, times it

    __host__ static LogNormal make(double mu, double sigma) {
        constexpr double k256_over_ln2 = 0x1.71547652b82fep+8;
        // (a sigma of 0 as one that changes no time but leaves the square root a positive argument)
        const double scaled = (sigma > 1e-100 ? sigma : 1e-100) * k256_over_ln2, square = scaled * scaled;
        return {mu, sigma, mu * k256_over_ln2, square,
                {-2.0 * square, square, -2.0 / 3.0 * square, 0.5 * square, -2.0 / 5.0 * square, 1.0 / 3.0 * square,
                 -2.0 / 7.0 * square}};
    }
    // |z| < 8.7, so exp stays within the normal numbers and the table-driven form applies.
    __host__ static bool tame(double mu, double sigma) { return fabs(mu) + 8.7 * sigma < 700.0; }
};

struct LogNormalTables {
    double2 log[128];                      // c_i, 2 ln c_i sigma'^2
    double2 sin_cos[kSinCosEntries];       // of 2 pi (j + 1/2) / 256
    double exp2[256];
    double exponent[56];                   // 2 ln 2 (54 - j) sigma'^2
};

// Filled by the whole CTA; a barrier has to follow.
__device__ __forceinline__ void fill_tables(LogNormalTables& t, const LogNormal& q) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) {
        t.exp2[i] = kExpTable[i];
        if (i < 128) t.log[i] = make_double2(kLogTable[i].x, kLogTable[i].y * q.square);
        if (i < 56) t.exponent[i] = (54 - i) * 0x1.62e42fefa39efp+0 * q.square;
        const double a = kSinTable[i & 63], b = kSinTable[63 - (i & 63)];
        const double s = i & 64 ? b : a, c = i & 64 ? -a : b;              // second quadrant: cos, -sin
        t.sin_cos[i] = i & 128 ? make_double2(-s, -c) : make_double2(s, c);
    }
}

// 2^(y / 256): y = k + f, |f| <= 1/2, k by adding 1.5 * 2^52.
__device__ __forceinline__ double exp2_256(const LogNormalTables& t, double y) {
    const double shifted = y + 0x1.8p52;
    const int k = __double2loint(shifted);
    const double f = y - (shifted - 0x1.8p52);
    // e^x - 1, x = f ln2 / 256, to x^4 (|x| <= 0.0014: the next term is 4e-17)
    constexpr double kX = 0x1.62e42fefa39efp-9;                          // ln2 / 256
    double p = fma(f, kX * kX * kX * kX / 24.0, kX * kX * kX / 6.0);
    p = fma(p, f, kX * kX / 2.0);
    p = fma(p, f, kX) * f;
    const double e = t.exp2[k & 255];
    const double v = fma(e, p, e);
    return __hiloint2double(__double2hiint(v) + ((k >> 8) << 20), __double2loint(v));
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
    // sigma'^2 (-2 ln u), u = v 2^-53 = m 2^e with m in [0.6875, 1.375), m c_i = 1 + r, |r| <= 2^-7.  Near u = 1 both e
    // and ln c_i vanish and nothing cancels; the 2^-120 kept in their place makes the result positive at u = 1.
    const double v = (double)(wa >> 11) + 0.5;
    const int above = __double2hiint(v) - 0x3FE60000;
    const int e = above >> 20;                                            // -1 .. 53
    const double m = __hiloint2double(__double2hiint(v) - (e << 20), __double2loint(v));
    const double2 cl = t.log[(above >> 13) & 127];
    const double r = fma(m, cl.x, -1.0);
    double p = fma(r, q.log_poly[6], q.log_poly[5]);
    p = fma(p, r, q.log_poly[4]);
    p = fma(p, r, q.log_poly[3]);
    p = fma(p, r, q.log_poly[2]);
    p = fma(p, r, q.log_poly[1]);
    const double x = fma(p, r * r, fma(r, q.log_poly[0], t.exponent[e + 1] + cl.y));
    // sqrt(x): y = x^-1/2 (1 + O(2^-20)), one step of third order
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double h = x * y, d = fma(-h, y, 1.0);
    const double radius = fma(h * d, fma(d, 0.375, 0.5), h);
    // angle: the table entry of the leading 8 bits, turned by the rest, a = pi 2^-53 i (|a| <= pi / 256)
    const uint32_t hi = (uint32_t)(wb >> 32), lo = (uint32_t)wb;
    const double i = __hiloint2double(0x43300000 | ((hi >> 10) & 0x3FFF), __funnelshift_r(lo, hi, 10) | 1) -
                     (0x1.0p52 + 0x1.0p45);
    constexpr double k = 0x1.921fb54442d18p-52;   // pi 2^-53
    const double2 sc = t.sin_cos[hi >> 24];
    const double i2 = i * i;
    const double sa = fma(i2, fma(i2, k * k * k * k * k / 120.0, -k * k * k / 6.0), k) * i;
    const double ca = fma(i2, fma(i2, -k * k * k * k * k * k / 720.0, k * k * k * k / 24.0), -0.5 * k * k) * i2;   // cos a - 1
    const double s = fma(sc.y, sa, fma(sc.x, ca, sc.x));
    const double c = fma(-sc.x, sa, fma(sc.y, ca, sc.y));
    t_cos = exp2_256(t, fma(radius, c, q.mu_scaled));
    t_sin = exp2_256(t, fma(radius, s, q.mu_scaled));
}

// The four times of one block.
template <bool TAME>
__device__ __forceinline__ void lognormal4(const LogNormalTables& t, const Philox4& b, const LogNormal& q, double (&out)[4]) {
    lognormal2<TAME>(t, b.w0, b.w1, q, out[0], out[1]);
    lognormal2<TAME>(t, b.w2, b.w3, q, out[2], out[3]);
}

}  // namespace

}  // namespace nolo
