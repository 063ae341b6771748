"""The table-driven log-normal times of the simulations, word by word, against extended precision."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2506_10911_b200 import build

pytestmark = pytest.mark.gpu

PROBE = r"""
#include "nolo_lognormal.cuh"
#include <cmath>
template <bool TAME>
__global__ void times(const uint64_t* wa, const uint64_t* wb, int count, nolo::LogNormal q, double2* out) {
    __shared__ nolo::LogNormalTables tables;
    nolo::fill_tables(tables, q);
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    double c, s;
    nolo::lognormal2<TAME>(tables, wa[i], wb[i], q, c, s);
    out[i] = make_double2(c, s);
}
extern "C" int run(const void* wa, const void* wb, int count, double mu, double sigma, void* out) {
    if (!nolo::LogNormal::tame(mu, sigma)) return -1;
    times<true><<<(count + 255) / 256, 256>>>((const uint64_t*)wa, (const uint64_t*)wb, count, nolo::LogNormal::make(mu, sigma),
                                              (double2*)out);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    d = tmp_path_factory.mktemp("lognormal")
    (d / "probe.cu").write_text(PROBE)
    subprocess.run([build.find_nvcc(), *build.NVCC_FLAGS, "-I", os.path.join(build.HERE, "csrc"), "-o", str(d / "probe.so"),
                    str(d / "probe.cu")], check=True)
    fn = ctypes.CDLL(str(d / "probe.so")).run
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_void_p]
    return fn


def words(sigma):
    """Both ends of every interval of the tables (of the power table next to them), the ends of the whole range, and random words."""
    rng = np.random.default_rng(3)
    radius, angle = [0, 1, 2, 3, 2**53 - 1, 2**53 - 2, 2**53 - 3], [0, 1, 2**53 - 1]
    # u = m 2^(e - 53), m at the ends of the logarithm's 512 intervals of [0.6875, 1.375), which are 2^-10 wide below 1
    ends = [0.6875 + j / 1024 for j in range(320)] + [1.0 + j / 512 for j in range(193)]
    for e in range(54):
        radius += [int(m * 2.0**e) + d for m in ends for d in (-1, 0, 1)]
    for j in range(1, 129):                                     # u next to 1, where nothing may cancel
        radius += [2**53 - j, 2**53 - (j << 40), 2**53 - (j << 45)]
    for j in range(513):                                        # the 512 entries of sine and cosine
        angle += [(j << 44) + d for d in (-1, 0, 1)]
        angle += [(j << 44) + (1 << 43) + d for d in (-1, 0, 1)]      # the middle of the entry
    radius = np.unique(np.array([x for x in radius if 0 <= x < 2**53], dtype=np.uint64))
    angle = np.array([x for x in angle if 0 <= x < 2**53], dtype=np.uint64)
    # sigma r half-way between two entries of the power table, 2^(1 / 2048) apart, at angles 0 and pi: of each sign
    half = (np.arange(0, 8.5 * sigma * 2048 / np.log(2), max(1.0, sigma)) + 0.5) * np.log(2) / 2048 / sigma
    half = (np.exp(-0.5 * half * half) * 2.0**53).astype(np.uint64)
    n = 1 << 19
    assert max(len(radius), 2 * len(half)) <= n // 4
    wa = rng.integers(0, 2**53, n, dtype=np.uint64)
    wb = rng.integers(0, 2**53, n, dtype=np.uint64)
    wa[:len(radius)] = radius
    wa[n // 4:n // 4 + len(radius)], wb[n // 4:n // 4 + len(radius)] = radius, rng.choice(angle, len(radius))
    wb[n // 2:n // 2 + len(angle)] = angle
    for at, turn in ((3 * n // 4, 0), (7 * n // 8, 2**52)):
        wa[at:at + len(half)], wb[at:at + len(half)] = half, turn
    low = rng.integers(0, 2**11, n, dtype=np.uint64)            # the bits that are not used
    return (wa << np.uint64(11)) | low, (wb << np.uint64(11)) | low


@pytest.mark.parametrize("mu,sigma", [(0.0, 1.0), (1.0, 0.5**0.5), (0.0, 0.1), (-3.0, 2.5), (0.5, 1e-9), (300.0, 40.0), (0.0, 80.0)])
def test_times_are_good_to_a_few_units_in_the_last_place(probe, mu, sigma):
    wa, wb = words(sigma)
    a, b = (torch.from_numpy(x.view(np.int64)).cuda() for x in (wa, wb))
    out = torch.empty((len(wa), 2), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert probe(a.data_ptr(), b.data_ptr(), len(wa), mu, sigma, out.data_ptr()) == 0
    got = out.cpu().numpy()
    L = np.longdouble
    assert np.finfo(L).eps < 2e-19
    u = (wa >> np.uint64(11)).astype(np.float64) + 0.5             # rounded to float64 (1 for the last word)
    v = (wb >> np.uint64(11)).astype(L) + L(0.5)                   # exact
    r = np.sqrt(-2 * np.log(u.astype(L) * L(2) ** -53))
    # the angle 2 pi v 2^-53, reduced exactly to an eighth of a turn before pi comes in
    turn = v * L(2) ** -53
    octant = np.floor(turn * 8 + L(0.5))
    rest = (turn - octant / 8) * 8 * np.arctan(L(1))
    q = octant.astype(np.int64) % 8
    half = np.sqrt(L(0.5))
    cos8, sin8 = np.array([1, half, 0, -half, -1, -half, 0, half], dtype=L), np.array([0, half, 1, half, 0, -half, -1, -half], dtype=L)
    c = cos8[q] * np.cos(rest) - sin8[q] * np.sin(rest)
    s = sin8[q] * np.cos(rest) + cos8[q] * np.sin(rest)
    # Units of 2^-53: the radius is good to 3 (logarithm and square root), sine and cosine to 2 of 1; the exponent is
    # formed from sigma scaled to units of ln 2 / 2048 (2 for the scaled value, 1 for the sum), and each unit
    # of it is a unit of the time relative to 1; the power itself, e^mu 2^(j / 2048) from a table, is good to 3.
    for k, trig in ((0, c), (1, s)):
        want = np.exp(L(mu) + L(sigma) * (r * trig))
        unit = 2.0 ** -53 * (3 + 8 * sigma * np.maximum(r, 1e-30).astype(np.float64))
        err = np.abs((got[:, k].astype(L) - want) / want).astype(np.float64)
        worst = int(np.argmax(err / unit))
        assert (err <= unit).all(), (hex(wa[worst]), hex(wb[worst]), err[worst] / unit[worst])
        print(f"mu {mu} sigma {sigma}: largest error {err.max():.2e}, of its bound {(err / unit).max():.2f}")
