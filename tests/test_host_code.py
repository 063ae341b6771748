"""Index arithmetic and bookkeeping of the library that needs no GPU, compiled alone with the host compiler."""

from tests.helpers import run_host_code


def test_shifted_copy_stays_inside_its_buffers(tmp_path):
    """Blocks of every small size, element size and pair of source and destination block: every 16-byte load lies in
    the input, and every byte of the block is stored exactly once."""
    run_host_code(tmp_path, r"""
#include "nolo_shifted.h"
#include <cstdio>
#include <cstring>
int main() {
    const uintptr_t in = 1 << 20, out = 1 << 24;
    for (int es = 2; es <= 4; es += 2)
        for (int64_t E = 1; E <= 200; ++E)
            for (int blocks = 1; blocks <= 17; ++blocks)
                for (int from = 0; from < blocks; ++from)
                    for (int to = 0; to < blocks; ++to) {
                        const int64_t bytes = E * es;
                        const uintptr_t end = in + blocks * bytes;
                        const nolo::ShiftedSpan s = nolo::shifted_span(
                            (const unsigned char*)in + from * bytes, (const unsigned char*)out + to * bytes, bytes, (const unsigned char*)end);
                        const uintptr_t first = (uintptr_t)s.from;
                        bool ok = first % 16 == 0 && (s.vecs == 0 || (out + to * bytes + s.head) % 128 == 0);
                        ok &= s.loads == 0 || (first >= in && first + 16 * s.loads <= end);
                        ok &= s.vecs == 0 || s.loads >= s.vecs + (s.shift != 0);      // both parts of every vector
                        ok &= s.head >= 0 && s.head <= 128 && s.vecs >= 0 && s.head + 16 * s.vecs <= bytes;
                        ok &= bytes - s.head - 16 * s.vecs < 32;                      // left to the elements
                        if (!ok) {
                            printf("es %d E %lld: block %d of %d to %d\n", es, (long long)E, from, blocks, to);
                            return 1;
                        }
                    }
    return 0;
}
""")


def test_inner_steps_of_any_int_count(tmp_path):
    """Up to the largest int, by any number of lanes: each lane's loop ends, the blocks hold H steps in all, and no
    signed sum overflows (the sanitizer is on)."""
    run_host_code(tmp_path, r"""
#include "nolo_steps.h"
#include <climits>
#include <cstdio>
int main() {
    for (int i = 0; i < 400; ++i) {
        const int H = i < 200 ? 1 + i : INT_MAX - (i - 200);
        const int blocks = nolo::step_blocks(H);
        long long steps = 0;
        for (int lanes = 1; lanes <= 32; lanes *= 2) {
            steps = 0;
            for (int lane = 0; lane < lanes; ++lane) {
                // the last turns of this lane; all before them have whole blocks
                int k = blocks > 4096 ? (blocks - 1024) / lanes * lanes + lane : lane;
                steps += 4ll * (k / lanes);
                for (; k < blocks; k += lanes) {
                    const int n = nolo::steps_in_block(H, k);
                    if (n < 1 || n > 4 || (n < 4 && k != blocks - 1)) return printf("H %d k %d: %d\n", H, k, n), 1;
                    steps += n;
                }
            }
            if (steps != H) return printf("H %d, %d lanes: %lld\n", H, lanes, steps), 1;
        }
    }
    return 0;
}
""")
