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
