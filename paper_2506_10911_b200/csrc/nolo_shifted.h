// Which bytes of a block are moved how by the copy of blocks that begin anywhere (nolo_route.cu).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define NOLO_BOTH __host__ __device__ __forceinline__
#else
#define NOLO_BOTH inline
#endif

namespace nolo {

constexpr int kLine = 128;

// The block's bytes [0, head) and [head + 16 vecs, bytes) go one element at a time, at most 124 and 30 of them; the
// vecs 16-byte vectors between are stored from the destination's first 128-byte line on, so that no two warps share
// one, and put together from the aligned source vectors from[0 .. loads).  No vector that is loaded reaches
// beyond in_end; one that would leaves its bytes to the elements.
struct ShiftedSpan {
    int64_t head, vecs, loads;
    int shift;                 // of the source from the vectors' boundary
    const unsigned char* from;
};

NOLO_BOTH ShiftedSpan shifted_span(const unsigned char* src, const unsigned char* dst, int64_t bytes, const unsigned char* in_end) {
    ShiftedSpan s;
    s.head = (kLine - (reinterpret_cast<uintptr_t>(dst) & (kLine - 1))) & (kLine - 1);
    if (s.head > bytes) s.head = bytes;
    s.shift = (int)(reinterpret_cast<uintptr_t>(src + s.head) & 15);
    s.from = src + s.head - s.shift;
    const int second = s.shift != 0;               // a vector straddles two of the source
    const int64_t inside = (in_end - s.from) / 16 - second;
    s.vecs = (bytes - s.head) / 16;
    if (s.vecs > inside) s.vecs = inside > 0 ? inside : 0;        // one less, at the end of the whole input
    s.loads = s.vecs > 0 ? s.vecs + second : 0;
    return s;
}

}  // namespace nolo
