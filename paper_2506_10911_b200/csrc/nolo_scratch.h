// Blocks of device memory kept between calls that have no handle to keep them in (the simulations).
#pragma once

#include <stddef.h>

#include <mutex>

namespace nolo {

// A few blocks, at most kBlocks of kMostBytes in all, each used by one call at a time and put back when the GPU is done
// with it.  A block keeps its size, whatever the call that had it asked for.  Where a block that is put back
// finds no room, those that have lain longest make it.
//
// Memory: static functions  Status device(int*), Status allocate(void**, size_t), bool exhausted(Status),
// void release(void*), and the Status kOk.
template <typename Memory>
class ScratchBlocks {
public:
    using Status = typename Memory::Status;
    static constexpr int kBlocks = 4;
    static constexpr size_t kMostBytes = size_t(64) << 20;
    struct Block {
        void* p = nullptr;
        size_t bytes = 0;
        int device = 0;
        unsigned long long put = 0;      // when it was put back
    };

    // The smallest kept block of the current device that will do, else a new one.
    Status take(size_t bytes, Block* out) {
        int device = 0;
        Status e = Memory::device(&device);
        if (e != Memory::kOk) return e;
        {
            std::lock_guard<std::mutex> lock(mutex_);
            Block* best = nullptr;
            for (Block& b : blocks_)
                if (b.p && b.device == device && b.bytes >= bytes && (!best || b.bytes < best->bytes)) best = &b;
            if (best) {
                *out = *best;
                remove(*best);
                return Memory::kOk;
            }
        }
        out->bytes = bytes;
        out->device = device;
        e = Memory::allocate(&out->p, bytes);
        if (Memory::exhausted(e)) {
            give_back();
            e = Memory::allocate(&out->p, bytes);
        }
        if (e != Memory::kOk) out->p = nullptr;
        return e;
    }

    // b was taken here and is no longer in use on the GPU.
    void put(const Block& b) {
        void* out[kBlocks + 1];
        int count = 0;
        if (b.bytes > kMostBytes) {
            out[count++] = b.p;
        } else {
            std::lock_guard<std::mutex> lock(mutex_);
            for (;;) {
                Block *room = nullptr, *oldest = nullptr;
                for (Block& k : blocks_) {
                    if (!k.p) room = &k;
                    else if (!oldest || k.put < oldest->put) oldest = &k;
                }
                if (room && kept_ + b.bytes <= kMostBytes) {
                    *room = b;
                    room->put = ++clock_;
                    kept_ += b.bytes;
                    break;
                }
                out[count++] = oldest->p;
                remove(*oldest);
            }
        }
        for (int i = 0; i < count; ++i) Memory::release(out[i]);
    }

    void give_back() {
        void* out[kBlocks];
        {
            std::lock_guard<std::mutex> lock(mutex_);
            for (int i = 0; i < kBlocks; ++i) {
                out[i] = blocks_[i].p;
                if (out[i]) remove(blocks_[i]);
            }
        }
        for (void* p : out)
            if (p) Memory::release(p);
    }

private:
    void remove(Block& b) {
        kept_ -= b.bytes;
        b = Block();
    }

    std::mutex mutex_;
    Block blocks_[kBlocks];
    size_t kept_ = 0;
    unsigned long long clock_ = 0;
};

}  // namespace nolo
