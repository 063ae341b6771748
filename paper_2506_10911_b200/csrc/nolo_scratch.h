// Blocks of device memory kept between calls that have no handle to keep them in (the simulations).
#pragma once

#include <stddef.h>
#include <stdint.h>
#include <string.h>

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

// What one call of a simulation needs, kept for the next one if the call comes to its end: device memory for the trials' values
// and for scratch, and page-locked memory for the results, which are the statistics and, up to kHostValues, the trials' values:
// the last kernel writes them there.  Where the host refuses that much page-locked memory the results stay on the device
// and are copied, as more values than that are.
//
// Memory as above, with a type Stream, Status copy(void* host, const void* device, size_t, Stream), which may return before it is done,
// and Status wait(Stream).
template <typename Memory, typename HostMemory>
class SimScratch {
public:
    using Status = typename Memory::Status;
    using Stream = typename Memory::Stream;
    using Pool = ScratchBlocks<Memory>;
    using HostPool = ScratchBlocks<HostMemory>;
    static constexpr int64_t kHostValues = 1 << 17;
    static constexpr int kMostStats = 4;

    SimScratch(Pool& pool, HostPool& host_pool) : pool_(pool), host_pool_(host_pool) {}
    SimScratch(const SimScratch&) = delete;
    ~SimScratch() {
        if (block_.p) Memory::release(block_.p);
        if (host_.p) HostMemory::release(host_.p);
    }

    // For `values` values and scratch; 1 MB and more, so that small calls of all sizes share blocks.
    Status take(int64_t values, size_t scratch) {
        values_ = values;
        const size_t want = scratch_at() + scratch;
        const Status e = pool_.take(want < (size_t(1) << 20) ? size_t(1) << 20 : want, &block_);
        if (e == Memory::kOk && host_pool_.take(sizeof(double) * (kMostStats + kHostValues), &host_) != HostMemory::kOk) host_.p = nullptr;
        return e;
    }
    // On the device: the values, scratch.
    double* values() const { return static_cast<double*>(block_.p) + kMostStats; }
    void* scratch() const { return static_cast<char*>(block_.p) + scratch_at(); }
    // Where a kernel leaves the statistics, and the values if the caller wants them and they are not copied (else NULL).
    double* stats() const { return static_cast<double*>(host_.p ? host_.p : block_.p); }
    double* values_in_place(bool wanted) const {
        return wanted && host_.p && values_ <= kHostValues ? static_cast<double*>(host_.p) + kMostStats : nullptr;
    }
    // Waits for the results and hands them over; e: how the launches went.
    Status finish(Status e, double* to_values, double* to_stats, int stats_count, Stream s) {
        const double* in_place = values_in_place(to_values != nullptr);
        if (e == Memory::kOk && !host_.p) e = Memory::copy(to_stats, stats(), sizeof(double) * (size_t)stats_count, s);
        if (e == Memory::kOk && to_values && !in_place) e = Memory::copy(to_values, values(), sizeof(double) * (size_t)values_, s);
        const Status end = Memory::wait(s);
        if (e == Memory::kOk) e = end;
        if (e != Memory::kOk) return e;
        if (host_.p) memcpy(to_stats, stats(), sizeof(double) * (size_t)stats_count);
        if (in_place) memcpy(to_values, in_place, sizeof(double) * (size_t)values_);
        pool_.put(block_);
        block_.p = nullptr;
        if (host_.p) host_pool_.put(host_);
        host_.p = nullptr;
        return e;
    }

private:
    size_t scratch_at() const { return sizeof(double) * (size_t)(kMostStats + ((values_ + 1) & ~int64_t(1))); }   // a multiple of 16

    Pool& pool_;
    HostPool& host_pool_;
    typename Pool::Block block_;
    typename HostPool::Block host_;
    int64_t values_ = 0;
};

}  // namespace nolo
