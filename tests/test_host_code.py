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


SCRATCH = r"""
#include "nolo_scratch.h"
#include <cstdio>
#include <cstdlib>
#include <map>
#include <thread>
#include <vector>
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); exit(1); } } while (0)
struct Fake {
    using Status = int;
    static constexpr int kOk = 0;
    static inline std::mutex m;
    static inline std::map<void*, size_t> held;
    static inline size_t total = 0, room = ~size_t(0);
    static inline int allocations = 0, fail_with = 0;
    static inline thread_local int current = 0;
    static int device(int* d) { *d = current; return 0; }
    static int allocate(void** p, size_t bytes) {
        std::lock_guard<std::mutex> lock(m);
        if (fail_with) return fail_with;
        if (total + bytes > room) return 2;
        *p = malloc(1);
        held[*p] = bytes; total += bytes; ++allocations;
        return 0;
    }
    static bool exhausted(int e) { return e == 2; }
    static void release(void* p) {
        std::lock_guard<std::mutex> lock(m);
        CHECK(held.count(p));
        total -= held[p]; held.erase(p); free(p);
    }
};
using Pool = nolo::ScratchBlocks<Fake>;
const size_t MB = size_t(1) << 20;
void call(Pool& pool, size_t bytes) {
    Pool::Block b;
    CHECK(pool.take(bytes, &b) == 0 && b.p && b.bytes >= bytes);
    { std::lock_guard<std::mutex> lock(Fake::m); CHECK(Fake::held[b.p] == b.bytes); }
    pool.put(b);
}
"""


def test_scratch_keeps_its_bound_and_its_blocks(tmp_path):
    run_host_code(tmp_path, SCRATCH + r"""
int main() {
    {   // a large block lent to small calls is a large block still
        Pool pool;
        for (int i = 0; i < 40; ++i) {
            call(pool, 40 * MB);
            call(pool, (1 + i % 3) * MB);
            CHECK(Fake::total <= Pool::kMostBytes);
        }
        CHECK(Fake::allocations == 1);
        // ... also to small calls that overlap
        Pool::Block b[4];
        for (int turn = 0; turn < 10; ++turn) {
            for (Pool::Block& x : b) CHECK(pool.take(MB, &x) == 0);
            for (Pool::Block& x : b) pool.put(x);
            CHECK(Fake::total <= Pool::kMostBytes);
        }
        CHECK(Fake::allocations == 4);
        pool.give_back();
        CHECK(Fake::total == 0);
    }
    {   // growing sizes: the largest, repeated, is not allocated again
        Pool pool;
        for (size_t mb = 1; mb <= 32; mb *= 2) { call(pool, mb * MB); CHECK(Fake::total <= Pool::kMostBytes); }
        call(pool, 33 * MB);
        const int before = Fake::allocations;
        for (int i = 0; i < 5; ++i) call(pool, 33 * MB);
        CHECK(Fake::allocations == before && Fake::total <= Pool::kMostBytes);
        call(pool, Pool::kMostBytes);
        CHECK(Fake::total == Pool::kMostBytes);
        call(pool, Pool::kMostBytes + 1);            // not kept
        CHECK(Fake::total == Pool::kMostBytes);
        pool.give_back();
        CHECK(Fake::total == 0);
    }
    {   // another device finds room, and never the first one's blocks
        Pool pool;
        for (int mb = 10; mb <= 16; mb += 2) call(pool, mb * MB);
        Fake::current = 1;
        call(pool, MB);
        const int before = Fake::allocations;
        for (int i = 0; i < 5; ++i) call(pool, MB);
        CHECK(Fake::allocations == before);
        Fake::current = 0;
        call(pool, 16 * MB);
        CHECK(Fake::allocations == before);
        pool.give_back();
    }
    {   // where memory is short what is kept goes first; other errors are passed on
        Pool pool;
        call(pool, 10 * MB);
        call(pool, 20 * MB);
        Fake::room = 40 * MB;
        call(pool, 35 * MB);
        CHECK(Fake::total == 35 * MB);
        Pool::Block b;
        CHECK(pool.take(41 * MB, &b) == 2 && !b.p);
        Fake::room = ~size_t(0);
        Fake::fail_with = 5;
        CHECK(pool.take(MB, &b) == 5 && !b.p);
        Fake::fail_with = 0;
        pool.give_back();
    }
    {   // threads
        Pool pool;
        std::vector<std::thread> threads;
        for (int t = 0; t < 8; ++t)
            threads.emplace_back([&pool, t] {
                Fake::current = t & 1;
                for (int i = 0; i < 2000; ++i) {
                    call(pool, (1 + (i * 7 + t) % 40) * MB);
                    if (i % 100 == 0) pool.give_back();
                }
            });
        for (std::thread& t : threads) t.join();
        CHECK(Fake::total <= Pool::kMostBytes);
        pool.give_back();
        CHECK(Fake::total == 0);
    }
    return 0;
}
""")


def test_units_of_the_straggler_simulation_are_filled(tmp_path):
    """However many trials leave a slab however few iterations, at most an eighth of the threads is idle, but for the last
    unit; and the units cover the items."""
    run_host_code(tmp_path, r"""
#include "nolo_steps.h"
#include <cstdio>
#include <initializer_list>
int main() {
    const int threads = 256;
    for (int W = 4; W <= 4096; W += W < 300 ? 1 : 37)
        for (int iterations = 1; iterations <= 60; iterations += iterations < 9 ? 1 : 7)
            for (long long trials : {1ll, 2ll, 3ll, 50ll, 700ll, 20000ll}) {
                const int64_t work = (int64_t)W * iterations * trials;
                if (work > 1 << 21) continue;
                const nolo::WorkUnits u = nolo::WorkUnits::of(W, iterations, trials, threads);
                const int64_t laid = u.count * threads;
                bool ok = 7 * laid <= 8 * work + 7 * threads;
                ok &= u.items == (int64_t)W * iterations * (u.across ? trials : 1);
                ok &= u.chunks * threads >= u.items && (u.chunks - 1) * threads < u.items;
                ok &= u.count == u.chunks * (u.across ? 1 : trials);
                if (!ok) return printf("W %d, %d iterations, %lld trials: %lld threads for %lld items\n", W, iterations, trials,
                                       (long long)laid, (long long)work), 1;
            }
    return 0;
}
""")


def test_simulations_do_without_page_locked_memory(tmp_path):
    """Results are left in page-locked memory where there is some, else on the device and copied; the caller gets the
    same, and either kind of block is kept or released once."""
    run_host_code(tmp_path, SCRATCH + r"""
#include <cstring>
struct Device : Fake {
    using Stream = int;
    struct Copy { void* to; const void* from; size_t bytes; };
    static inline std::vector<Copy> pending;
    static inline int copies = 0, wait_fails = 0;
    static int allocate(void** p, size_t bytes) {
        *p = calloc(1, bytes);
        held[*p] = bytes; total += bytes;
        return 0;
    }
    static int copy(void* to, const void* from, size_t bytes, int) { pending.push_back({to, from, bytes}); ++copies; return 0; }
    static int wait(int) {
        for (const Copy& c : pending) memcpy(c.to, c.from, c.bytes);
        pending.clear();
        return wait_fails;
    }
};
struct Host : Device {
    static inline int refuses = 0;
    static int device(int* d) { *d = 0; return 0; }
    static int allocate(void** p, size_t bytes) { return refuses ? refuses : Device::allocate(p, bytes); }
};
using Sim = nolo::SimScratch<Device, Host>;
int main() {
    nolo::ScratchBlocks<Device> pool;
    nolo::ScratchBlocks<Host> host_pool;
    const int64_t most = Sim::kHostValues;
    for (int refuses : {0, 2, 5})                       // 2: exhausted, 5: any other error
        for (int64_t values : {int64_t(1), int64_t(7), most, most + 1, 3 * most})
            for (int wanted = 0; wanted < 2; ++wanted)
                for (int fails : {0, 7, 8}) {           // 7: of the launches, 8: of the wait
                    pool.give_back();
                    host_pool.give_back();
                    CHECK(Fake::total == 0);
                    Host::refuses = refuses;
                    Device::copies = 0;
                    std::vector<double> got(values, -1.0), stats(4, -1.0);
                    {
                        Sim s(pool, host_pool);
                        CHECK(s.take(values, 1000) == 0);
                        CHECK((uintptr_t)s.values() % 16 == 0 && (uintptr_t)s.scratch() % 16 == 0);
                        CHECK((char*)s.scratch() >= (char*)(s.values() + values));
                        double* in_place = s.values_in_place(wanted);
                        CHECK((in_place != nullptr) == (wanted && !refuses && values <= most));
                        for (int64_t i = 0; i < values; ++i) s.values()[i] = 0.5 * i;
                        for (int64_t i = 0; in_place && i < values; ++i) in_place[i] = 0.5 * i;
                        memset(s.scratch(), 255, 1000);
                        for (int i = 0; i < 3; ++i) s.stats()[i] = 10.0 + i;
                        Device::wait_fails = fails == 8 ? 8 : 0;
                        CHECK(s.finish(fails == 7 ? 7 : 0, wanted ? got.data() : nullptr, stats.data(), 3, 0) == fails);
                        Device::wait_fails = 0;
                    }
                    if (fails) {
                        CHECK(Fake::total == 0);        // nothing of a call that failed is kept
                        continue;
                    }
                    CHECK(stats == std::vector<double>({10.0, 11.0, 12.0, -1.0}));
                    for (int64_t i = 0; i < values; ++i) CHECK(got[i] == (wanted ? 0.5 * i : -1.0));
                    CHECK(Device::copies == (refuses != 0) + (wanted && (refuses || values > most)));
                    const size_t kept = Fake::total;
                    Sim again(pool, host_pool);
                    CHECK(again.take(values, 1000) == 0 && Fake::total == kept);
                }
    pool.give_back();
    host_pool.give_back();
    CHECK(Fake::total == 0);
    return 0;
}
""")
