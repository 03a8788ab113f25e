// The kept arena blocks (csrc/blocks.cu) on a made-up CUDA runtime that knows which work is ordered behind which: every
// stream counts its operations, an event carries what its stream had and had waited for, and a use, a release or a hand-out
// of memory that is not ordered behind the memory's last use ends the program.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "blocks.h"

#define CHECK(c)                                                                     \
    do {                                                                             \
        if (!(c)) {                                                                  \
            std::printf("line %d: %s\n", __LINE__, #c);                              \
            std::exit(1);                                                            \
        }                                                                            \
    } while (0)

using Clock = std::map<cudaStream_t, long>;
static std::map<cudaStream_t, Clock> known;       // what each stream is ordered behind, itself included
static Clock host;                                // what the host has waited for
static Clock ended;                               // what has ended on the device
static std::map<void *, std::pair<cudaStream_t, long>> used;
static std::map<void *, size_t> live;             // allocated, in bytes
static std::map<void *, size_t> pool;             // freed, in bytes
static std::map<cudaEvent_t, Clock> events;
static size_t total = 80ull << 30, taken = 0, mallocs = 0, waits = 0, created = 0, deny = 0;   // deny: allocations to fail
static long next_id = 1;

static void merge(Clock &a, const Clock &b) {
    for (auto &x : b) a[x.first] = std::max(a[x.first], x.second);
}
static bool behind(cudaStream_t s, void *p) {
    if (!used.count(p)) return true;
    const auto u = used[p];
    return known[s][u.first] >= u.second || host[u.first] >= u.second || ended[u.first] >= u.second;
}
static void use(cudaStream_t s, void *p) {
    CHECK(live.count(p));
    CHECK(behind(s, p));
    used[p] = {s, ++known[s][s]};
}
static void end(cudaStream_t s) { merge(ended, known[s]); }
static void wait_host(cudaStream_t s) {
    end(s);
    merge(host, known[s]);
}

extern "C" {
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) {
    ++mallocs;
    if (deny && deny--) return cudaErrorMemoryAllocation;
    if (taken + n > total) return cudaErrorMemoryAllocation;
    *p = reinterpret_cast<void *>(next_id++ << 40);
    live[*p] = n;
    taken += n;
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t s) {
    CHECK(live.count(p));
    CHECK(behind(s, p));
    taken -= live[p];
    live.erase(p);
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    ++created;
    *e = reinterpret_cast<cudaEvent_t>(next_id++);
    events[*e];
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    CHECK(events.erase(e) == 1);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
    CHECK(events.count(e));
    events[e] = known[s];
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
    CHECK(events.count(e));
    merge(known[s], events[e]);
    ++waits;
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) {
    CHECK(events.count(e));
    for (auto &x : events[e])
        if (ended[x.first] < x.second && host[x.first] < x.second) return cudaErrorNotReady;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(enum cudaStreamCaptureMode *m) {
    static cudaStreamCaptureMode now = cudaStreamCaptureModeGlobal;
    std::swap(now, *m);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(1000);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    merge(ended, known[s]);
    merge(host, known[s]);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) {
    for (auto &k : known) merge(host, k.second);
    return cudaSuccess;
}
}

namespace gsi {
uint64_t device_total_mem(int) { return total; }
cudaStream_t library_stream(int) { return reinterpret_cast<cudaStream_t>(9); }
}

using namespace gsi;
static cudaStream_t S(long i) { return reinterpret_cast<cudaStream_t>(i); }
constexpr uint64_t MB = 1ull << 20, GB = 1ull << 30;

static Block get(cudaStream_t s, uint64_t bytes) {
    Block b;
    CHECK(block_get(0, bytes, s, &b) == cudaSuccess && b.bytes >= bytes && live[b.p] == b.bytes);
    return b;
}
// A block that a stream (the library's, unless said otherwise) gave back with work on it.
static void *given_back(uint64_t bytes, cudaStream_t s = S(9)) {
    const Block b = get(s, bytes);
    use(s, b.p);
    block_put(0, b, s, false);
    return b.p;
}

int main(int, char **argv) {
    const std::string what = argv[1];
    Block a, b, c;
    block_users(0, 1);
    // first, sets that end with work on stream 2, be it a wait for the library's stream: stream 3 asks next, and may not have
    // the block before that work has ended
    if (what == "abandoned set") {
        void *p = given_back(GB);
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &a) == cudaSuccess && a.p == p);
            deny = 1;
            CHECK(set.get(GB, &b) != cudaSuccess);
        }
        deny = 0;
        b = get(S(3), GB);
        CHECK(b.p != p);
        use(S(3), b.p);
        end(S(9));
        end(S(2));
        use(S(3), (c = get(S(3), GB)).p);
        CHECK(c.p == p);
    } else if (what == "failed wait") {
        void *p = given_back(GB);
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &a) == cudaSuccess && a.p == p);
            use(S(2), a.p);
            CHECK(!set.waited(cudaErrorUnknown) && set.busy());
        }
        use(S(3), (b = get(S(3), GB)).p);
        CHECK(b.p != p);
        use(S(2), get(S(2), GB).p);
    } else if (what == "work after the wait") {
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &a) == cudaSuccess);
            use(S(2), a.p);
            wait_host(S(2));
            CHECK(set.waited(cudaSuccess) && !set.busy());
            set.enqueued();
            use(S(2), a.p);
        }
        use(S(3), (b = get(S(3), GB)).p);
        CHECK(b.p != a.p);
    } else if (what == "second attempt") {        // a retry takes blocks of an attempt that was waited for
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &a) == cudaSuccess);
            use(S(2), a.p);
            wait_host(S(2));
            set.waited(cudaSuccess);
        }
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &b) == cudaSuccess && b.p == a.p);
            use(S(2), b.p);                       // and ends without a wait
        }
        use(S(3), (b = get(S(3), GB)).p);
        CHECK(b.p != a.p);
    } else if (what == "another stream's work") {  // a block is not waited for, be it the only one, but on its own stream
        void *p = given_back(GB, S(1));
        const size_t before = waits;
        a = get(S(2), GB);
        CHECK(a.p != p && waits == before);
        b = get(S(1), GB);
        CHECK(b.p == p);
        use(S(1), p);
        block_put(0, b, S(1), false);
        end(S(1));                                // it has ended: anyone's
        CHECK(get(S(2), GB).p == p);
        use(S(2), p);
    } else if (what == "the library's stream") {  // nothing is held up there: its blocks are waited for
        void *p = given_back(GB);
        a = get(S(2), GB);
        CHECK(a.p == p);
        use(S(2), p);
    } else if (what == "given back to the pool") {   // behind its last use, without making the caller's stream wait for it
        given_back(GB, S(1));
        given_back(3 * GB, S(1));
        a = get(S(2), GB);                        // neither is taken
        CHECK(block_trim(0, false) == 4 * GB && live.size() == 1);
        CHECK(known[S(2)][S(1)] == 0 && known[S(9)][S(1)] == 0);
    } else if (what == "waited for") {            // no event between the two
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &a) == cudaSuccess);
            use(S(2), a.p);
            wait_host(S(2));
            set.waited(cudaSuccess);
        }
        const size_t before = waits;
        b = get(S(3), GB);
        CHECK(b.p == a.p && waits == before);
        use(S(3), b.p);
    } else if (what == "taken block") {           // a result keeps it: the set does not give it back
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &a) == cudaSuccess && set.get(GB, &b) == cudaSuccess);
            set.take(a.p);
        }
        CHECK(get(S(2), GB).p == b.p && get(S(2), GB).p != a.p && live.count(a.p));
        block_put(0, a, S(2), false);
    } else if (what == "near size") {             // taken, with its own size; not one half as large again or more
        a = get(S(1), 3 * GB);
        block_put(0, a, S(1), true);
        b = get(S(1), 2 * GB);
        CHECK(b.p == a.p && b.bytes == 3 * GB);
        block_put(0, b, S(1), true);
        CHECK(get(S(1), 2 * GB - 1).p != a.p);
        CHECK(live.count(a.p) && get(S(1), 3 * GB + 1).p != a.p && !live.count(a.p));     // the larger one replaces it
    } else if (what == "smallest that fits") {
        Block x[3];
        for (int i = 0; i < 3; ++i) x[i] = get(S(1), (24 + 4 * ((i + 1) % 3)) * GB / 8);     // 3.5, 4, 3
        for (Block &k : x) block_put(0, k, S(1), true);
        CHECK(get(S(1), 3 * GB).p == x[2].p && get(S(1), 3 * GB).p == x[0].p && get(S(1), 3 * GB).p == x[1].p);
    } else if (what == "idle first") {            // a larger idle block goes before one with work on it
        a = get(S(9), GB);
        b = get(S(9), GB + 64 * MB);
        block_put(0, b, S(9), true);
        use(S(9), a.p);
        block_put(0, a, S(9), false);
        const size_t before = waits;
        CHECK(get(S(2), GB).p == b.p && waits == before);
        c = get(S(2), GB);
        CHECK(c.p == a.p && waits == before + 1);
        use(S(2), c.p);
    } else if (what == "changing budgets") {      // no two calls of one size: what is kept stays a few blocks
        size_t most = 0;
        for (uint64_t i = 0; i < 400; ++i) {
            const uint64_t bytes = 64 * MB + (i * 7919 % 400) * 2 * MB;
            BlockSet set(0, S(1));
            for (Block *k : {&a, &b, &c}) CHECK(set.get(bytes, k) == cudaSuccess && k->bytes <= bytes + bytes / 2);
            set.waited(cudaSuccess);
            most = std::max(most, live.size());
        }
        // no two of a call's three blocks are kept in sizes nearer than half as large again, and from 64 to 862 MB there
        // are at most seven such sizes
        CHECK(most <= 3 * 7);
        CHECK(mallocs <= 3 * 400 / 10);
    } else if (what == "passed over") {           // sizes that nobody asks for any more go back to the pool
        for (uint64_t i = 0; i < 10; ++i) a = get(S(1), (2 + 2 * i) * GB / 2 + GB), block_put(0, a, S(1), true);
        for (uint64_t i = 0; i <= 2 * KEPT_TURNS; ++i) {
            b = get(S(1), 100 * MB);
            block_put(0, b, S(1), true);
        }
        c = get(S(1), 300 * MB);                  // the miss on which they go
        CHECK(live.size() == 2);
    } else if (what == "a quarter of the memory") {
        total = 16 * GB;
        Block x[6];
        for (Block &k : x) k = get(S(1), GB);
        use(S(1), x[0].p);
        for (Block &k : x) block_put(0, k, S(1), false);
        CHECK(live.size() == 4 && !live.count(x[0].p) && !live.count(x[1].p));     // the oldest two went
        a = get(S(1), 5 * GB);
        block_put(0, a, S(1), true);              // larger than the share: not kept
        CHECK(live.size() == 4);
    } else if (what == "number of blocks") {
        total = 1024 * GB;
        std::vector<Block> x(KEPT_MOST + 3);
        for (Block &k : x) k = get(S(1), 64 * MB);
        for (Block &k : x) block_put(0, k, S(1), true);
        CHECK(live.size() == (size_t)KEPT_MOST && !live.count(x[2].p) && live.count(x[3].p));
    } else if (what == "small ones") {            // left to the pool
        a = get(S(1), 64 * MB - 1);
        block_put(0, a, S(1), true);
        CHECK(live.empty());
    } else if (what == "out of memory") {         // any failed allocation gives the kept blocks back and tries again
        total = 8 * GB;
        given_back(GB);
        given_back(GB + GB / 8);
        void *p = nullptr;
        CHECK(device_alloc(&p, 7 * GB, S(2)) == cudaSuccess && live.size() == 1);
        CHECK(device_alloc(&p, 2 * GB, S(2)) == cudaErrorMemoryAllocation);
    } else if (what == "trim") {
        given_back(GB);
        a = get(S(2), 5 * GB);
        block_put(0, a, S(2), true);
        CHECK(block_trim(0, true) == 6 * GB && live.empty() && block_trim(0, true) == 0);
    } else if (what == "events") {                // made for the first blocks only, and never more than there are blocks
        for (int i = 0; i < 300; ++i) {
            Block x[3];
            for (Block &k : x) use(S(1 + i % 3), (k = get(S(1 + i % 3), GB)).p);
            for (Block &k : x) block_put(0, k, S(1 + i % 3), false);
            end(S(1 + i % 3));
            if (i % 100 == 99) block_trim(0, false);
        }
        CHECK(events.size() == 3 && created == 3);
    } else if (what == "last graph") {            // nothing is kept without one; a result that outlives it frees its block
        block_users(0, 1);
        a = get(S(1), GB);
        given_back(GB);
        wait_host(S(1));                          // a graph goes with the device idle
        block_users(0, -1);
        CHECK(live.size() == 2);
        block_users(0, -1);
        CHECK(live.size() == 1);
        block_put(0, a, S(1), false);
        CHECK(live.empty() && events.empty());
    } else {
        std::printf("no such case\n");
        return 1;
    }
    std::printf("ok\n");
    return 0;
}
