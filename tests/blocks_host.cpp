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
static std::map<void *, std::pair<cudaStream_t, long>> used;
static std::map<void *, size_t> live;             // allocated, in bytes
static std::map<void *, size_t> pool;             // freed, in bytes
static std::map<cudaEvent_t, Clock> events;
static size_t total = 80ull << 30, taken = 0, mallocs = 0, waits = 0, deny = 0;   // deny: allocations to fail
static long next_id = 1;

static void merge(Clock &a, const Clock &b) {
    for (auto &x : b) a[x.first] = std::max(a[x.first], x.second);
}
static bool behind(cudaStream_t s, void *p) {
    if (!used.count(p)) return true;
    const auto u = used[p];
    return known[s][u.first] >= u.second || host[u.first] >= u.second;
}
static void use(cudaStream_t s, void *p) {
    CHECK(live.count(p));
    CHECK(behind(s, p));
    used[p] = {s, ++known[s][s]};
}
static void wait_host(cudaStream_t s) { merge(host, known[s]); }

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
cudaError_t cudaDeviceSynchronize(void) {
    for (auto &k : known) merge(host, k.second);
    return cudaSuccess;
}
}

namespace gsi {
uint64_t device_total_mem(int) { return total; }
}

using namespace gsi;
static cudaStream_t S(long i) { return reinterpret_cast<cudaStream_t>(i); }
constexpr uint64_t MB = 1ull << 20, GB = 1ull << 30;

// A block that stream 1 gave back with work on it.
static void *from_stream_1(uint64_t bytes) {
    void *p = nullptr;
    CHECK(block_get(0, bytes, S(1), &p) == cudaSuccess);
    use(S(1), p);
    block_put(0, p, bytes, S(1), false);
    return p;
}

int main(int, char **argv) {
    const std::string what = argv[1];
    void *p = nullptr, *q = nullptr;
    block_users(0, 1);
    if (what == "abandoned set") {                // its stream waits for stream 1, but nobody has waited for it
        void *b = from_stream_1(GB);
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &p) == cudaSuccess && p == b);
            deny = 1;
            CHECK(set.get(GB, &q) != cudaSuccess);
        }
        deny = 0;
        CHECK(block_get(0, GB, S(3), &q) == cudaSuccess);
        use(S(3), q);
    } else if (what == "failed wait") {
        from_stream_1(GB);
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &p) == cudaSuccess);
            use(S(2), p);
            CHECK(!set.waited(cudaErrorUnknown) && set.busy());
        }
        CHECK(block_get(0, GB, S(3), &q) == cudaSuccess && q == p);
        use(S(3), q);
    } else if (what == "work after the wait") {
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &p) == cudaSuccess);
            use(S(2), p);
            wait_host(S(2));
            CHECK(set.waited(cudaSuccess) && !set.busy());
            set.enqueued();
            use(S(2), p);
        }
        CHECK(block_get(0, GB, S(3), &q) == cudaSuccess && q == p);
        use(S(3), q);
    } else if (what == "second attempt") {        // a retry takes blocks of an attempt that was waited for
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &p) == cudaSuccess);
            use(S(2), p);
            wait_host(S(2));
            set.waited(cudaSuccess);
        }
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &q) == cudaSuccess && q == p);
            use(S(2), q);                         // and ends without a wait
        }
        CHECK(block_get(0, GB, S(3), &q) == cudaSuccess && q == p);
        use(S(3), q);
    } else if (what == "waited for") {            // no event between the two
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &p) == cudaSuccess);
            use(S(2), p);
            wait_host(S(2));
            set.waited(cudaSuccess);
        }
        const size_t before = waits;
        CHECK(block_get(0, GB, S(3), &q) == cudaSuccess && q == p);
        use(S(3), q);
        CHECK(waits == before);
    } else if (what == "taken block") {           // a result keeps it: the set does not give it back
        {
            BlockSet set(0, S(2));
            CHECK(set.get(GB, &p) == cudaSuccess && set.get(GB, &q) == cudaSuccess);
            set.take(p);
        }
        void *r = nullptr, *t = nullptr;
        CHECK(block_get(0, GB, S(2), &r) == cudaSuccess && block_get(0, GB, S(2), &t) == cudaSuccess);
        CHECK(r != p && t != p && live.count(p));
        block_put(0, p, GB, S(2), false);
    } else {
        std::printf("no such case\n");
        return 1;
    }
    std::printf("ok\n");
    return 0;
}
