// Threads that come and go (csrc/thread_kit.cu) on a made-up CUDA runtime that counts what they are given.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <set>
#include <thread>
#include <vector>

#include "thread_kit.h"

#define CHECK(c)                                             \
    do {                                                     \
        if (!(c)) {                                          \
            std::printf("line %d: %s\n", __LINE__, #c);      \
            std::exit(1);                                    \
        }                                                    \
    } while (0)

static std::atomic<long> pinned{0}, events{0};
extern "C" {
cudaError_t cudaMallocHost(void **p, size_t n) {
    ++pinned;
    *p = std::malloc(n);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    *e = reinterpret_cast<cudaEvent_t>(++events);
    return cudaSuccess;
}
}

int main() {
    using namespace gsi;
    for (int i = 0; i < 200; ++i)                     // one after another
        std::thread([] { CHECK(thread_pinned() && thread_pinned() == thread_pinned() && thread_event(0) == thread_event(0)); }).join();
    CHECK(pinned == 1 && events == 1);
    for (int round = 0; round < 20; ++round) {        // eight at a time: none shares
        std::mutex mu;
        std::set<void *> mine, ev;
        std::atomic<int> in{0};
        std::vector<std::thread> t;
        for (int i = 0; i < 8; ++i)
            t.emplace_back([&] {
                void *p = thread_pinned(), *e = thread_event(0);
                {
                    std::lock_guard<std::mutex> lk(mu);
                    CHECK(p && e && mine.insert(p).second && ev.insert(e).second);
                }
                ++in;
                while (in < 8) std::this_thread::yield();     // all eight hold theirs
            });
        for (auto &x : t) x.join();
    }
    CHECK(pinned == 8 && events == 8);
    CHECK(thread_event(1) != thread_event(0) && !thread_event(-1) && !thread_event(64));
    std::printf("ok\n");
    return 0;
}
