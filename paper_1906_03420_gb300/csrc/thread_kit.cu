// What a host thread keeps between its calls (see thread_kit.h).
#include "thread_kit.h"

#include <mutex>
#include <new>

namespace gsi {
namespace {

struct Kit {
    unsigned char *pinned = nullptr;
    cudaEvent_t ev[64] = {};
    Kit *next = nullptr;             // of the kits that no thread has
};
struct Kits {
    std::mutex mu;
    Kit *unused = nullptr;
};
Kits &kits() {                       // never destroyed: threads may outlive static objects
    static Kits *const k = new Kits;
    return *k;
}

struct Holder {
    Kit *kit = nullptr;
    ~Holder() {
        if (!kit) return;
        Kits &k = kits();
        std::lock_guard<std::mutex> lk(k.mu);
        kit->next = k.unused;
        k.unused = kit;
    }
};

Kit *thread_kit() {
    static thread_local Holder h;
    if (!h.kit) {
        Kits &k = kits();
        std::lock_guard<std::mutex> lk(k.mu);
        if (k.unused) {
            h.kit = k.unused;
            k.unused = h.kit->next;
        } else {
            h.kit = new (std::nothrow) Kit;
        }
    }
    return h.kit;
}

}  // namespace

unsigned char *thread_pinned() {
    Kit *const k = thread_kit();
    if (!k) return nullptr;
    if (!k->pinned && cudaMallocHost(reinterpret_cast<void **>(&k->pinned), PINNED_READ + PINNED_STAGE) != cudaSuccess)
        k->pinned = nullptr;
    return k->pinned;
}

cudaEvent_t thread_event(int dev) {
    Kit *const k = dev >= 0 && dev < 64 ? thread_kit() : nullptr;
    if (!k) return nullptr;
    if (!k->ev[dev] && cudaEventCreateWithFlags(&k->ev[dev], cudaEventDisableTiming) != cudaSuccess) k->ev[dev] = nullptr;
    return k->ev[dev];
}

}  // namespace gsi
