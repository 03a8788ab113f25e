// The device's kept arena blocks (see blocks.h).
#include "blocks.h"

#include <mutex>
#include <vector>

namespace gsi {

namespace {
struct KeptBlock {
    void *p;
    uint64_t bytes;
    cudaEvent_t done;                // null: idle
};
struct BlockCache {
    std::mutex mu;
    std::vector<KeptBlock> kept;     // oldest first
    uint64_t bytes = 0;
    int users = 0;
};
BlockCache &block_cache(int dev) {   // never destroyed: results may outlive static objects
    static BlockCache *const c = new BlockCache[64];
    return c[dev];
}
// Gives the first `n` kept blocks back to the pool, behind their last use.
void block_release(BlockCache &c, size_t n, cudaStream_t st) {
    for (size_t i = 0; i < n; ++i) {
        KeptBlock &b = c.kept[i];
        if (b.done) {
            cudaStreamWaitEvent(st, b.done, 0);
            cudaEventDestroy(b.done);
        }
        cudaFreeAsync(b.p, st);
        c.bytes -= b.bytes;
    }
    c.kept.erase(c.kept.begin(), c.kept.begin() + (std::ptrdiff_t)n);
}
}  // namespace

cudaError_t device_alloc(void **p, size_t bytes, cudaStream_t st) {
    cudaError_t e = cudaMallocAsync(p, bytes, st);
    int dev = 0;
    if (e != cudaErrorMemoryAllocation || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return e;
    BlockCache &c = block_cache(dev);
    {
        std::lock_guard<std::mutex> lk(c.mu);
        if (c.kept.empty()) return e;
        block_release(c, c.kept.size(), st);
    }
    (void)cudaGetLastError();
    return cudaMallocAsync(p, bytes, st);
}

cudaError_t block_get(int dev, uint64_t bytes, cudaStream_t st, void **p) {
    if (bytes >= BLOCK_MIN && dev >= 0 && dev < 64) {
        BlockCache &c = block_cache(dev);
        std::lock_guard<std::mutex> lk(c.mu);
        for (size_t i = c.kept.size(); i-- > 0;) {
            const KeptBlock b = c.kept[i];
            if (b.bytes != bytes) continue;
            if (b.done) {
                const cudaError_t e = cudaStreamWaitEvent(st, b.done, 0);
                if (e != cudaSuccess) return e;
                cudaEventDestroy(b.done);
            }
            c.kept.erase(c.kept.begin() + (std::ptrdiff_t)i);
            c.bytes -= bytes;
            *p = b.p;
            return cudaSuccess;
        }
    }
    return device_alloc(p, bytes, st);
}

void block_put(int dev, void *p, uint64_t bytes, cudaStream_t st, bool idle) {
    if (bytes >= BLOCK_MIN && dev >= 0 && dev < 64) {
        const uint64_t most = device_total_mem(dev) / 4;
        BlockCache &c = block_cache(dev);
        std::lock_guard<std::mutex> lk(c.mu);
        if (c.users > 0 && bytes <= most) {
            cudaEvent_t done = nullptr;
            if (!idle && (cudaEventCreateWithFlags(&done, cudaEventDisableTiming) != cudaSuccess ||
                          cudaEventRecord(done, st) != cudaSuccess)) {
                (void)cudaGetLastError();
                if (done) cudaEventDestroy(done);
                done = nullptr;
                cudaDeviceSynchronize();              // the stream is gone: wait for what it had
            }
            c.kept.push_back({p, bytes, done});
            c.bytes += bytes;
            size_t n = 0;
            for (uint64_t left = c.bytes; left > most; ++n) left -= c.kept[n].bytes;
            if (n) block_release(c, n, st);
            return;
        }
    }
    cudaFreeAsync(p, st);
}

void block_users(int dev, int change) {
    if (dev < 0 || dev >= 64) return;
    BlockCache &c = block_cache(dev);
    std::lock_guard<std::mutex> lk(c.mu);
    c.users += change;
    if (c.users == 0) block_release(c, c.kept.size(), nullptr);
}

BlockSet::~BlockSet() {
    for (int i = 0; i < n_; ++i) block_put(dev_, held_[i].p, held_[i].bytes, st_, !busy_);
}

cudaError_t BlockSet::get(uint64_t bytes, void **p) {
    if (n_ == MOST) return cudaErrorInvalidValue;
    busy_ = true;
    const cudaError_t e = block_get(dev_, bytes, st_, p);
    if (e == cudaSuccess) held_[n_++] = {*p, bytes};
    return e;
}

void BlockSet::take(void *p) {
    for (int i = 0; i < n_; ++i)
        if (held_[i].p == p) {
            held_[i] = held_[--n_];
            return;
        }
}

}  // namespace gsi
