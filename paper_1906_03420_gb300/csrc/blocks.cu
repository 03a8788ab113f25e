// The device's kept arena blocks (see blocks.h).
#include "blocks.h"

#include <mutex>

namespace gsi {
namespace {

struct KeptBlock {
    void *p;
    uint64_t bytes;
    cudaEvent_t done;                // null: idle
    cudaStream_t st;                 // where it was recorded
    uint64_t turn;                   // requests before it was given back
};
struct BlockCache {
    std::mutex mu;
    KeptBlock kept[KEPT_MOST];       // oldest first; no allocation, as results are destroyed without exceptions
    int n = 0, users = 0;
    uint64_t bytes = 0, turn = 0;
    // events that no block has: creating or destroying one waits for any thread
    // that is in a copy to pageable memory, until that copy's stream gets there
    cudaEvent_t spare[KEPT_MOST];
    int nspare = 0;
    cudaStream_t out = nullptr;      // blocks go back to the pool here, behind their last use and nothing else
};

BlockCache &block_cache(int dev) {   // never destroyed: results may outlive static objects
    static BlockCache *const c = new BlockCache[64];
    return c[dev];
}

// An event recorded on st; null, with the device waited for, if there is none.
cudaEvent_t take_event(BlockCache &c, cudaStream_t st) {
    cudaEvent_t e = nullptr;
    if (c.nspare) e = c.spare[--c.nspare];
    else if (cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) e = nullptr;
    if (e && cudaEventRecord(e, st) == cudaSuccess) return e;
    (void)cudaGetLastError();
    if (e) c.spare[c.nspare++] = e;
    cudaDeviceSynchronize();                          // the stream is gone: wait for what it had
    return nullptr;
}

void block_remove(BlockCache &c, int i) {
    c.bytes -= c.kept[i].bytes;
    for (--c.n; i < c.n; ++i) c.kept[i] = c.kept[i + 1];
}

// Gives kept block i back to the pool, behind its last use.
void block_release(BlockCache &c, int i) {
    const KeptBlock b = c.kept[i];
    if (!c.out && cudaStreamCreateWithFlags(&c.out, cudaStreamNonBlocking) != cudaSuccess) c.out = nullptr;
    if (b.done) {
        cudaStreamWaitEvent(c.out, b.done, 0);
        c.spare[c.nspare++] = b.done;
    }
    cudaFreeAsync(b.p, c.out);
    block_remove(c, i);
}

// Whether the work on a kept block has ended.
bool block_idle(BlockCache &c, KeptBlock &k) {
    if (!k.done) return true;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;    // a query is no part of anyone's capture
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaEventQuery(k.done);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    c.spare[c.nspare++] = k.done;
    k.done = nullptr;
    return true;
}

}  // namespace

cudaError_t device_alloc(void **p, size_t bytes, cudaStream_t st) {
    cudaError_t e = cudaMallocAsync(p, bytes, st);
    int dev = 0;
    if (e != cudaErrorMemoryAllocation || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return e;
    if (!block_trim(dev, false)) return e;
    (void)cudaGetLastError();
    e = cudaMallocAsync(p, bytes, st);
    if (e != cudaErrorMemoryAllocation) return e;
    block_trim(dev, true);                            // not all of it had arrived
    (void)cudaGetLastError();
    return cudaMallocAsync(p, bytes, st);
}

cudaError_t block_get(int dev, uint64_t bytes, cudaStream_t st, Block *b) {
    if (bytes >= BLOCK_MIN && dev >= 0 && dev < 64) {
        BlockCache &c = block_cache(dev);
        std::lock_guard<std::mutex> lk(c.mu);
        ++c.turn;
        const cudaStream_t own = library_stream(dev);
        int at = -1;
        for (int i = 0; i < c.n; ++i) {
            KeptBlock &k = c.kept[i];
            if (k.bytes < bytes || k.bytes - bytes > bytes / 2) continue;
            if (!block_idle(c, k) && k.st != st && k.st != own) continue;
            const KeptBlock *best = at < 0 ? nullptr : &c.kept[at];
            if (!best || (best->done && !k.done) || (!best->done == !k.done && k.bytes < best->bytes)) at = i;
        }
        if (at >= 0) {
            const KeptBlock k = c.kept[at];
            if (k.done) {
                const cudaError_t e = cudaStreamWaitEvent(st, k.done, 0);
                if (e != cudaSuccess) return e;
                c.spare[c.nspare++] = k.done;
            }
            block_remove(c, at);
            *b = {k.p, k.bytes};
            return cudaSuccess;
        }
        // a new block: one a little too small, which it will serve in place of,
        // goes back to the pool, and so do those passed over for long
        int less = -1, old = 0;
        for (int i = 0; i < c.n; ++i)
            if (c.kept[i].bytes < bytes && bytes - c.kept[i].bytes <= c.kept[i].bytes / 2 &&
                (less < 0 || c.kept[i].bytes > c.kept[less].bytes))
                less = i;
        if (less >= 0) block_release(c, less);
        while (old < c.n && c.turn - c.kept[old].turn > KEPT_TURNS) ++old;
        while (old-- > 0) block_release(c, 0);
    }
    b->bytes = bytes;
    return device_alloc(&b->p, bytes, st);
}

void block_put(int dev, Block b, cudaStream_t st, bool idle) {
    if (b.bytes >= BLOCK_MIN && dev >= 0 && dev < 64) {
        const uint64_t most = device_total_mem(dev) / 4;
        BlockCache &c = block_cache(dev);
        std::lock_guard<std::mutex> lk(c.mu);
        if (c.users > 0 && b.bytes <= most) {
            while (c.n == KEPT_MOST || c.bytes + b.bytes > most) block_release(c, 0);
            const cudaEvent_t done = idle ? nullptr : take_event(c, st);
            c.kept[c.n++] = {b.p, b.bytes, done, st, c.turn};
            c.bytes += b.bytes;
            return;
        }
    }
    cudaFreeAsync(b.p, st);
}

uint64_t block_trim(int dev, bool wait) {
    if (dev < 0 || dev >= 64) return 0;
    BlockCache &c = block_cache(dev);
    uint64_t bytes = 0;
    cudaStream_t out = nullptr;
    {
        std::lock_guard<std::mutex> lk(c.mu);
        bytes = c.bytes;
        while (c.n) block_release(c, 0);
        out = c.out;
    }
    if (wait && out) cudaStreamSynchronize(out);
    return bytes;
}

void block_users(int dev, int change) {
    if (dev < 0 || dev >= 64) return;
    BlockCache &c = block_cache(dev);
    std::lock_guard<std::mutex> lk(c.mu);
    c.users += change;
    if (c.users) return;
    while (c.n) block_release(c, 0);
    while (c.nspare) cudaEventDestroy(c.spare[--c.nspare]);
}

BlockSet::~BlockSet() {
    for (int i = 0; i < n_; ++i) block_put(dev_, held_[i], st_, !busy_);
}

cudaError_t BlockSet::get(uint64_t bytes, Block *b) {
    if (n_ == MOST) return cudaErrorInvalidValue;
    busy_ = true;
    const cudaError_t e = block_get(dev_, bytes, st_, b);
    if (e == cudaSuccess) held_[n_++] = *b;
    return e;
}

void BlockSet::take(const void *p) {
    for (int i = 0; i < n_; ++i)
        if (held_[i].p == p) {
            held_[i] = held_[--n_];
            return;
        }
}

}  // namespace gsi
