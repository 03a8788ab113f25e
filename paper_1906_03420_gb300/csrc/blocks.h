// Device memory: stream-ordered allocations, and the arena blocks of queries
// and batches that are kept for the next call.  Host code only.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace gsi {

// The library's own stream on a device (null: none).
cudaStream_t library_stream(int dev);
// Total memory of a device (looked up once per device).
uint64_t device_total_mem(int dev);

// cudaMallocAsync; where that fails, the blocks kept by the device's cache are
// given back first.
cudaError_t device_alloc(void **p, size_t bytes, cudaStream_t st);
template <typename T>
cudaError_t device_alloc(T **p, size_t bytes, cudaStream_t st) { return device_alloc(reinterpret_cast<void **>(p), bytes, st); }

// Blocks of the arenas of queries and batches, gigabytes each, kept for the
// next call.  The stream-ordered pool serves them well as long as no smaller
// request is cut out of a free one; then the next query waits milliseconds for
// new memory (four queries with rows took 14 to 25 ms instead of 2).
//
// Any thread and stream may take a block that another gave back: `idle` says
// that the stream had completed, otherwise an event orders the two.  A block
// whose event has not come yet is only taken on the stream that it was given
// back on, or from the library's own stream, where nothing waits for a caller's
// work: a request never waits for what another caller has put on a stream since,
// as one of the pool does not.
//
// A call takes the smallest kept block that holds what it asks for and is at
// most half as large again, an idle one first: calls whose budgets differ a
// little share blocks, and none ties up twice what it asked for.  A request that
// finds none gives back to the pool one that is a little too small, as the new
// block will serve in its place, and those that KEPT_TURNS requests have passed
// over: there they can be cut for other sizes.  At most KEPT_MOST blocks and a
// quarter of the device's memory are kept, none under BLOCK_MIN, and none at all
// without a graph on the device.
constexpr uint64_t BLOCK_MIN = 64ull << 20;
constexpr int KEPT_MOST = 64;
constexpr uint64_t KEPT_TURNS = 256;
struct Block {
    void *p = nullptr;
    uint64_t bytes = 0;              // of the whole block, which may be larger than asked for
};
cudaError_t block_get(int dev, uint64_t bytes, cudaStream_t st, Block *b);
void block_put(int dev, Block b, cudaStream_t st, bool idle);
// Gives every kept block back to the pool, behind its last use (wait: returns
// when they have arrived); their bytes.
uint64_t block_trim(int dev, bool wait);
// A graph was made on the device (+1) or destroyed (-1, with the device idle).
void block_users(int dev, int change);

// The blocks of one attempt on a stream, given back when it ends.  A block that
// another thread gave back may still be in use by the work that `st` was made
// to wait for, so the set counts as in use from its first get(); it goes back
// as idle only if a wait for the stream has succeeded since and nothing was
// enqueued after it.
class BlockSet {
public:
    BlockSet(int dev, cudaStream_t st) : dev_(dev), st_(st) {}
    BlockSet(const BlockSet &) = delete;
    BlockSet &operator=(const BlockSet &) = delete;
    ~BlockSet();
    cudaError_t get(uint64_t bytes, Block *b);
    void enqueued() { busy_ = true; }
    // The outcome of a wait for the stream.
    bool waited(cudaError_t e) {
        if (e == cudaSuccess) busy_ = false;
        return e == cudaSuccess;
    }
    bool busy() const { return busy_; }
    // Leaves the block at p to the caller, who gives it back by block_put.
    void take(const void *p);

private:
    static constexpr int MOST = 4;
    int dev_, n_ = 0;
    cudaStream_t st_;
    bool busy_ = false;
    Block held_[MOST];
};

}  // namespace gsi
