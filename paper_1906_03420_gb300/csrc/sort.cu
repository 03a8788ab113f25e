// LSD radix sort of 64-bit keys, used by the graph build: the vertices by
// label, the vertex pairs (duplicate check) and the directed edge entries by
// (vertex, edge label, neighbour).
//
// Each pass: per-tile digit histograms, one device scan of the bin-major
// histogram, then a stable scatter.  Inside a tile each warp owns a contiguous
// run of keys and walks it 32 keys at a time; lanes with equal digits find one
// another in a mask per digit, so ranks follow input order and every pass is
// stable.
//
// A pass reads the keys twice and writes them once, so the passes are few
// (digits of up to 9 bits, no wider than the fewest passes need) and the scatter
// first orders its tile in shared memory, from where each digit's keys leave as
// one run (16 of the 8,192 on average at 512 bins).  The scatter is bound by the
// instructions of its ranking (195 for 32 keys, half of the issue slots, with
// DRAM at 1.6 TB/s, when lanes were matched by ballots).  32M keys take 190-240
// us, and 78 for the histogram, for 9 bits; with __match_any_sync 190-330; with
// 10-bit digits 350; written straight from registers 265-450 for 8 bits.
#include "internal.h"
#include "scan.cuh"

namespace gsi {
namespace {

constexpr int RS_NT = 512;
constexpr int RS_WARPS = RS_NT / 32;
constexpr int RS_VT = 16;
constexpr int RS_TILE = RS_NT * RS_VT;
constexpr int RS_WARP_KEYS = 32 * RS_VT;
constexpr int RS_MAX_BITS = 9;
constexpr int RS_BINS_PER_THREAD = (1 << RS_MAX_BITS) / RS_NT;

__global__ void __launch_bounds__(RS_NT) k_rs_hist(const uint64_t *__restrict__ keys, int64_t n, int shift, int nbins,
                                                   uint32_t *__restrict__ hist, int64_t nblocks) {
    __shared__ uint32_t h[1 << RS_MAX_BITS];
    for (int b = threadIdx.x; b < nbins; b += RS_NT) h[b] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    const uint32_t dmask = (uint32_t)nbins - 1u;
#pragma unroll 8
    for (int j = 0; j < RS_VT; ++j) {
        int64_t i = base + j * RS_NT + threadIdx.x;
        if (i < n) atomicAdd(&h[(uint32_t)(keys[i] >> shift) & dmask], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < nbins; b += RS_NT) hist[(int64_t)b * nblocks + blockIdx.x] = h[b];
}

// Dynamic shared memory: the tile in digit order, then each warp's digit
// counts (at most RS_WARP_KEYS, 16 bits).
constexpr size_t rs_smem(int nbins) { return (size_t)RS_TILE * 8 + (size_t)RS_WARPS * nbins * 2; }

__global__ void __launch_bounds__(RS_NT, 2) k_rs_scatter(const uint64_t *__restrict__ in, uint64_t *__restrict__ out,
                                                         int64_t n, int shift, int nbins,
                                                         const uint32_t *__restrict__ offs, int64_t nblocks) {
    extern __shared__ __align__(16) unsigned char rs_sm[];
    uint64_t *stage = reinterpret_cast<uint64_t *>(rs_sm);
    uint16_t *wcnt = reinterpret_cast<uint16_t *>(stage + RS_TILE);        // [RS_WARPS][nbins]
    __shared__ uint32_t start[1 << RS_MAX_BITS];                           // a digit's first place in the tile
    __shared__ uint32_t delta[1 << RS_MAX_BITS];                           // its place in out less that one (mod 2^32)
    __shared__ uint32_t wt[RS_WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t dmask = (uint32_t)nbins - 1u;
    // each warp's lanes by digit, in the tile's place until that is filled
    static_assert(RS_TILE * 8 >= RS_WARPS * (1 << RS_MAX_BITS) * 4, "the lane masks fit the tile");
    uint32_t *peer = reinterpret_cast<uint32_t *>(stage) + warp * nbins;
    uint16_t *wc = wcnt + warp * nbins;
    for (int i = lane; i < nbins; i += 32) peer[i] = 0;
    for (int i = lane; i < nbins / 2; i += 32) reinterpret_cast<uint32_t *>(wc)[i] = 0;

    const int64_t tbase = (int64_t)blockIdx.x * RS_TILE;
    const uint32_t cnt = n - tbase < RS_TILE ? (uint32_t)(n - tbase) : (uint32_t)RS_TILE;
    const uint32_t first = (uint32_t)(warp * RS_WARP_KEYS + lane);
    in += tbase;
    uint64_t key[RS_VT];
    uint32_t pos[RS_VT / 2];                                               // two to a word: all are below RS_WARP_KEYS
    const unsigned lt = lanemask_lt(), me = 1u << lane;
#pragma unroll
    for (int r = 0; r < RS_VT; ++r) key[r] = first + r * 32 < cnt ? in[first + r * 32] : 0ull;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RS_VT; ++r) {
        const bool valid = first + r * 32 < cnt;
        const uint32_t dig = (uint32_t)(key[r] >> shift) & dmask;
        if (valid) atomicOr(&peer[dig], me);
        __syncwarp();
        const uint32_t peers = peer[dig], before = wc[dig];
        const uint32_t rank = __popc(peers & lt);
        __syncwarp();
        if (valid && rank == 0) {
            peer[dig] = 0;
            wc[dig] = (uint16_t)(before + __popc(peers));
        }
        __syncwarp();
        if (r & 1) pos[r / 2] |= (before + rank) << 16;
        else pos[r / 2] = before + rank;
    }
    __syncthreads();
    {   // per digit: exclusive scan over the warps, then over the digits
        uint32_t tot[RS_BINS_PER_THREAD], sum = 0;
#pragma unroll
        for (int q = 0; q < RS_BINS_PER_THREAD; ++q) {
            const int b = (int)threadIdx.x * RS_BINS_PER_THREAD + q;
            uint32_t run = 0;
            if (b < nbins) {
                uint32_t c[RS_WARPS];
#pragma unroll
                for (int w = 0; w < RS_WARPS; ++w) c[w] = wcnt[w * nbins + b];
#pragma unroll
                for (int w = 0; w < RS_WARPS; ++w) {
                    wcnt[w * nbins + b] = (uint16_t)run;
                    run += c[w];
                }
            }
            tot[q] = run;
            sum += run;
        }
        uint32_t all;
        uint32_t at = block_exclusive_scan<RS_NT, uint32_t>(sum, wt, &all);
#pragma unroll
        for (int q = 0; q < RS_BINS_PER_THREAD; ++q) {
            const int b = (int)threadIdx.x * RS_BINS_PER_THREAD + q;
            if (b < nbins) {
                start[b] = at;
                delta[b] = offs[(int64_t)b * nblocks + blockIdx.x] - at;
            }
            at += tot[q];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_VT; ++r)
        if (first + r * 32 < cnt) {
            const uint32_t dig = (uint32_t)(key[r] >> shift) & dmask;
            stage[start[dig] + wc[dig] + (r & 1 ? pos[r / 2] >> 16 : pos[r / 2] & 0xffffu)] = key[r];
        }
    __syncthreads();
#pragma unroll 4
    for (uint32_t j = threadIdx.x; j < cnt; j += RS_NT) {
        const uint64_t k = stage[j];
        out[(uint32_t)(delta[(uint32_t)(k >> shift) & dmask] + j)] = k;
    }
}

}  // namespace

gsi_status radix_sort_u64(uint64_t *keys, uint64_t *tmp, int64_t n, int lo, int hi, uint64_t **sorted, cudaStream_t st) {
    *sorted = keys;
    if (n <= 1 || hi <= lo) return GSI_OK;
    if (n >= (int64_t)1 << 32) {
        set_error("radix_sort_u64: more than 2^32 keys");
        return GSI_EINVAL;
    }
    const int passes = (hi - lo + RS_MAX_BITS - 1) / RS_MAX_BITS, width = (hi - lo + passes - 1) / passes;
    const int64_t nblocks = (n + RS_TILE - 1) / RS_TILE;
    const int64_t nh = ((int64_t)1 << width) * nblocks;
    GSI_CUDA_TRY(cudaFuncSetAttribute(k_rs_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)rs_smem(1 << RS_MAX_BITS)));
    uint32_t *hist = nullptr, *scr = nullptr;
    GSI_CUDA_TRY(device_alloc(&hist, sizeof(uint32_t) * (size_t)(nh + 1), st));
    if (device_alloc(&scr, sizeof(uint32_t) * (size_t)(scan_blocks(nh) + 1), st) != cudaSuccess) {
        cudaFreeAsync(hist, st);
        set_error("radix sort: no memory for the scan");
        return GSI_ENOMEM;
    }
    uint64_t *a = keys, *b = tmp;
    gsi_status rc = GSI_OK;
    for (int shift = lo; shift < hi && rc == GSI_OK; shift += width) {
        const int nbins = 1 << (hi - shift < width ? hi - shift : width);
        k_rs_hist<<<(unsigned)nblocks, RS_NT, 0, st>>>(a, n, shift, nbins, hist, nblocks);
        cudaError_t e = device_scan<uint32_t>(LoadProducer<uint32_t>{hist}, nbins * nblocks, StoreWriter<uint32_t>{hist},
                                              scr, st);
        if (e == cudaSuccess) {
            k_rs_scatter<<<(unsigned)nblocks, RS_NT, rs_smem(nbins), st>>>(a, b, n, shift, nbins, hist, nblocks);
            e = cudaGetLastError();
        }
        if (e != cudaSuccess) {
            set_error(std::string("radix sort: ") + cudaGetErrorString(e));
            rc = GSI_ECUDA;
        }
        uint64_t *s = a; a = b; b = s;
    }
    *sorted = a;
    cudaFreeAsync(hist, st);
    cudaFreeAsync(scr, st);
    return rc;
}

}  // namespace gsi
