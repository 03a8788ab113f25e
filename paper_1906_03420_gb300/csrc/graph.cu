// Device graph build: label-partitioned CSR, label frequencies and the
// column-first signature table.
//
// Layout (Sec. IV, "basic representation" of the edge-label-partitioned
// graphs P(G,l)): every (vertex v, label l) pair owns one row-offset entry, so
// N(v,l) = ci[off[v*L+l] .. off[v*L+l+1]) is located with one 8-byte read.
// With the label counts of the target workloads (8-16 edge labels) this costs
// (L+1) * 4 bytes per vertex and replaces the paper's hashed PCSR groups,
// which exist to save that space when labels number in the tens of thousands.
// Each list N(v,l) is sorted by (label rank of the neighbour, neighbour id),
// with the label ranks kept in a parallel uint16 array cl: the neighbours of
// one vertex label form a contiguous, id-sorted sub-list, found by binary
// search on cl, and membership inside it is a binary search on ci.
//
// Signatures (Sec. III-A): N = 512 bits = 16 words per vertex, stored
// column-first (word w of vertex v at sig[w*n + v]) so a warp's 32 lanes read
// 32 consecutive words.  Word 0 is the vertex label itself (the K = 32 label
// bits).  Words 1..15 hold 240 two-bit groups: each (edge label, neighbour
// label) pair of v is hashed to a group whose state goes 00 -> 01 -> 11 as the
// first and second pair arrive.
#include <algorithm>
#include <climits>
#include <vector>

#include "internal.h"
#include "scan.cuh"

namespace gsi {
namespace {

constexpr int NT = 256;
constexpr int64_t COPY_APART = 1 << 20;               // below, an array arrives in 25 us

enum : unsigned { BAD_ID = 1u, SELF_LOOP = 2u, NEG_LABEL = 4u, DUP_PAIR = 8u };

__global__ void k_validate(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                           const int32_t *__restrict__ elab, int64_t m, int32_t n, unsigned *flags, int *maxlab) {
    unsigned f = 0;
    int ml = -1;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        int32_t a = src[e], b = dst[e], l = elab[e];
        if (a < 0 || a >= n || b < 0 || b >= n) f |= BAD_ID;
        if (a == b) f |= SELF_LOOP;
        if (l < 0) f |= NEG_LABEL;
        ml = max(ml, l);
    }
    f = __reduce_or_sync(FULL_MASK, f);
    ml = __reduce_max_sync(FULL_MASK, ml);
    if ((threadIdx.x & 31) == 0) {
        if (f) atomicOr(flags, f);
        atomicMax(maxlab, ml);
    }
}

__global__ void k_pair_keys(const int32_t *__restrict__ src, const int32_t *__restrict__ dst, int64_t m, int nb,
                            uint64_t *__restrict__ keys) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        uint64_t a = (uint32_t)src[e], b = (uint32_t)dst[e];
        keys[e] = a < b ? (a << nb) | b : (b << nb) | a;
    }
}

__global__ void k_adjacent_equal(const uint64_t *__restrict__ keys, int64_t n, unsigned *flags) {
    bool dup = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x + 1; i < n; i += (int64_t)gridDim.x * blockDim.x)
        dup |= keys[i] == keys[i - 1];
    if (__any_sync(FULL_MASK, dup) && (threadIdx.x & 31) == 0) atomicOr(flags, (unsigned)DUP_PAIR);
}

// Smallest and largest vertex label (range[0], range[1]: INT_MAX and INT_MIN before).
__global__ void k_label_range(const int32_t *__restrict__ vlab, int32_t n, int *range) {
    int lo = INT_MAX, hi = INT_MIN;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        lo = min(lo, vlab[v]);
        hi = max(hi, vlab[v]);
    }
    lo = __reduce_min_sync(FULL_MASK, lo);
    hi = __reduce_max_sync(FULL_MASK, hi);
    if ((threadIdx.x & 31) == 0) {
        atomicMin(range, lo);
        atomicMax(range + 1, hi);
    }
}

__global__ void k_vertex_keys(const int32_t *__restrict__ vlab, int32_t n, int32_t lo, int nb, uint64_t *__restrict__ keys) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        keys[v] = ((uint64_t)((uint32_t)vlab[v] - (uint32_t)lo) << nb) | (uint64_t)v;
}

// The vertices in the order of (label, id): at[i] holds the vertex of position
// i in its low half and its label rank in the high one (one gather for both),
// gpos is the position of each vertex, and label rank r begins at position
// start[r] and stands for label uniq[r].  One scan over the sorted
// keys: a position that differs from the one before it in its label starts a
// rank.  Ranks past MAX_LABELS are not written (the graph is refused).
constexpr int32_t MAX_LABELS = 65535;

struct LabelHead {
    const uint64_t *keys;
    int nb;
    __device__ uint32_t operator()(int64_t i) const { return i == 0 || (keys[i] >> nb) != (keys[i - 1] >> nb); }
};
struct LabelRanks {
    LabelHead head;
    int64_t n;
    int32_t lo;
    uint64_t *at;
    uint32_t *gpos;
    uint32_t *nlabels;
    int32_t *uniq, *start;
    __device__ void operator()(int64_t i, uint32_t before) const {
        if (i == n) {
            *nlabels = before;
            return;
        }
        const uint64_t k = head.keys[i];
        const uint32_t h = head(i), r = before + h - 1;
        const uint64_t v = k & ((1ull << head.nb) - 1);
        at[i] = (uint64_t)r << 32 | v;
        gpos[v] = (uint32_t)i;
        if (h && r < (uint32_t)MAX_LABELS) {
            uniq[r] = (int32_t)((uint32_t)(k >> head.nb) + (uint32_t)lo);
            start[r] = (int32_t)i;
        }
    }
};

// gperm: position i of the order above goes to its group's padded place.
__global__ void k_group_perm(const uint64_t *__restrict__ at, const int64_t *__restrict__ shift, int32_t n,
                             int32_t *__restrict__ gperm) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        gperm[i + shift[at[i] >> 32]] = (int32_t)at[i];
}

// Directed entry keys, two per edge: ((v << Lb | l) << nb) | gpos(neighbour).
// The neighbour stands as its position in the order of (label, id), which a
// list is sorted by: one field of nb bits instead of a label rank and an id.
__global__ void k_csr_keys(const int32_t *__restrict__ src, const int32_t *__restrict__ dst,
                           const int32_t *__restrict__ elab, const uint32_t *__restrict__ gpos, int64_t m, int Lb,
                           int nb, uint64_t *__restrict__ keys) {
    ulonglong2 *out = reinterpret_cast<ulonglong2 *>(keys);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = (uint32_t)src[e], b = (uint32_t)dst[e];
        const uint64_t l = (uint32_t)elab[e];
        out[e] = make_ulonglong2((((uint64_t)a << Lb | l) << nb) | gpos[b], (((uint64_t)b << Lb | l) << nb) | gpos[a]);
    }
}

// From sorted keys: ci[p] = neighbour, cl[p] = its label rank, off[s] = first
// position of segment s = v*L + l, and the group bits of the signatures
// (zeroed before).
//
// A pair's state needs its first two occurrences only, and equal pairs of a
// vertex stand together here: the first entry of a run counts one, the second
// sets both bits, the others do nothing.  A CTA takes FILL_TILE entries, which
// belong to few vertices: those between its first and its last one have all
// their entries here, so their words are put together in shared memory and
// written plainly; the two at the ends, and those past the FILL_V-th (in a
// sparse graph), set their bits by atomics.  The rank and the id of a neighbour
// come from one gather.  32M entries take 340 us (389 with an atomic for each
// pair and two gathers; 459 with the signatures made from the edge list).
constexpr int FILL_VT = 8;
constexpr int FILL_TILE = NT * FILL_VT;
constexpr int FILL_V = 256;

__global__ void __launch_bounds__(NT) k_csr_fill(const uint64_t *__restrict__ keys, int64_t n2, int Lb, int nb, int32_t L,
                                                 uint64_t nseg, const uint64_t *__restrict__ at,
                                                 const int32_t *__restrict__ uniq, int32_t n, uint32_t *__restrict__ off, int32_t *__restrict__ ci,
                                                 uint16_t *__restrict__ cl, uint32_t *__restrict__ sig) {
    __shared__ uint32_t words[(GSI_SIG_WORDS - 1) * FILL_V];
    const uint64_t mask = (1ull << nb) - 1, lmask = (1ull << Lb) - 1;
    const int lane = threadIdx.x & 31, vsh = Lb + nb;
    const int64_t t0 = (int64_t)blockIdx.x * FILL_TILE, t1 = min(n2, t0 + FILL_TILE);
    const uint64_t vfirst = keys[t0] >> vsh, vlast = keys[t1 - 1] >> vsh;
    const uint32_t inner = vlast - vfirst > 1 ? (uint32_t)min(vlast - vfirst - 1, (uint64_t)FILL_V) : 0u;   // vertices in `words`
    for (uint32_t i = threadIdx.x; i < (GSI_SIG_WORDS - 1) * FILL_V; i += NT) words[i] = 0;
    __syncthreads();
#pragma unroll 2
    for (int64_t p0 = t0 + (threadIdx.x & ~31u); p0 < t1; p0 += NT) {
        const int64_t p = p0 + lane;
        const bool valid = p < t1;
        const uint64_t k = valid ? keys[p] : 0ull;
        const uint64_t here = at[k & mask];
        const uint32_t r = (uint32_t)(here >> 32);
        // the two entries before the warp's, in lanes 0 and 1
        const bool xv = lane < 2 && p >= 2;
        const uint64_t x = xv ? keys[p - 2] : 0ull;
        const uint32_t xr = xv ? (uint32_t)(at[x & mask] >> 32) : 0u;
        const uint64_t seg = k >> nb, xseg = x >> nb;
        uint64_t s1 = __shfl_up_sync(FULL_MASK, seg, 1), s2 = __shfl_up_sync(FULL_MASK, seg, 2);
        uint32_t r1 = __shfl_up_sync(FULL_MASK, r, 1), r2 = __shfl_up_sync(FULL_MASK, r, 2);
        const uint64_t y = __shfl_sync(FULL_MASK, xseg, 1);
        const uint32_t yr = __shfl_sync(FULL_MASK, xr, 1);
        if (lane < 2) {
            s2 = xseg;
            r2 = xr;
        }
        if (lane == 0) {
            s1 = y;
            r1 = yr;
        }
        const bool same1 = p >= 1 && s1 == seg && r1 == r, same2 = p >= 2 && s2 == seg && r2 == r;
        if (!valid) continue;
        ci[p] = (int32_t)here;
        cl[p] = (uint16_t)r;
        const uint64_t v = seg >> Lb, l = seg & lmask, s = v * (uint64_t)L + l;
        uint64_t prev = 0;
        if (p > 0) prev = (s1 >> Lb) * (uint64_t)L + (s1 & lmask) + 1;
        for (uint64_t q = prev; q <= s; ++q) off[q] = (uint32_t)p;
        if (p == n2 - 1)
            for (uint64_t q = s + 1; q <= nseg; ++q) off[q] = (uint32_t)n2;
        if (!(same1 && same2)) {
            const uint32_t g = sig_group((int32_t)l, uniq[r]), bit = 1u << sig_bit(g);
            const uint64_t j = v - vfirst - 1;                // vfirst itself: past every bound
            uint32_t *word = j < inner && v < vlast ? words + (sig_word(g) - 1) * FILL_V + j
                                                    : sig + (int64_t)sig_word(g) * n + (int64_t)v;
            if (same1) atomicOr(word, 3u * bit);
            else if (atomicOr(word, bit) & bit) atomicOr(word, 2u * bit);
        }
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < (GSI_SIG_WORDS - 1) * inner; i += NT) {
        const uint32_t w = i / inner, j = i - w * inner;
        sig[(int64_t)(w + 1) * n + (int64_t)(vfirst + 1 + j)] = words[w * FILL_V + j];
    }
}

// Label directories of the lists of at least dir_min entries (gsi_graph::dir):
// each lane looks at one segment, and the warp fills the directories of the
// long ones together, one binary search of cl per label rank.  Most segments
// are short, so this is one read of off plus the few directories.
__global__ void k_label_dir(const uint32_t *__restrict__ off, const uint16_t *__restrict__ cl, uint64_t nseg, int32_t LV,
                            uint32_t dir_min, uint32_t *__restrict__ dir) {
    const int lane = threadIdx.x & 31;
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t s0 = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); s0 < nseg; s0 += step) {
        const uint64_t s = s0 + (uint64_t)lane;
        const uint32_t a = s < nseg ? off[s] : 0u, b = s < nseg ? off[s + 1] : 0u;
        for (unsigned m = __ballot_sync(FULL_MASK, b - a >= dir_min); m; m &= m - 1) {
            const int j = __ffs(m) - 1;
            const uint32_t x = __shfl_sync(FULL_MASK, a, j), y = __shfl_sync(FULL_MASK, b, j);
            for (int32_t r = lane; r <= LV; r += 32) {
                uint32_t lo = x, hi = y;
                while (lo < hi) {
                    const uint32_t mid = lo + ((hi - lo) >> 1);
                    if ((int32_t)cl[mid] < r) lo = mid + 1;
                    else hi = mid;
                }
                dir[((x + 1) >> 1) + (uint32_t)r] = lo;
            }
        }
    }
}

__global__ void k_fill_u32(uint32_t *a, uint64_t n, uint32_t v) {
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
        a[i] = v;
}

// Words 1..15 of every grouped position's vertex (zero for padding).
__global__ void k_group_sig(const uint32_t *__restrict__ sig, int32_t n, const int32_t *__restrict__ gperm,
                            int64_t np, uint32_t *__restrict__ gsig) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np; p += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = gperm[p];
#pragma unroll
        for (int w = 1; w < GSI_SIG_WORDS; ++w) gsig[(int64_t)(w - 1) * np + p] = v >= 0 ? sig[(int64_t)w * n + v] : 0u;
    }
}

// Directed entries per edge label, from the lists' lengths: a thread's
// segments all have one label (the grid's threads are a multiple of L), so it
// adds up in a register (one shared-memory atomic per edge, on 8 addresses,
// took 198 us of 16M edges; this takes 33).
__global__ void __launch_bounds__(NT) k_label_count(const uint32_t *__restrict__ off, uint64_t nseg, int32_t L,
                                                    uint64_t step, unsigned long long *freq) {
    constexpr int32_t LOCAL = 1024;
    __shared__ unsigned long long h[LOCAL];
    for (int32_t i = threadIdx.x; i < min(L, LOCAL); i += NT) h[i] = 0;
    __syncthreads();
    const uint64_t t = (uint64_t)blockIdx.x * NT + threadIdx.x;
    unsigned long long c = 0;
    if (t < step)
        for (uint64_t s = t; s < nseg; s += step) c += off[s + 1] - off[s];
    const uint64_t l = t % (uint64_t)L;
    if (c) atomicAdd(L <= LOCAL ? &h[l] : &freq[l], c);
    __syncthreads();
    if (L <= LOCAL)
        for (int32_t i = threadIdx.x; i < L; i += NT)
            if (h[i]) atomicAdd(&freq[i], h[i]);
}

// Device buffers of one build, released on its stream when it ends.
struct Temps {
    cudaStream_t st;
    std::vector<void *> all;
    explicit Temps(cudaStream_t s) : st(s) {}
    ~Temps() {
        if (other) {
            cudaStreamSynchronize(other);             // an error may leave copies behind
            cudaStreamDestroy(other);
        }
        if (ev) cudaEventDestroy(ev);
        for (void *p : all) cudaFreeAsync(p, st);
    }
    // A second stream, behind what this one has so far; join() orders the first
    // behind it.  It is the build's own: on a shared one, whatever else goes
    // there (results that are released) would wait for the caller's stream too.
    cudaStream_t other = nullptr;
    cudaEvent_t ev = nullptr;
    gsi_status beside() {
        GSI_CUDA_TRY(cudaStreamCreateWithFlags(&other, cudaStreamNonBlocking));
        GSI_CUDA_TRY(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        GSI_CUDA_TRY(cudaEventRecord(ev, st));
        GSI_CUDA_TRY(cudaStreamWaitEvent(other, ev, 0));
        return GSI_OK;
    }
    gsi_status join() {
        if (!other) return GSI_OK;
        GSI_CUDA_TRY(cudaEventRecord(ev, other));
        GSI_CUDA_TRY(cudaStreamWaitEvent(st, ev, 0));
        return GSI_OK;
    }
    template <typename T>
    gsi_status alloc(T **p, uint64_t count) {
        GSI_CUDA_TRY(device_alloc(p, sizeof(T) * (size_t)(count + 1), st));
        all.push_back(*p);
        return GSI_OK;
    }
};

// Reads device memory once the stream's work is done.  The wait comes first: a
// copy to pageable memory waits for it inside the driver, where other threads'
// calls that create or destroy an event then wait too.
gsi_status read_back(void *dst, const void *src, size_t bytes, cudaStream_t st) {
    GSI_CUDA_TRY(cudaStreamSynchronize(st));
    GSI_CUDA_TRY(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st));
    GSI_CUDA_TRY(cudaStreamSynchronize(st));
    return GSI_OK;
}

unsigned grid_for(int64_t n) {
    int64_t b = (n + NT - 1) / NT;
    if (b < 1) b = 1;
    if (b > 152 * 64) b = 152 * 64;
    return (unsigned)b;
}

// For kernels that end with an atomic per warp on one word: thousands of warps
// wait for it (51 us for 2^20 labels with one element per thread, 74 us for 16M
// edges), so fewer threads take more each.
unsigned few_blocks(int64_t n) { return std::min(grid_for(n), 152u * 6); }

}  // namespace

gsi_status build_graph(gsi_graph *g, const int32_t *vlab, int32_t n, const int32_t *src, const int32_t *dst,
                       const int32_t *elab, int64_t m, cudaStream_t st) {
    if (n < 1 || m < 0) {
        set_error("gsi_graph_create: need n >= 1 and m >= 0");
        return GSI_EINVAL;
    }
    if (2 * m >= ((int64_t)1 << 32)) {
        set_error("gsi_graph_create: 2m must be below 2^32");
        return GSI_EINVAL;
    }
    if (m > 0 && (!src || !dst || !elab)) {
        set_error("gsi_graph_create: null edge arrays");
        return GSI_EINVAL;
    }
    if (!vlab) {
        set_error("gsi_graph_create: null vertex labels");
        return GSI_EINVAL;
    }
    cudaEvent_t e0, e1;
    GSI_CUDA_TRY(cudaEventCreate(&e0));
    GSI_CUDA_TRY(cudaEventCreate(&e1));
    GSI_CUDA_TRY(cudaEventRecord(e0, st));

    Temps tmps(st);
    int32_t *d_vlab = nullptr, *d_src = nullptr, *d_dst = nullptr, *d_elab = nullptr;
    // error bits, largest edge label, vertex label range, distinct vertex labels
    struct Words {
        unsigned flags;
        int maxlab, lo, hi;
        uint32_t nlabels;
    } hw = {0u, -1, INT_MAX, INT_MIN, 0u};
    Words *d_w = nullptr;
    GSI_TRY(tmps.alloc(&d_vlab, (uint64_t)n));
    GSI_TRY(tmps.alloc(&d_src, (uint64_t)m));
    GSI_TRY(tmps.alloc(&d_dst, (uint64_t)m));
    GSI_TRY(tmps.alloc(&d_elab, (uint64_t)m));
    GSI_TRY(tmps.alloc(&d_w, 1));
    GSI_CUDA_TRY(cudaMemcpyAsync(d_w, &hw, sizeof hw, cudaMemcpyHostToDevice, st));
    GSI_CUDA_TRY(cudaMemcpyAsync(d_vlab, vlab, sizeof(int32_t) * (size_t)n, cudaMemcpyDefault, st));
    k_label_range<<<few_blocks(n), NT, 0, st>>>(d_vlab, n, &d_w->lo);
    // a large edge list is copied on a stream of its own: the vertices are
    // sorted meanwhile, and the pairs while the edge labels arrive (16M edges:
    // 365 us an array; 4.58 -> 4.26 ms)
    if (m >= COPY_APART) GSI_TRY(tmps.beside());
    const cudaStream_t cs = tmps.other ? tmps.other : st;
    GSI_TRY(read_back(&hw, d_w, sizeof hw, st));
    const int nb = ceil_log2_bits((uint64_t)(n > 1 ? n - 1 : 1));

    // the vertices in the order of (label, id), the checks of the edges behind
    // them on the stream, one readback for all
    const uint64_t nkeys = std::max((uint64_t)(2 * m), (uint64_t)n);
    uint64_t *keys = nullptr, *tmp = nullptr, *sorted = nullptr;
    GSI_TRY(tmps.alloc(&keys, nkeys));
    GSI_TRY(tmps.alloc(&tmp, nkeys));
    int32_t *d_labels = nullptr;
    uint64_t *at = nullptr;
    uint32_t *gpos = nullptr, *scr = nullptr;
    const int32_t most = (int32_t)std::min<int64_t>(n, MAX_LABELS);
    GSI_TRY(tmps.alloc(&at, (uint64_t)n));
    GSI_TRY(tmps.alloc(&gpos, (uint64_t)n));
    GSI_TRY(tmps.alloc(&d_labels, 2 * (uint64_t)most));
    GSI_TRY(tmps.alloc(&scr, (uint64_t)scan_blocks(n) + 1));
    const uint32_t range = (uint32_t)hw.hi - (uint32_t)hw.lo;
    k_vertex_keys<<<grid_for(n), NT, 0, st>>>(d_vlab, n, hw.lo, nb, keys);
    GSI_TRY(radix_sort_u64(keys, tmp, n, nb, range ? nb + ceil_log2_bits(range) : nb, &sorted, st));
    const LabelHead head{sorted, nb};
    GSI_CUDA_TRY(device_scan<uint32_t>(
        head, n, LabelRanks{head, n, hw.lo, at, gpos, &d_w->nlabels, d_labels, d_labels + most}, scr, st));
    if (m > 0) {
        GSI_CUDA_TRY(cudaMemcpyAsync(d_src, src, sizeof(int32_t) * (size_t)m, cudaMemcpyDefault, cs));
        GSI_CUDA_TRY(cudaMemcpyAsync(d_dst, dst, sizeof(int32_t) * (size_t)m, cudaMemcpyDefault, cs));
        GSI_TRY(tmps.join());
    }
    if (m > 1) {                                      // of ids that may yet turn out to be bad
        k_pair_keys<<<grid_for(m), NT, 0, st>>>(d_src, d_dst, m, nb, keys);
        GSI_TRY(radix_sort_u64(keys, tmp, m, 0, 2 * nb, &sorted, st));
        k_adjacent_equal<<<grid_for(m), NT, 0, st>>>(sorted, m, &d_w->flags);
    }
    if (m > 0) {
        GSI_CUDA_TRY(cudaMemcpyAsync(d_elab, elab, sizeof(int32_t) * (size_t)m, cudaMemcpyDefault, cs));
        GSI_TRY(tmps.join());
        k_validate<<<few_blocks(m), NT, 0, st>>>(d_src, d_dst, d_elab, m, n, &d_w->flags, &d_w->maxlab);
    }
    std::vector<int32_t> labels(2 * (size_t)most);     // the distinct labels, then where each begins
    GSI_TRY(read_back(&hw, d_w, sizeof hw, st));
    GSI_TRY(read_back(labels.data(), d_labels, sizeof(int32_t) * labels.size(), st));
    if (hw.flags & ~(unsigned)DUP_PAIR) {
        set_error(std::string("gsi_graph_create: ") + ((hw.flags & BAD_ID) ? "vertex id out of range " : "") +
                  ((hw.flags & SELF_LOOP) ? "self-loop " : "") + ((hw.flags & NEG_LABEL) ? "negative edge label" : ""));
        return GSI_EINVAL;
    }
    const int32_t L = hw.maxlab < 0 ? 1 : hw.maxlab + 1;
    if (hw.nlabels > (uint32_t)MAX_LABELS) {
        set_error("gsi_graph_create: more than 65535 distinct vertex labels");
        return GSI_EINVAL;
    }
    const int32_t LV = (int32_t)hw.nlabels;
    const int lb = ceil_log2_bits((uint64_t)(LV > 1 ? LV - 1 : 1));
    const uint64_t nseg = (uint64_t)n * (uint64_t)L;
    const int sb = ceil_log2_bits(nseg - 1);
    if (sb + lb + nb > 64 || nseg + 1 >= ((uint64_t)1 << 34)) {
        set_error("gsi_graph_create: n * L * labels too large for the label-partitioned layout");
        return GSI_EINVAL;
    }
    if (hw.flags & DUP_PAIR) {
        set_error("gsi_graph_create: a vertex pair appears more than once");
        return GSI_EINVAL;
    }

    // label groups, each padded to whole warps
    std::vector<int64_t> goff((size_t)LV + 1, 0), shift((size_t)LV, 0);
    for (int32_t r = 0; r < LV; ++r) {
        const int64_t begin = labels[(size_t)(most + r)], end = r + 1 < LV ? labels[(size_t)(most + r + 1)] : n;
        goff[r + 1] = goff[r] + (end - begin + 31) / 32 * 32;
        shift[r] = goff[r] - begin;
    }

    // CSR and signatures
    g->n = n; g->m = m; g->L = L; g->LV = LV; g->nwords = (n + 31) / 32;
    g->vlabels.assign(labels.begin(), labels.begin() + LV);
    GSI_CUDA_TRY(device_alloc(&g->off, sizeof(uint32_t) * (size_t)(nseg + 1), st));
    GSI_CUDA_TRY(device_alloc(&g->ci, sizeof(int32_t) * (size_t)(2 * m + 1), st));
    GSI_CUDA_TRY(device_alloc(&g->cl, sizeof(uint16_t) * (size_t)(2 * m + 1), st));
    GSI_CUDA_TRY(device_alloc(&g->dir, sizeof(uint32_t) * (size_t)(m + 1), st));
    g->dir_min = 2u * ((uint32_t)LV + 1u);
    GSI_CUDA_TRY(device_alloc(&g->sig, sizeof(uint32_t) * (size_t)GSI_SIG_WORDS * (size_t)n, st));
    GSI_CUDA_TRY(cudaMemsetAsync(g->sig, 0, sizeof(uint32_t) * (size_t)GSI_SIG_WORDS * (size_t)n, st));
    GSI_CUDA_TRY(cudaMemcpyAsync(g->sig, d_vlab, sizeof(uint32_t) * (size_t)n, cudaMemcpyDeviceToDevice, st));
    if (m > 0) {
        // nb + Lb + nb is at most sb + 1 + nb, and lb at least 1: it fits 64 bits
        const int Lb = L > 1 ? ceil_log2_bits((uint64_t)L - 1) : 0;
        k_csr_keys<<<grid_for(m), NT, 0, st>>>(d_src, d_dst, d_elab, gpos, m, Lb, nb, keys);
        GSI_TRY(radix_sort_u64(keys, tmp, 2 * m, 0, nb + Lb + nb, &sorted, st));
        k_csr_fill<<<(unsigned)((2 * m + FILL_TILE - 1) / FILL_TILE), NT, 0, st>>>(sorted, 2 * m, Lb, nb, L, nseg, at,
                                                                                   d_labels, n, g->off, g->ci, g->cl, g->sig);
        k_label_dir<<<grid_for((int64_t)nseg), NT, 0, st>>>(g->off, g->cl, nseg, LV, g->dir_min, g->dir);
    } else {
        k_fill_u32<<<grid_for((int64_t)nseg + 1), NT, 0, st>>>(g->off, nseg + 1, 0u);
    }

    // signatures grouped by label
    g->np = goff[LV];
    g->goff = goff;
    GSI_CUDA_TRY(device_alloc(&g->gperm, sizeof(int32_t) * (size_t)g->np, st));
    GSI_CUDA_TRY(device_alloc(&g->gsig, sizeof(uint32_t) * (size_t)(GSI_SIG_WORDS - 1) * (size_t)g->np, st));
    int64_t *d_shift = nullptr;
    GSI_TRY(tmps.alloc(&d_shift, (uint64_t)LV));
    GSI_CUDA_TRY(cudaMemcpyAsync(d_shift, shift.data(), sizeof(int64_t) * (size_t)LV, cudaMemcpyHostToDevice, st));
    GSI_CUDA_TRY(cudaMemsetAsync(g->gperm, 0xff, sizeof(int32_t) * (size_t)g->np, st));     // -1: padding
    k_group_perm<<<grid_for(n), NT, 0, st>>>(at, d_shift, n, g->gperm);
    k_group_sig<<<grid_for(g->np), NT, 0, st>>>(g->sig, n, g->gperm, g->np, g->gsig);

    // freq(l): each edge has two entries
    unsigned long long *d_freq = nullptr;
    GSI_TRY(tmps.alloc(&d_freq, (uint64_t)L));
    GSI_CUDA_TRY(cudaMemsetAsync(d_freq, 0, sizeof(unsigned long long) * (size_t)L, st));
    {
        const uint64_t threads = std::max<uint64_t>((uint64_t)L, 152 * 1024);
        const uint64_t step = threads / (uint64_t)L * (uint64_t)L;
        k_label_count<<<(unsigned)((step + NT - 1) / NT), NT, 0, st>>>(g->off, nseg, L, step, d_freq);
    }
    g->freq.assign((size_t)L, 0);
    GSI_CUDA_TRY(cudaGetLastError());
    GSI_CUDA_TRY(cudaEventRecord(e1, st));
    GSI_TRY(read_back(g->freq.data(), d_freq, sizeof(uint64_t) * (size_t)L, st));
    for (uint64_t &f : g->freq) f /= 2;
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    g->build_ms = ms;
    g->device_bytes = sizeof(uint32_t) * (nseg + 1) + sizeof(int32_t) * (uint64_t)(2 * m + 1) +
                      sizeof(uint16_t) * (uint64_t)(2 * m + 1) + sizeof(uint32_t) * (uint64_t)(m + 1) +
                      sizeof(uint32_t) * GSI_SIG_WORDS * (uint64_t)n +
                      sizeof(uint32_t) * GSI_SIG_WORDS * (uint64_t)g->np;
    return GSI_OK;
}

}  // namespace gsi
