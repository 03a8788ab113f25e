// Join iterations (Sec. V, Algs. 3-4), in two forms.
//
// Host-sized (the splitting path of the memory-bounded driver, the
// allocation-free join step, and gsi_join_step where its cooperative launch
// cannot take the step): one iteration as three launches,
//   1. scan   F[i] = sum_{r<i} (cap_r + W), where cap_r bounds row r's output
//             (Alg. 4's preallocation bound), plus W "row slots" per row that
//             pay for staging the row (load balancing, below);
//   2. part   for every tile of NV consecutive slots, its first row;
//   3. join   the fused kernel: one CTA per tile of NV slots.
//
// Device-driven (k_query): the seed and every iteration of one query in one
// cooperative launch, or one iteration over a caller's table (gsi_join_step):
// per step the row pass (join_rows.cuh), which joins short rows and sets long
// ones aside with their slot offsets, and the long rows' slot tiles, with a
// bounded grid barrier after each.
//
// Output bound.  Every neighbour list N(v,l) is stored sorted by (label rank
// of the neighbour, neighbour id), so the neighbours of v via l that carry
// the new query vertex's label form one contiguous, id-sorted sub-list.  Any
// survivor w of row i lies in that sub-list of every linking edge, so each
// row takes as its candidate list (and output bound, Alg. 4) the shortest of
// these sub-lists; Alg. 4's global choice of the least frequent edge label is
// the same bound taken once for all rows.
//
// Work decomposition.  Instead of the paper's warp-per-row with a 4-layer
// balance scheme and dynamically launched child kernels (Sec. VI-A), every
// candidate of every row is one slot of a flat index space whose row offsets
// are F, and each CTA takes a fixed NV slots.  A hub row with 10^5
// candidates is spread over many CTAs; rows with one candidate are packed
// NV/W to a CTA.  The W per-row slots bound the rows one CTA stages, so its
// shared memory holds every row it touches.
//
// Per CTA (Sec. V "GPU-friendly set operation"):
//   * the partial matches m_i of its rows are staged in shared memory with
//     the bounds of every label sub-list they need (small lists);
//   * a slot -> row map is built with one block-wide max-scan;
//   * slots read consecutive elements of the row's candidate sub-list
//     (coalesced medium list);
//   * C(u) is probed as a bitset, one 4-byte load per candidate (large list);
//   * set subtraction (w not in m_i) is checked against the staged row;
//   * the other linking edges test w in their sub-list by binary search (the
//     intersection), only for candidates that survived the cheaper checks;
//   * survivors are compacted with one block-wide prefix sum and one global
//     atomic per CTA, then written once as rows of M' (Prealloc-Combine: the
//     join runs once; the output buffer is sized by F's total).
#include <algorithm>
#include <cstddef>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "internal.h"
#include "join_rows.cuh"
#include "join_tile.cuh"
#include "scan.cuh"

namespace gsi {
namespace {

// Reduce pass: stores each row's bound for the down pass.
struct CapStoreProducer {
    const int32_t *M;
    const uint32_t *off;
    LabelIndex cl;
    uint32_t *caps;
    uint64_t W;
    StepDev s;
    __device__ uint64_t operator()(int64_t i) const {
        uint32_t c = row_bound(s, M + i * s.t, off, cl);
        caps[i] = c;
        return (uint64_t)c + W;
    }
};
struct CapLoadProducer {
    const uint32_t *caps;
    uint64_t W;
    __device__ uint64_t operator()(int64_t i) const { return (uint64_t)caps[i] + W; }
};


template <typename P1, typename P2, typename Wr>
cudaError_t two_producer_scan(P1 p1, P2 p2, int64_t n, Wr write, uint64_t *scratch, cudaStream_t st) {
    if (n <= 0) {
        k_scan_empty<uint64_t, Wr><<<1, 1, 0, st>>>(write);
        return cudaGetLastError();
    }
    int64_t nb = scan_blocks(n);
    k_scan_reduce<uint64_t, P1><<<(unsigned)nb, SCAN_NT, 0, st>>>(p1, n, scratch);
    k_scan_spine<uint64_t><<<1, 1024, 0, st>>>(scratch, nb);
    k_scan_down<uint64_t, P2, Wr><<<(unsigned)nb, SCAN_NT, 0, st>>>(p2, n, scratch, nb, write);
    return cudaGetLastError();
}

__global__ void k_partition(const uint64_t *__restrict__ F, int64_t R, uint64_t total, int64_t ntiles,
                            int64_t *__restrict__ part) {
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b > ntiles) return;
    uint64_t s = (uint64_t)b * JOIN_NV;
    if (s > total) s = total;
    int64_t lo = 0, hi = R;            // largest r in [0, R] with F[r] <= s
    while (lo < hi) {
        int64_t mid = (lo + hi + 1) >> 1;
        if (F[mid] <= s) lo = mid;
        else hi = mid - 1;
    }
    part[b] = lo;
}

template <int NT, int VT>
__global__ void __launch_bounds__(NT) k_join(const __grid_constant__ JoinArgs a) {
    join_tile<NT, VT>(a, a.M, a.R, a.F, a.total, a.part[blockIdx.x], a.part[blockIdx.x + 1], a.out, a.out_cap,
                      a.out_count, blockIdx.x);
}

// ------------------------------------------------- one launch per query
// The whole join of one query in a single cooperative launch: the seed, then
// for every step the row pass and, when it set rows aside, the long rows'
// tiles, with a grid barrier after each.  All CTAs are co-resident (cooperative
// launch), so the barrier is one counter of arrivals; every wait is bounded,
// and a CTA that gives up sets a bit in that word and returns, as does every
// CTA that later sees the bit, so the kernel always terminates.

constexpr unsigned long long BARRIER_SPIN_LIMIT = 1ull << 24;   // x a 64 ns sleep and a read of L2: a second at least
constexpr unsigned BAR_FAIL = 1u << 31;

// What a barrier hands to its CTA: the step's counters as of the barrier, read
// by the thread that waited.
struct BarrierView {
    unsigned long long count, nlong;
    unsigned fail;
    int ok;
};

// One word counts the arrivals of all barriers of the launch, so a CTA knows
// the number to wait for (epoch: barriers passed), the last one to arrive has
// nothing to reset or release, and a wait that gave up shows in the same word.
// A step of few rows costs little but its chain of L2 round trips (some 0.6 us
// each): a generation word, a fail word and counters that all 4,864 warps read
// for themselves took 2.3 us at least for a barrier and 2-3 us for the start of
// a step; now 1.6 and 0.3 us (a 4-vertex query on 1,000 vertices: 42 -> 33 us).
__device__ __forceinline__ bool grid_barrier(QueryCtl *ctl, unsigned nblocks, unsigned &epoch, const DStep *st,
                                             BarrierView *view) {
    __syncthreads();
    ++epoch;
    if (threadIdx.x == 0) {
        const unsigned long long limit = ctl->spin_limit ? ctl->spin_limit : BARRIER_SPIN_LIMIT;
        const unsigned target = epoch * nblocks;
        __threadfence();
        unsigned v = atomicAdd(&ctl->bar, 1u) + 1u;
        for (unsigned long long spins = 0; v < target;) {     // BAR_FAIL ends it too
            if (++spins > limit) {
                atomicOr(&ctl->fail, 4u);
                v = atomicOr(&ctl->bar, BAR_FAIL) | BAR_FAIL;
                break;
            }
            if (spins > 1) __nanosleep(64);
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->bar) : "memory");
        }
        __threadfence();
        view->ok = v < BAR_FAIL;
        if (st) {
            view->count = __ldcg(&st->count);
            view->nlong = __ldcg(&st->nlong);
            view->fail = __ldcg(&st->fail);
        }
    }
    __syncthreads();
    return view->ok != 0;
}

// Copies a struct of 8-byte words to shared memory with the whole CTA, behind
// what it does next: complete after copy_wait and a barrier.
template <int NT, typename T>
__device__ __forceinline__ void copy_words(T *dst, const T *src) {
    static_assert(sizeof(T) % 8 == 0 && alignof(T) >= 8, "whole words");
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    for (unsigned i = threadIdx.x; i < (unsigned)(sizeof(T) / 8); i += NT)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d + 8 * i),
                     "l"(reinterpret_cast<const unsigned char *>(src) + 8 * i)
                     : "memory");
}
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <int NT, bool LW>
__global__ void __launch_bounds__(NT, 4) k_query(const JoinArgs *__restrict__ cfgs, DStep *steps, int t0, int k,
                                              QueryCtl *ctl, const uint32_t *__restrict__ seed_bitmap, int64_t nwords) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long wt[NT / 32];
    __shared__ unsigned long long at_s;
    __shared__ __align__(16) JoinArgs args_s[2];      // this step's configuration and the next one's
    __shared__ __align__(16) DStepIn ins_s[2];
    __shared__ BarrierView view_s;
    const unsigned G = gridDim.x;
    unsigned epoch = 0;
    copy_words<NT>(&args_s[t0 & 1], cfgs + 1);
    copy_words<NT>(&ins_s[t0 & 1], &steps[1].in);

    // ---- seed: C(u_first) as the one-column table in the first region (Alg.
    // 2).  Each CTA lists the set bits of an equal share of the words, at a
    // place that one atomic reserves (the order of rows is free): one read of
    // the bitmap and one grid barrier.  Without a seed bitmap (step_coop) the
    // first step's table is there, and steps[0] has its row count.
    if (!seed_bitmap) {
        copy_wait();
        if (threadIdx.x == 0) view_s.count = steps[0].count;
        __syncthreads();
    } else {
        int32_t *seed_out = const_cast<int32_t *>(steps[1].in.M);
        const uint64_t chunk = (((uint64_t)nwords + G - 1) / G + 31) & ~31ull;
        const uint64_t lo = (uint64_t)blockIdx.x * chunk, hi = min((uint64_t)nwords, lo + chunk);
        for (uint64_t base = lo; base < hi; base += NT) {
            const uint64_t i = base + threadIdx.x;
            uint32_t x = i < hi ? seed_bitmap[i] : 0u;
            unsigned long long tot;
            unsigned long long pos = block_exclusive_scan<NT, unsigned long long>(__popc(x), wt, &tot);
            if (tot == 0) continue;
            if (threadIdx.x == 0) at_s = atomicAdd(&steps[0].count, tot);
            __syncthreads();
            for (pos += at_s; x; x &= x - 1) seed_out[pos++] = (int32_t)(i * 32 + (uint64_t)(__ffs(x) - 1));
            __syncthreads();
        }
        copy_wait();
        if (!grid_barrier(ctl, G, epoch, steps, &view_s)) return;
    }

    uint64_t prev_cap = ~0ull;                                // rows that the step's input region holds
    for (int t = t0; t < k; ++t) {                            // cfgs[1] and steps[1] are step t0's
        DStep *st = steps + (t - t0 + 1);
        const JoinArgs &a = args_s[t & 1];
        const DStepIn &in_s = ins_s[t & 1];
        const uint64_t R = view_s.count;
        // the previous table must have fit its region
        if (R > prev_cap) {
            if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&ctl->fail, 2u);
            return;
        }
        if (R == 0) return;                                   // no embeddings: the counts stay zero
        if (t + 1 < k) {                                      // read behind this step's barriers
            copy_words<NT>(&args_s[(t + 1) & 1], cfgs + (t - t0 + 2));
            copy_words<NT>(&ins_s[(t + 1) & 1], &st[1].in);
        }
        const LongTable lt = long_table(in_s.S, in_s.S_rows, t, R, &st->nlong);
        int32_t *const out = in_s.out;
        const uint64_t cap = in_s.out_rows;                   // from the host: 64-bit divisions take as long as a round trip
        if (blockIdx.x == 0 && threadIdx.x == 0) st->out_cap = cap;
        prev_cap = cap;
        // ---- short rows joined inline, long rows set aside (one pass over M)
        unsigned long long abytes = 0, items = 0, lbytes = 0;
        // neighbouring runs of warp work go to different SMs
        const unsigned warp = threadIdx.x >> 5;
        const uint64_t wi = (uint64_t)warp * G + blockIdx.x, nw = (uint64_t)G * (NT / 32);
        if (a.mult) {                                         // a counting query's last step
            count_tail<LW>(a, in_s.M, R, wi, nw, lt, &st->fail, &st->count, &abytes, &items, &lbytes);
        } else {
            const int nb = batch_rows(R, G, NT * ROW_RPT);
            row_pass<NT, true, ROW_RPT, LW>(a, in_s.M, R, (uint64_t)blockIdx.x * nb, (uint64_t)G * nb, nb, out, cap,
                                            &st->count, lt, &st->fail, smem, &abytes, &items, &lbytes, &st->row_ticket);
        }
        if (a.stats) {                       // one add per CTA and step
            abytes = block_sum<NT, unsigned long long>(abytes, wt);
            items = block_sum<NT, unsigned long long>(items, wt);
            if (LW) lbytes = block_sum<NT, unsigned long long>(lbytes, wt);
            if (threadIdx.x == 0) {
                if (abytes) atomicAdd(a.stats, abytes);
                if (items) atomicAdd(a.stats + 1, items);
                if (lbytes) atomicAdd(a.stats + 2, lbytes);
            }
        }
        copy_wait();
        if (!grid_barrier(ctl, G, epoch, st, &view_s)) return;
        if (view_s.fail) {                                    // the long rows do not fit
            if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&ctl->fail, view_s.fail & LONG_NEVER ? 8u : 1u);
            return;
        }
        // ---- long rows through the candidate-slot tiles
        const uint64_t ctr = view_s.nlong, L = ctr & ((1ull << lt.rbits) - 1ull), total = ctr >> lt.rbits;
        if (L > 0) {
            unsigned char *const sm = smem + warp * long_warp_smem(t, a.s.d);
            if (a.mult) long_rows_mode<LONG_TAIL>(a, lt, L, total, wi, nw, out, 0, &st->count, sm, &st->slot_ticket);
            else long_rows_join(a, lt, L, total, wi, nw, out, cap, &st->count, sm, &st->slot_ticket);
            if (!grid_barrier(ctl, G, epoch, st, &view_s)) return;
        }
        if (a.stats && blockIdx.x == 0 && threadIdx.x == 0) {      // survivors written (both models)
            const unsigned long long wbytes = 4ull * (uint64_t)(t + 1) * min((uint64_t)view_s.count, cap);
            atomicAdd(a.stats, wbytes);
            if (LW) atomicAdd(a.stats + 2, wbytes);
        }
    }
}

__global__ void k_barrier_selftest(QueryCtl *ctl, unsigned expect) {
    // every CTA waits at a barrier that expects one CTA more than exist
    __shared__ BarrierView view_s;
    unsigned epoch = 0;
    grid_barrier(ctl, expect, epoch, nullptr, &view_s);
}

std::once_flag g_join_attr_once[64];

StepDev step_dev(const gsi_graph *g, const JoinStep &s) {
    StepDev d;
    d.t = s.t;
    d.d = s.d;
    d.L = g->L;
    d.ulab = s.ulab;
    d.hom = s.hom;
    const uint32_t tmask = s.t >= 32 ? 0xffffffffu : ((1u << s.t) - 1u);
    d.inj = s.hom ? 0u : (s.inj & tmask);
    for (int i = 0; i < GSI_MAX_QUERY_VERTICES; ++i) {
        d.col[i] = i < s.d ? s.col[i] : 0;
        d.lab[i] = i < s.d ? s.lab[i] : 0;
    }
    return d;
}

}  // namespace

int64_t join_scan_scratch(uint64_t R) { return scan_blocks((int64_t)R) + 1 + ((int64_t)R + 1) / 2 + 1; }

gsi_status launch_join_scan(const gsi_graph *g, const int32_t *M, uint64_t R, const JoinStep &s, uint64_t *F,
                            uint64_t *scratch, cudaStream_t st) {
    // scratch: [scan block sums][per-row bounds as uint32]
    uint32_t *caps = reinterpret_cast<uint32_t *>(scratch + scan_blocks((int64_t)R) + 1);
    CapStoreProducer p1{M, g->off, LabelIndex{g->cl, g->dir, g->dir_min}, caps, (uint64_t)JOIN_ROW_WEIGHT, step_dev(g, s)};
    CapLoadProducer p2{caps, (uint64_t)JOIN_ROW_WEIGHT};
    GSI_CUDA_TRY(two_producer_scan(p1, p2, (int64_t)R, StoreWriter<uint64_t>{F}, scratch, st));
    return GSI_OK;
}

size_t join_smem(int rmax, int t, int d) {
    return (size_t)JOIN_NV * 8 + (size_t)(rmax + 1) * 8 + (size_t)rmax * 4 + (size_t)rmax * 2 * (d - 1) * 4 +
           (size_t)rmax * t * 4 + (size_t)JOIN_NV * 2;
}

gsi_status launch_partition(const uint64_t *F, uint64_t R, uint64_t total, int64_t *part, cudaStream_t st) {
    if (R == 0 || total == 0) return GSI_OK;
    const uint64_t ntiles = join_tiles(total);
    if (ntiles >= (1ull << 31)) {
        set_error("join: too many tiles in one launch");
        return GSI_EINVAL;
    }
    k_partition<<<(unsigned)((ntiles + 1 + 255) / 256), 256, 0, st>>>(F, (int64_t)R, total, (int64_t)ntiles, part);
    GSI_CUDA_TRY(cudaGetLastError());
    return GSI_OK;
}

gsi_status launch_join(const gsi_graph *g, const int32_t *M, uint64_t R, const JoinStep &s, const uint64_t *F,
                       uint64_t total, const int64_t *part, const uint32_t *cand, int32_t *out, uint64_t out_cap,
                       unsigned long long *out_count, int count_only, unsigned long long *stats, cudaStream_t st) {
    if (R == 0 || total == 0) return GSI_OK;
    const uint64_t ntiles = join_tiles(total);
    if (ntiles >= (1ull << 31)) {
        set_error("join: too many tiles in one launch");
        return GSI_EINVAL;
    }
    JoinArgs a;
    a.M = M; a.R = (int64_t)R; a.F = F; a.total = total; a.part = part;
    a.off = g->off; a.ci = g->ci; a.cl = LabelIndex{g->cl, g->dir, g->dir_min}; a.cand = cand;
    a.out = out; a.out_cap = out_cap; a.out_count = out_count; a.stats = stats;
    a.W = JOIN_ROW_WEIGHT;
    a.rmax = JOIN_NV / JOIN_ROW_WEIGHT + 2;
    a.count_only = count_only;
    a.s = step_dev(g, s);
    for (int i = 0; i <= GSI_MAX_QUERY_VERTICES; ++i) a.iperm[i] = i;
    for (int c = 0; c <= s.t; ++c) a.iperm[s.perm[c]] = c;
    size_t sm = join_smem(a.rmax, s.t, s.d);
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64) {                 // once per device, safe across host threads
        cudaError_t e = cudaSuccess;
        std::call_once(g_join_attr_once[dev], [&e]() {
            e = cudaFuncSetAttribute(k_join<JOIN_NT, JOIN_VT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     200 * 1024);
        });
        GSI_CUDA_TRY(e);
    }
    if (sm > 200 * 1024) {
        set_error("join: shared memory need exceeds 200 KB");
        return GSI_EINVAL;
    }
    k_join<JOIN_NT, JOIN_VT><<<(unsigned)ntiles, JOIN_NT, sm, st>>>(a);
    GSI_CUDA_TRY(cudaGetLastError());
    return GSI_OK;
}

JoinArgs make_join_args(const gsi_graph *g, const JoinStep &s, const uint32_t *cand, int count_only,
                        unsigned long long *stats) {
    JoinArgs a;
    std::memset(&a, 0, sizeof a);
    a.off = g->off; a.ci = g->ci; a.cl = LabelIndex{g->cl, g->dir, g->dir_min}; a.cand = cand;
    a.stats = stats;
    a.W = JOIN_ROW_WEIGHT;
    a.rmax = JOIN_NV / JOIN_ROW_WEIGHT + 2;
    a.count_only = count_only;
    a.s = step_dev(g, s);
    for (int i = 0; i <= GSI_MAX_QUERY_VERTICES; ++i) a.iperm[i] = i;
    for (int c = 0; c <= s.t; ++c) a.iperm[s.perm[c]] = c;
    return a;
}

size_t join_args_size() { return sizeof(JoinArgs); }

int query_memo_tables(const std::vector<JoinStep> &steps, int k) {
    int m = 0;
    for (int t = 1; t < k; ++t) m = std::max(m, std::min(steps[t].d, MEMO_EDGES));
    return m;
}

bool query_counts_tail(const std::vector<JoinStep> &steps, int k, int count_only, bool nodedup) {
    return count_only && !nodedup && k > 1 && steps[k - 1].d == 1;
}

gsi_status query_coop_configs(const gsi_graph *g, const std::vector<JoinStep> &steps, int k, const uint32_t *bitmaps,
                              const int32_t *order, int count_only, unsigned long long *stats, uint64_t *memo, bool nodedup,
                              void *cfg_host, size_t *smem) {
    JoinArgs *cfg = static_cast<JoinArgs *>(cfg_host);
    std::memset(cfg, 0, sizeof(JoinArgs));
    size_t sm = 0;
    for (int t = 1; t < k; ++t) {
        const int co = (t == k - 1) && count_only;
        cfg[t] = make_join_args(g, steps[t], bitmaps + (uint64_t)order[t] * (uint64_t)g->nwords, co, stats);
        cfg[t].memo = nodedup ? nullptr : memo;
        cfg[t].memo_n = g->n;
        cfg[t].nodedup = nodedup ? 1 : 0;
        if (co && query_counts_tail(steps, k, count_only, nodedup))
            cfg[t].mult = reinterpret_cast<unsigned long long *>(memo + (uint64_t)query_memo_tables(steps, k) * (uint64_t)g->n);
        sm = std::max(sm, long_warp_smem(steps[t].t, steps[t].d) * (JOIN_NT / 32));
        sm = std::max(sm, rows_smem(JOIN_NT, steps[t].t));
    }
    if (sm > 200 * 1024) {
        set_error("join: shared memory need exceeds 200 KB");
        return GSI_EINVAL;
    }
    *smem = sm;
    return GSI_OK;
}

gsi_status launch_query_coop(const gsi_graph *g, int t0, int k, const uint32_t *seed_bitmap, size_t sm, void *cfg_dev,
                             DStep *dsteps, QueryCtl *ctl, int *grid_out, bool listwise,
                             cudaStream_t st) {
    // the variant that also counts whole-list bytes costs registers: only on request
    const void *kern = listwise ? (const void *)k_query<JOIN_NT, true>
                                : (const void *)k_query<JOIN_NT, false>;
    int dev = 0;
    cudaGetDevice(&dev);
    // occupancy depends only on the dynamic shared memory: looked up once per
    // (device, size), as are the function attribute and the SM count
    static std::mutex mu;
    static std::map<std::tuple<int, size_t, bool>, int> occ;
    static int nsm[64];
    int per_sm = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (dev >= 0 && dev < 64 && !nsm[dev]) {
            GSI_CUDA_TRY(cudaFuncSetAttribute(k_query<JOIN_NT, false>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
            GSI_CUDA_TRY(cudaFuncSetAttribute(k_query<JOIN_NT, true>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
            GSI_CUDA_TRY(cudaDeviceGetAttribute(&nsm[dev], cudaDevAttrMultiProcessorCount, dev));
        }
        auto it = occ.find({dev, sm, listwise});
        if (it != occ.end()) {
            per_sm = it->second;
        } else {
            GSI_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, JOIN_NT, sm));
            occ[{dev, sm, listwise}] = per_sm;
        }
    }
    if (per_sm < 1) {
        set_error("join: the query kernel does not fit on an SM");
        return GSI_EINVAL;
    }
    if (per_sm > 1024 / JOIN_NT) per_sm = 1024 / JOIN_NT;     // at most 32 warps per SM
    int grid = (dev >= 0 && dev < 64 ? nsm[dev] : 152) * per_sm;
    if (grid > QUERY_MAX_CTAS) grid = QUERY_MAX_CTAS;
    *grid_out = grid;
    const JoinArgs *cfgp = static_cast<const JoinArgs *>(cfg_dev);
    int64_t nwords = g->nwords;
    void *args[] = {(void *)&cfgp, (void *)&dsteps, (void *)&t0, (void *)&k, (void *)&ctl, (void *)&seed_bitmap, (void *)&nwords};
    GSI_CUDA_TRY(cudaLaunchCooperativeKernel(kern, dim3(grid), dim3(JOIN_NT), args, sm, st));
    return GSI_OK;
}

// One step over the caller's table as a launch of k_query without the seed.
// Device memory in one block: configurations (the second is the step's), step
// records and control words, the memo, the long-row table with room for every
// row.  *ran is false, with nothing written but rows of `out`, when the block
// could not be reserved, the long rows' candidates do not fit their counter or a
// barrier wait ran past its limit (give_up: as if one had, for tests): the
// caller then takes the path without barriers.
gsi_status step_coop(const gsi_graph *g, const int32_t *M, uint64_t R, const JoinStep &s, const uint32_t *cand,
                     int32_t *out, uint64_t out_cap, uint64_t *count, bool give_up, bool *ran, cudaStream_t st) {
    *ran = false;
    struct Head {
        JoinArgs cfg[2];
        DStep steps[2];
        QueryCtl ctl;
    } h;
    std::memset(static_cast<void *>(&h), 0, sizeof h);
    const size_t sm = std::max(long_warp_smem(s.t, s.d) * (JOIN_NT / 32), rows_smem(JOIN_NT, s.t));
    if (sm > 200 * 1024 || R >> 40) return GSI_OK;
    // a memo once each vertex is met by a row on average: its clearing is 8
    // bytes a vertex and list
    const uint64_t tables = R >= (uint64_t)g->n ? (uint64_t)std::min(s.d, MEMO_EDGES) : 0;
    const uint64_t head = (sizeof h + 255) / 256 * 256, memo = tables * (uint64_t)g->n * 8;
    const uint64_t scratch = (R * (4 * (uint64_t)s.t + 16) + 64 + 15) / 16 * 16;
    unsigned char *d = nullptr;
    if (device_alloc(&d, head + memo + scratch, st) != cudaSuccess) {
        (void)cudaGetLastError();
        return GSI_OK;
    }
    h.cfg[1] = make_join_args(g, s, cand, out_cap == 0, nullptr);
    if (tables) h.cfg[1].memo = reinterpret_cast<uint64_t *>(d + head);
    h.cfg[1].memo_n = g->n;
    DStepIn &in = h.steps[1].in;
    in.M = M;
    in.out = out;
    in.out_rows = out_cap;
    in.S = reinterpret_cast<uint64_t *>(d + head + memo);
    in.S_rows = long_room(scratch / 8, s.t);
    in.t = s.t;
    h.steps[0].count = R;
    if (give_up) {
        h.ctl.bar = BAR_FAIL;
        h.ctl.fail = 4u;
    }
    Head *hd = reinterpret_cast<Head *>(d);
    int grid = 0;
    gsi_status rc = GSI_OK;
    if ((memo && cudaMemsetAsync(d + head, 0, memo, st) != cudaSuccess) ||
        cudaMemcpyAsync(d, &h, sizeof h, cudaMemcpyHostToDevice, st) != cudaSuccess) {
        set_error("join step: scratch setup failed");
        rc = GSI_ECUDA;
    }
    if (rc == GSI_OK)
        rc = launch_query_coop(g, s.t, s.t + 1, nullptr, sm, hd->cfg, hd->steps, &hd->ctl, &grid, false, st);
    if (rc == GSI_OK && (cudaMemcpyAsync(&h.steps[1], &hd->steps[1], sizeof h - offsetof(Head, steps[1]),
                                         cudaMemcpyDeviceToHost, st) != cudaSuccess ||
                         cudaStreamSynchronize(st) != cudaSuccess)) {
        set_error("join step: kernel or readback failed");
        rc = GSI_ECUDA;
    }
    cudaFreeAsync(d, st);
    *ran = rc == GSI_OK && h.ctl.fail == 0;
    if (*ran) *count = h.steps[1].count;
    return rc;
}

gsi_status selftest_barrier_timeout(int dev, unsigned long long spin_limit, double *ms) {
    GSI_CUDA_TRY(cudaSetDevice(dev));
    QueryCtl *ctl = nullptr;
    GSI_CUDA_TRY(cudaMalloc(&ctl, sizeof(QueryCtl)));
    QueryCtl h;
    std::memset(&h, 0, sizeof h);
    h.spin_limit = spin_limit;
    gsi_status rc = GSI_OK;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    if (cudaMemcpy(ctl, &h, sizeof h, cudaMemcpyHostToDevice) != cudaSuccess) rc = GSI_ECUDA;
    const unsigned grid = 8;
    unsigned expect = grid + 1;
    void *args[] = {(void *)&ctl, (void *)&expect};
    if (rc == GSI_OK) {
        cudaEventRecord(e0, 0);
        if (cudaLaunchCooperativeKernel((const void *)k_barrier_selftest, dim3(grid), dim3(JOIN_NT), args, 0, 0) !=
            cudaSuccess)
            rc = GSI_ECUDA;
        cudaEventRecord(e1, 0);
    }
    if (rc == GSI_OK && cudaMemcpy(&h, ctl, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) rc = GSI_ECUDA;
    float t = 0;
    if (rc == GSI_OK) cudaEventElapsedTime(&t, e0, e1);
    if (ms) *ms = t;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    cudaFree(ctl);
    if (rc != GSI_OK) {
        set_error("barrier self-test: launch or copy failed");
        return rc;
    }
    if (h.fail & 4u) {
        set_error("barrier self-test: the wait ran out as intended");
        return GSI_ETIMEOUT;
    }
    return GSI_OK;
}

}  // namespace gsi
