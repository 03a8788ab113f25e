// Batched execution: many queries' joins in one persistent launch.
//
// Work units come from two queues.  Seed units, listed by the host, are
// (query, range of words of the query's seed bitmap C(u_first)) pairs: a CTA
// seeds its table with the set bits of its word range and runs the query's
// join steps on those rows depth-first inside its own slice of the batch
// arena (a scratch region and two table regions used in turn), with CTA-local
// long-row tables and survivor counters.  When a step leaves more than
// split_rows rows and steps remain, the CTA keeps the first split_rows rows
// and moves the rest, in pieces of split_rows rows, to a spill area and a
// spill queue; any CTA continues such a piece from the next step.  Long rows
// with more than SPLIT_SLOTS candidates in all are handed over in the same
// way before their join.  Idle CTAs take spill units before new seed units, so
// a query whose tables grow is spread over the GPU instead of running on one
// CTA.
//
// A unit's final rows are appended to a result arena shared by all units (one
// atomic reservation per unit) and recorded in a unit record.  A unit whose
// table does not fit its slice, or whose rows do not fit the result arena,
// marks its query failed; the host runs failed queries again on the plain
// path.  Every wait (for work, for a spill unit being published) is bounded:
// a CTA that gives up sets the error word and returns, and the host then
// treats every query of the batch as failed.
#include <algorithm>
#include <cstring>
#include <vector>

#include "internal.h"
#include "join_rows.cuh"
#include "join_tile.cuh"
#include "runtime.h"

namespace gsi {
namespace {

constexpr uint64_t SPILL_SLOTS = 1ull << 18;                  // spill queue capacity (units)
constexpr unsigned long long WAIT_SPIN_LIMIT = 1ull << 26;    // x a 500 ns sleep and two round trips: half a minute at least
constexpr long long UNIT_DONE = -(1ll << 62);
// Candidate slots of a unit's long rows in one step above which the rows past
// that many slots go to other CTAs.  8,192 slots are four tiles for each warp,
// some 20 us, and handing a piece over costs about as much.  Without it one
// CTA took all hub rows of its 1,024 (10^5 slots and more, whose survivors it
// then queued: rows of many times the size), and a batch of 768 queries kept a
// tenth of the GPU busy for most of its time.
constexpr uint64_t SPLIT_SLOTS = 1ull << 13;

struct BatchQuery {
    const uint32_t *seed_bm;       // bitmap of C(u_first)
    int32_t k;
    int32_t count_only;
    unsigned status;               // 1 = failed (table or result arena overflow)
    int32_t cfg0;                  // the query's step t uses cfgs[cfg0 + t]
    unsigned long long count;      // embeddings (summed over units)
};

struct BatchItem {                 // a seed unit
    int32_t q;
    int32_t pad;
    int64_t word_lo, word_hi;
};

struct SpillUnit {                 // rows of a table to continue from step t
    int32_t q;
    int32_t t;                     // step | COUNTED: the rows are already in the step's statistics
    unsigned long long off;        // int32 offset of the rows in the spill area
    unsigned long long rows;
};

constexpr int32_t COUNTED = 1 << 8;

struct BatchRec {                  // one per unit that kept rows
    int32_t q;
    int32_t pad;
    unsigned long long off;        // int32 offset of the unit's rows in the result arena
    unsigned long long rows;
};

struct BatchCtl {                  // written by the host before every launch
    int32_t *result;               // result arena
    unsigned long long result_cap; // int32 elements
    unsigned long long next_item;  // seed queue head
    unsigned long long result_used;
    unsigned long long spill_used; // int32 elements
    unsigned long long sq_head, sq_tail;
    unsigned long long pending;    // units listed or queued and not yet finished
    unsigned long long nrecs;
    unsigned long long units;      // units processed (seed + spill)
    unsigned error;                // 1: a wait ran past its limit
    unsigned pad;
};

struct BatchArgs {
    const JoinArgs *cfgs;          // [cfg0 of the query + t]
    BatchQuery *queries;
    const BatchItem *items;
    int64_t nitems;
    BatchRec *recs;
    SpillUnit *sq;
    unsigned *sq_ready;
    unsigned long long sq_cap;
    int32_t *spill;
    unsigned long long spill_cap;  // int32 elements
    BatchCtl *ctl;
    unsigned char *arena;          // per-CTA slices
    uint64_t slice_bytes, s_bytes, t_bytes;
    uint64_t split_rows;           // 0: never split
    unsigned long long spin_limit;
};

__device__ __forceinline__ unsigned long long vload(const unsigned long long *p) {
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}

// Thread 0 only: the next unit (seed item >= 0, spill slot s as -(s + 1)),
// or UNIT_DONE once no unit is pending (or a wait ran out).
//
// Spill slots go before seed units.  While there are seed units, a CTA takes a
// slot that it sees waiting by compare-and-swap, and a seed unit where another
// was faster.  Once there are none, slots are dealt by tickets: a CTA takes the
// next number with one atomic add and owns that slot; where several race for the
// last one, the others' numbers are ahead of the queue, and each keeps its ticket
// (*ticket) until the slot is there.  So a CTA at work never holds a slot.
// (Compare-and-swap alone lets one CTA through per round trip to L2: 0.55 us a
// unit, however many CTAs were idle, which was all of the time of a batch with
// 50,000 units.  With tickets alone a slot could wait for its owner to finish a
// seed unit: 768 counting queries on 2^20 vertices took 8.55 ms, now 8.22.)
__device__ long long next_unit(const BatchArgs &b, long long *ticket) {
    BatchCtl *c = b.ctl;
    unsigned long long spins = 0;
    for (;;) {
        // read together: one round trip to L2, not one for each queue
        const unsigned long long head = vload(&c->sq_head), tail = vload(&c->sq_tail), item = vload(&c->next_item);
        const bool seeds = item < (unsigned long long)b.nitems;
        if (*ticket < 0 && head < tail) {
            if (!seeds) *ticket = (long long)atomicAdd(&c->sq_head, 1ull);
            else if (atomicCAS(&c->sq_head, head, head + 1) == head) *ticket = (long long)head;
        }
        // published (a number past the queue's end never is)
        if (*ticket >= 0 && (unsigned long long)*ticket < b.sq_cap &&
            *reinterpret_cast<volatile unsigned *>(&b.sq_ready[*ticket]) != 0u) {
            __threadfence();
            const long long h = *ticket;
            *ticket = -1;
            return -h - 1;
        }
        if (seeds && *ticket < 0) {
            const unsigned long long i = atomicAdd(&c->next_item, 1ull);
            if (i < (unsigned long long)b.nitems) return (long long)i;
        }
        if (vload(&c->pending) == 0) return UNIT_DONE;
        if (*reinterpret_cast<volatile unsigned *>(&c->error)) return UNIT_DONE;
        if (++spins > b.spin_limit) {
            atomicOr(&c->error, 1u);
            return UNIT_DONE;
        }
        // idle CTAs look less and less often: hundreds of them polling the
        // control words slow down the atomics of those at work
        __nanosleep(spins < 8 ? 64u : 500u);
    }
}

// Copies n int32, eight 16-byte pieces in flight per thread when both ends are
// 16-byte aligned (one int32 per thread and round trip was 1 KB per
// microsecond and CTA: 2.7 ms for the 3.3 MB that a unit queues at once).
template <int NT>
__device__ __forceinline__ void copy_ints(int32_t *__restrict__ dst, const int32_t *__restrict__ src, uint64_t n) {
    uint64_t i = threadIdx.x;
    if (((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0) {
        const uint64_t nv = n >> 2;
        const int4 *s4 = reinterpret_cast<const int4 *>(src);
        int4 *d4 = reinterpret_cast<int4 *>(dst);
        for (; i + 3 * NT < nv; i += 4 * NT) {
            int4 v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = __ldcg(s4 + i + j * NT);
#pragma unroll
            for (int j = 0; j < 4; ++j) d4[i + j * NT] = v[j];
        }
        for (; i < nv; i += NT) d4[i] = __ldcg(s4 + i);
        i = nv * 4 + threadIdx.x;
    }
    for (; i + 3 * NT < n; i += 4 * NT) {
        int32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = __ldcg(src + i + j * NT);
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[i + j * NT] = v[j];
    }
    for (; i < n; i += NT) dst[i] = __ldcg(src + i);
}

// Moves `rows` rows of w columns at src to the spill area and queues them as
// units of `per` rows that continue query q with step t (see SpillUnit).  All
// threads call it; false, with nothing done, when the area or the queue is
// full.  sh: two words of shared memory.
template <int NT>
__device__ bool queue_rows(const BatchArgs &b, int32_t q, int32_t t, const int32_t *src, uint64_t rows, uint64_t w,
                           uint64_t per, unsigned long long *sh) {
    BatchCtl *c = b.ctl;
    const uint64_t nch = (rows + per - 1) / per;
    if (threadIdx.x == 0) {
        const uint64_t need = (rows * w + 3) & ~3ull;         // pieces of the area start on 16 bytes
        sh[0] = ~0ull;
        const unsigned long long sp = atomicAdd(&c->spill_used, need);
        if (sp + need <= b.spill_cap) {
            unsigned long long tl = vload(&c->sq_tail);
            while (tl + nch <= b.sq_cap) {
                const unsigned long long old = atomicCAS(&c->sq_tail, tl, tl + nch);
                if (old == tl) {
                    sh[0] = sp;
                    sh[1] = tl;
                    atomicAdd(&c->pending, (unsigned long long)nch);
                    break;
                }
                tl = old;
            }
        }
    }
    __syncthreads();
    const unsigned long long sp = sh[0], s0 = sh[1];
    if (sp == ~0ull) return false;
    copy_ints<NT>(b.spill + sp, src, rows * w);
    __threadfence();                                  // the rows, before any unit that holds them
    __syncthreads();
    for (uint64_t ch = threadIdx.x; ch < nch; ch += NT) {
        SpillUnit u;
        u.q = q;
        u.t = t;
        u.off = sp + ch * per * w;
        u.rows = min(per, rows - ch * per);
        b.sq[s0 + ch] = u;
        __threadfence();
        atomicExch(&b.sq_ready[s0 + ch], 1u);
    }
    return true;
}

// Drops, without a write-back, the L2 lines that lie wholly inside
// [p, p + bytes): for a CTA's own tables once they have been read for the
// last time, so that dead rows are not written to HBM when L2 evicts them.
// The contents become undefined.  Called by all threads between a barrier
// after the last read and one before the next write of the range.
template <int NT>
__device__ __forceinline__ void discard_l2(const void *p, uint64_t bytes) {
    const uint64_t a = (uint64_t)reinterpret_cast<uintptr_t>(p);
    const uint64_t end = (a + bytes) & ~127ull;
    for (uint64_t x = ((a + 127) & ~127ull) + 128ull * threadIdx.x; x < end; x += 128ull * NT)
        asm volatile("discard.global.L2 [%0], 128;" ::"l"(x) : "memory");
}

// This CTA's slice of the arena, and its two table regions behind the scratch.
__device__ __forceinline__ unsigned char *slice(const BatchArgs &b) { return b.arena + (uint64_t)blockIdx.x * b.slice_bytes; }
__device__ __forceinline__ int32_t *table(const BatchArgs &b, int i) {
    return reinterpret_cast<int32_t *>(slice(b) + b.s_bytes + (i ? b.t_bytes : 0));
}

// The unit that a CTA works on, in shared memory: what stays the same through
// its steps and what one step leaves to the next.  Thread 0 writes it between
// barriers.  Held in registers beside the row pass and the slot tiles, which
// need all 64, it was spilled: 334 bytes of stores and 478 of loads a thread, now
// 24 and 48.  768 counting queries on 2^20 vertices: 9.5 -> 8.55 ms; 233 small
// ones on 410,886: join 172 -> 149 us.
struct Work {
    long long unit;                // seed item, -(spill slot + 1) or UNIT_DONE
    long long ticket;              // this CTA's spill slot to come, or -1
    struct {
        const int32_t *M;
        uint64_t R;
    } in[2];                       // input table and its rows of the even and the odd steps
    const uint32_t *seed_bm;
    uint64_t cap;                  // rows that the step's output table holds
    unsigned long long cnt;        // survivors of the step
    unsigned long long lctr;       // its long rows and their slots (LongTable::ctr)
    unsigned long long off, queue[2];
    uint64_t rows;                 // rows that go to the result arena
    int64_t word_lo, word_hi;
    int32_t q, k, t, cfg0, count_only;
    int32_t counted;               // the step whose statistics hold this unit's rows already
    unsigned rfail;
    int32_t skip;                  // the query already failed: its rerun redoes this work
    int32_t failed;
};

// Thread 0: takes the next unit.
__device__ void take_unit(const BatchArgs &b, Work &u) {
    const long long unit = next_unit(b, &u.ticket);
    u.unit = unit;
    if (unit == UNIT_DONE) return;
    u.counted = 0;
    u.failed = 0;
    if (unit >= 0) {
        const BatchItem it = b.items[unit];
        u.q = it.q;
        u.t = 1;
        u.word_lo = it.word_lo;
        u.word_hi = it.word_hi;
        u.in[1] = {table(b, 0), 0};
    } else {
        const SpillUnit su = b.sq[-unit - 1];
        u.q = su.q;
        u.t = su.t & (COUNTED - 1);
        u.counted = su.t & COUNTED ? u.t : 0;
        u.in[u.t & 1] = {b.spill + su.off, su.rows};
    }
    const BatchQuery *bq = b.queries + u.q;
    u.k = bq->k;
    u.cfg0 = bq->cfg0;
    u.count_only = bq->count_only;
    u.seed_bm = bq->seed_bm;
    u.skip = *reinterpret_cast<const volatile unsigned *>(&bq->status) != 0u;
    u.cap = u.count_only ? 0 : b.t_bytes / 4;         // of a one-vertex query
}

// Rows whose slots begin past SPLIT_SLOTS go to other CTAs, which join them
// from this step on; *L and *total are what is left.
template <int NT>
__device__ __noinline__ void share_long(const BatchArgs &b, Work &u, const LongTable &lt, int t, uint64_t *L, uint64_t *total,
                                        unsigned long long *wt) {
    unsigned long long keep = 0;
    for (uint64_t i = threadIdx.x; i < *L; i += NT) keep += __ldcg(lt.F + i) < SPLIT_SLOTS;
    keep = block_sum<NT, unsigned long long>(keep, wt);
    if (keep == *L) return;
    const uint64_t first = __ldcg(lt.F + keep), extra = *L - keep;
    const uint64_t per = max((uint64_t)1, extra * SPLIT_SLOTS / (*total - first));
    if (queue_rows<NT>(b, u.q, t | COUNTED, lt.rows + keep * (uint64_t)t, extra, (uint64_t)t, per, u.queue)) {
        *L = keep;
        *total = first;
    }
}

// One instance per block shape: NT threads per CTA, RPT rows per thread in
// the row pass (the batched autotuner picks one).
template <int NT, int RPT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_batch(const __grid_constant__ BatchArgs b) {
    constexpr int BNT = NT;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long wt[BNT / 32];
    __shared__ Work u;
    __shared__ LongTable lt;
    __shared__ __align__(16) JoinArgs a_s;
    const JoinArgs &a = a_s;

    if (threadIdx.x == 0) u.ticket = -1;
    for (;;) {
        if (threadIdx.x == 0) take_unit(b, u);
        __syncthreads();
        if (u.unit == UNIT_DONE) return;
        if (u.unit >= 0 && !u.skip) {
            // ---- seed: set bits of the item's words, ascending
            int32_t *const seeds = table(b, 0);
            unsigned long long run = 0;
            for (int64_t base = u.word_lo; base < u.word_hi; base += BNT) {
                const int64_t i = base + threadIdx.x;
                uint32_t x = i < u.word_hi ? u.seed_bm[i] : 0u;
                unsigned long long tot;
                unsigned long long pos = block_exclusive_scan<BNT, unsigned long long>(__popc(x), wt, &tot) + run;
                while (x) {
                    seeds[pos++] = (int32_t)(i * 32 + (int64_t)(__ffs(x) - 1));
                    x &= x - 1;
                }
                run += tot;
            }
            if (threadIdx.x == 0) u.in[1].R = run;
        }
        int t = u.t;
        for (; t < u.k && !u.skip; ++t) {
            __syncthreads();                      // the step's input is there, the previous step's readers are done
            const auto &in = u.in[t & 1];
            if (in.R == 0) break;
            int32_t *const out = table(b, t & 1);
            {   // this step's configuration in shared memory
                const uint32_t *src = reinterpret_cast<const uint32_t *>(b.cfgs + u.cfg0 + t);
                uint32_t *dst = reinterpret_cast<uint32_t *>(&a_s);
                for (int i = threadIdx.x; i < (int)(sizeof(JoinArgs) / 4); i += BNT) dst[i] = src[i];
            }
            if (threadIdx.x == BNT - 1) {         // in a warp that has little to copy
                u.cnt = 0;
                u.lctr = 0;
                u.rfail = 0;
                const JoinArgs *const cfg = b.cfgs + u.cfg0 + t;
                u.cap = cfg->out_cap;
                // long rows (bound above SHORT_MAX) in the scratch region; its
                // room from the host, as a 64-bit division takes as long as the copy
                lt = long_table(reinterpret_cast<uint64_t *>(slice(b)), cfg->total, t, in.R, &u.lctr);
            }
            __syncthreads();
            // short rows joined inline, long rows set aside
            unsigned long long abytes = 0, items = 0, lbytes = 0;
            row_pass<BNT, true, RPT, false, false>(a, in.M, in.R, 0, (uint64_t)BNT * RPT, BNT * RPT, out, u.cap, &u.cnt, lt,
                                                   &u.rfail, smem, &abytes, &items, &lbytes);
            if (a.stats && t != u.counted) {     // one add per step of a unit
                abytes = block_sum<BNT, unsigned long long>(abytes, wt);
                items = block_sum<BNT, unsigned long long>(items, wt);
                lbytes = block_sum<BNT, unsigned long long>(lbytes, wt);
                if (threadIdx.x == 0) {
                    if (abytes) atomicAdd(a.stats, abytes);
                    if (items) atomicAdd(a.stats + 1, items);
                    if (lbytes) atomicAdd(a.stats + 2, lbytes);
                }
            }
            __syncthreads();
            if (u.rfail) {                        // long-row table full: the plain path
                if (threadIdx.x == 0) u.failed = 1;
                break;
            }
            if (u.lctr) {
                uint64_t L = u.lctr & ((1ull << lt.rbits) - 1ull), total = u.lctr >> lt.rbits;
                if (b.split_rows && total > SPLIT_SLOTS && L > 1) share_long<BNT>(b, u, lt, t, &L, &total, wt);
                // the long rows' slot tiles, CTA-local
                const unsigned warp = threadIdx.x >> 5;
                long_rows_join<false>(a, lt, L, total, warp, BNT / 32, out, u.cap, &u.cnt, smem + warp * long_warp_smem(t, a.s.d));
                __syncthreads();
            }
            discard_l2<BNT>(in.M, in.R * (uint64_t)t * 4);    // this step's input is dead
            uint64_t R = u.cnt;
            if (a.stats && threadIdx.x == 0) {   // survivors written (both models)
                atomicAdd(a.stats, 4ull * (uint64_t)(t + 1) * min(R, u.cap));
                atomicAdd(a.stats + 2, 4ull * (uint64_t)(t + 1) * min(R, u.cap));
            }
            const bool last = t == u.k - 1;
            if (!last && R > u.cap) {
                if (threadIdx.x == 0) u.failed = 1;
                break;
            }
            // ---- split: keep split_rows rows, queue the rest for other CTAs
            if (!last && b.split_rows && R > b.split_rows) {
                const uint64_t keep = b.split_rows, w = (uint64_t)(t + 1);
                if (queue_rows<BNT>(b, u.q, t + 1, out + keep * w, R - keep, w, keep, u.queue)) {
                    __syncthreads();
                    discard_l2<BNT>(out + keep * w, (R - keep) * w * 4);      // the queued rows now live in the spill area
                    R = keep;
                }
            }
            if (threadIdx.x == 0) u.in[(t + 1) & 1] = {out, R};
        }
        __syncthreads();                          // readers of the last step's state are done
        // ---- final rows to the result arena
        const auto &fin = u.in[t & 1];
        if (threadIdx.x == 0) {
            // the final table must also have fit (rows past the region are lost)
            if (!u.skip && !u.count_only && fin.R > u.cap) u.failed = 1;
            BatchCtl *const c = b.ctl;
            BatchQuery *const bq = b.queries + u.q;
            uint64_t rows = (u.skip || u.failed) ? 0 : min(fin.R, u.cap);
            u.off = 0;
            if (rows > 0) {
                const unsigned long long need = (rows * (unsigned long long)u.k + 3) & ~3ull;    // on 16 bytes
                const unsigned long long o = atomicAdd(&c->result_used, need);
                if (o + need > c->result_cap) u.failed = 1;
                else u.off = o;
            }
            if (u.failed) {
                rows = 0;
                atomicOr(&bq->status, 1u);
            } else if (!u.skip) {
                atomicAdd(&bq->count, (unsigned long long)fin.R);
            }
            if (rows > 0) {
                const unsigned long long r = atomicAdd(&c->nrecs, 1ull);
                BatchRec rec;
                rec.q = u.q;
                rec.pad = 0;
                rec.off = u.off;
                rec.rows = rows;
                b.recs[r] = rec;
            }
            u.rows = rows;
        }
        __syncthreads();
        if (u.rows > 0) {
            copy_ints<BNT>(b.ctl->result + u.off, fin.M, u.rows * (uint64_t)u.k);
            __syncthreads();
            discard_l2<BNT>(fin.M, u.rows * (uint64_t)u.k * 4);   // copied out
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            BatchCtl *const c = b.ctl;
            atomicAdd(&c->units, 1ull);
            __threadfence();
            atomicAdd(&c->pending, ~0ull);        // this unit is finished (its children were added first)
        }
    }
}

// Copies every kept unit's rows from the staging area to its place in one
// tight buffer (dst[j] in int32 elements; ~0 = not kept), one CTA per record.
__global__ void __launch_bounds__(256) k_gather(const BatchQuery *__restrict__ queries,
                                                const BatchRec *__restrict__ recs,
                                                const unsigned long long *__restrict__ dst,
                                                const int32_t *__restrict__ src, int32_t *__restrict__ out,
                                                int64_t nrecs) {
    for (int64_t j = blockIdx.x; j < nrecs; j += gridDim.x) {
        const unsigned long long d = dst[j];
        if (d == ~0ull) continue;
        const uint64_t n = recs[j].rows * (uint64_t)queries[recs[j].q].k;
        const int32_t *s = src + recs[j].off;
        int32_t *o = out + d;
        for (uint64_t i = threadIdx.x; i < n; i += blockDim.x) o[i] = s[i];
    }
}

}  // namespace


// The batch kernel for a block shape (threads per CTA, rows per thread).
using BatchKernel = void (*)(BatchArgs);
BatchKernel batch_kernel(int nt, int rpt) {
    if (nt == 128) return rpt == 1 ? k_batch<128, 1> : k_batch<128, 2>;
    return rpt == 1 ? k_batch<256, 1> : k_batch<256, 2>;
}

// ------------------------------------------------------------------- host
// Sizes the launch, lists the seed units, builds the per-step configurations
// and reserves the control block (and the work area unless a workspace brings
// one).  With keep_template the initial query records also stay on the device
// so that replays can reset them with a device copy.
gsi_status batch_setup(BatchLaunch &L, gsi_graph *g, std::vector<BatchPlan> &plans, const gsi_batch_opts &o,
                       uint64_t budget, cudaStream_t st, BatchWorkspace *ws, bool stats, bool keep_template) {
    L = BatchLaunch();
    const int nq = (int)plans.size();
    L.nq = (size_t)nq;
    L.device = g->device;
    if ((o.block_threads != 0 && o.block_threads != 128 && o.block_threads != 256) ||
        (o.rows_per_thread != 0 && o.rows_per_thread != 1 && o.rows_per_thread != 2) || o.isect < 0 ||
        o.isect > ISECT_BITMAP) {
        set_error("batch: block_threads must be 128 or 256, rows_per_thread 1 or 2, isect a GSI_ISECT_* value");
        return GSI_EINVAL;
    }
    L.nt = o.block_threads ? o.block_threads : 256;
    L.rpt = o.rows_per_thread ? o.rows_per_thread : 2;
    if (stats) {
        GSI_CUDA_TRY(device_alloc(&L.dstats, 24, st));
    }
    size_t sm = long_warp_smem(1, 1) * (size_t)(L.nt / 32);
    for (int i = 0; i < nq; ++i) {
        BatchPlan &p = plans[i];
        if (!p.active) continue;
        for (int t = 1; t < p.k; ++t) {
            sm = std::max(sm, long_warp_smem(p.steps[t].t, p.steps[t].d) * (size_t)(L.nt / 32));
            sm = std::max(sm, rows_smem(L.nt, p.steps[t].t, L.rpt));
        }
    }
    if (sm > 200 * 1024) {
        set_error("batch: shared memory need exceeds 200 KB");
        return GSI_EINVAL;
    }
    L.sm = sm;
    int dev = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&L.nsm, cudaDevAttrMultiProcessorCount, dev);
    const BatchKernel kern = batch_kernel(L.nt, L.rpt);
    GSI_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    GSI_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, L.nt, sm));
    if (per_sm < 1) {
        set_error("batch: kernel does not fit on an SM");
        return GSI_EINVAL;
    }
    // memory: result arena 30% and work area 70% of the budget (a workspace
    // brings its own); the work area is a quarter spill area and three
    // quarters per-CTA slices (scratch 20%, two tables 40% each), with fewer
    // CTAs when the slices would be too small
    const uint64_t align = 256, min_table = 1ull << 20;
    L.result_bytes = ws ? ws->result_bytes : (budget * 3 / 10) / align * align;
    L.work_bytes = ws ? ws->arena_bytes : (budget - L.result_bytes) / align * align;
    L.split_rows = o.item_rows < 0 ? 0 : (o.item_rows > 0 ? (uint64_t)o.item_rows : 1024);
    L.spill_bytes = L.split_rows ? (L.work_bytes / 4) / align * align : 0;
    L.slices_bytes = L.work_bytes - L.spill_bytes;
    int grid = L.nsm * per_sm;
    while (grid > 1 && (L.slices_bytes / (uint64_t)grid) * 2 / 5 < min_table) grid /= 2;
    L.grid = grid;
    L.slice = (L.slices_bytes / (uint64_t)grid) / align * align;
    L.s_bytes = (L.slice / 5) / align * align;
    L.t_bytes = ((L.slice - L.s_bytes) / 2) / align * align;
    if (L.t_bytes < min_table) {
        L.all_plain = true;                 // too small for any slice: all on the plain path
        return GSI_OK;
    }
    // per-query records, step configurations and seed units
    std::vector<BatchQuery> bqs((size_t)nq);
    std::vector<JoinArgs> cfg;
    std::vector<BatchItem> items;
    {
        size_t total = 0;
        for (const BatchPlan &p : plans) total += p.active ? (size_t)p.k : 0;
        cfg.reserve(total);
    }
    const uint64_t max_words = std::max<uint64_t>(1, (L.t_bytes - 1024) / 128);   // seeds fit a table region
    for (int i = 0; i < nq; ++i) {
        BatchPlan &p = plans[i];
        std::memset(&bqs[i], 0, sizeof(BatchQuery));
        bqs[i].k = p.k;
        bqs[i].count_only = o.count_only;
        if (!p.active) continue;
        bqs[i].seed_bm = p.bitmaps + (uint64_t)p.order[0] * (uint64_t)g->nwords;
        bqs[i].cfg0 = (int32_t)cfg.size();
        cfg.resize(cfg.size() + (size_t)p.k);
        for (int t = 1; t < p.k; ++t) {
            const int co = (t == p.k - 1) && o.count_only;
            cfg[(size_t)bqs[i].cfg0 + t] =
                make_join_args(g, p.steps[t], p.bitmaps + (uint64_t)p.order[t] * (uint64_t)g->nwords, co, L.dstats);
            JoinArgs &c = cfg[(size_t)bqs[i].cfg0 + t];
            c.isect = o.isect;
            c.out_cap = co ? 0 : L.t_bytes / (4ull * (uint64_t)(t + 1));
            c.total = long_room(L.s_bytes / 8, t);
        }
        // word ranges of the seed bitmap holding about seeds_per_item seeds each
        const uint64_t nw = (uint64_t)g->nwords;
        const uint64_t per = o.seeds_per_item > 0 ? (uint64_t)o.seeds_per_item : 32;
        uint64_t parts = std::max<uint64_t>((p.seed_count + per - 1) / per, (nw + max_words - 1) / max_words);
        if (parts < 1) parts = 1;
        if (parts > nw) parts = nw;
        for (uint64_t j = 0; j < parts; ++j) {
            BatchItem it;
            it.q = i;
            it.pad = 0;
            it.word_lo = (int64_t)(nw * j / parts);
            it.word_hi = (int64_t)(nw * (j + 1) / parts);
            if (it.word_hi > it.word_lo) items.push_back(it);
        }
    }
    if (cfg.empty()) cfg.resize(1);
    L.nitems = items.size();
    L.ncfg = cfg.size();
    // control block: [configs][queries][query template][items][records][gather offsets][spill units][ready][ctl]
    L.sq_cap = L.split_rows ? SPILL_SLOTS : 0;
    L.rec_cap = items.size() + L.sq_cap;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    L.o_q = up(sizeof(JoinArgs) * cfg.size());
    L.o_tpl = L.o_q + up(sizeof(BatchQuery) * bqs.size());
    L.o_items = L.o_tpl + (keep_template ? up(sizeof(BatchQuery) * bqs.size()) : 0);
    L.o_recs = L.o_items + up(sizeof(BatchItem) * items.size());
    L.o_dst = L.o_recs + up(sizeof(BatchRec) * L.rec_cap);
    L.o_sq = L.o_dst + up(sizeof(unsigned long long) * L.rec_cap);
    L.o_ready = L.o_sq + up(sizeof(SpillUnit) * L.sq_cap);
    L.o_ctl = L.o_ready + up(sizeof(unsigned) * L.sq_cap);
    L.ctl_bytes = L.o_ctl + up(sizeof(BatchCtl));
    L.has_template = keep_template;
    if (device_alloc(&L.ctl, L.ctl_bytes, st) != cudaSuccess) {
        (void)cudaGetLastError();
        L.ctl = nullptr;
        set_error("batch: could not reserve the control block");
        return GSI_ENOMEM;
    }
    if (ws) {
        L.arena = ws->arena;
    } else {
        if (block_get(g->device, L.work_bytes, st, &L.own_arena) != cudaSuccess) {
            (void)cudaGetLastError();
            L.own_arena = Block();
            set_error("batch: could not reserve the batch arena");
            return GSI_ENOMEM;
        }
        L.arena = static_cast<unsigned char *>(L.own_arena.p);
    }
    GSI_CUDA_TRY(cudaMemcpyAsync(L.ctl, cfg.data(), sizeof(JoinArgs) * cfg.size(), cudaMemcpyHostToDevice, st));
    if (items.size())
        GSI_CUDA_TRY(cudaMemcpyAsync(L.ctl + L.o_items, items.data(), sizeof(BatchItem) * items.size(),
                                     cudaMemcpyHostToDevice, st));
    if (keep_template)
        GSI_CUDA_TRY(cudaMemcpyAsync(L.ctl + L.o_tpl, bqs.data(), sizeof(BatchQuery) * bqs.size(),
                                     cudaMemcpyHostToDevice, st));
    L.q_init.assign(reinterpret_cast<const unsigned char *>(bqs.data()),
                    reinterpret_cast<const unsigned char *>(bqs.data()) + sizeof(BatchQuery) * bqs.size());
    return GSI_OK;
}

// The launch's control words: counters zeroed, every seed unit pending, the
// result arena (host to device, ahead of the kernel on the stream).
gsi_status batch_enqueue_ctl(BatchLaunch &L, int32_t *result, uint64_t result_bytes, cudaStream_t st) {
    if (L.all_plain) return GSI_OK;
    BatchCtl h;
    std::memset(&h, 0, sizeof h);
    h.result = result;
    h.result_cap = result_bytes / 4;
    h.pending = L.nitems;
    GSI_CUDA_TRY(cudaMemcpyAsync(L.ctl + L.o_ctl, &h, sizeof h, cudaMemcpyHostToDevice, st));
    return GSI_OK;
}

// Query records reset, spill queue cleared, counters zeroed, then the kernel.
// With a template every step is device work only, so it can be captured.
gsi_status batch_enqueue_kernel(BatchLaunch &L, cudaStream_t st) {
    if (L.all_plain) return GSI_OK;
    BatchQuery *d_q = reinterpret_cast<BatchQuery *>(L.ctl + L.o_q);
    if (L.has_template)
        GSI_CUDA_TRY(cudaMemcpyAsync(d_q, L.ctl + L.o_tpl, L.q_init.size(), cudaMemcpyDeviceToDevice, st));
    else
        GSI_CUDA_TRY(cudaMemcpyAsync(d_q, L.q_init.data(), L.q_init.size(), cudaMemcpyHostToDevice, st));
    if (L.sq_cap) GSI_CUDA_TRY(cudaMemsetAsync(L.ctl + L.o_ready, 0, sizeof(unsigned) * L.sq_cap, st));
    if (L.dstats) GSI_CUDA_TRY(cudaMemsetAsync(L.dstats, 0, 24, st));
    if (L.nitems == 0) return GSI_OK;
    BatchArgs ba;
    ba.cfgs = reinterpret_cast<const JoinArgs *>(L.ctl);
    ba.queries = d_q;
    ba.items = reinterpret_cast<const BatchItem *>(L.ctl + L.o_items);
    ba.nitems = (int64_t)L.nitems;
    ba.recs = reinterpret_cast<BatchRec *>(L.ctl + L.o_recs);
    ba.sq = reinterpret_cast<SpillUnit *>(L.ctl + L.o_sq);
    ba.sq_ready = reinterpret_cast<unsigned *>(L.ctl + L.o_ready);
    ba.sq_cap = L.sq_cap;
    ba.spill = reinterpret_cast<int32_t *>(L.arena + L.slices_bytes);
    ba.spill_cap = L.spill_bytes / 4;
    ba.ctl = reinterpret_cast<BatchCtl *>(L.ctl + L.o_ctl);
    ba.arena = L.arena;
    ba.slice_bytes = L.slice;
    ba.s_bytes = L.s_bytes;
    ba.t_bytes = L.t_bytes;
    ba.split_rows = L.split_rows;
    ba.spin_limit = WAIT_SPIN_LIMIT;
    batch_kernel(L.nt, L.rpt)<<<L.grid, L.nt, L.sm, st>>>(ba);
    GSI_CUDA_TRY(cudaGetLastError());
    return GSI_OK;
}

// After the kernel: each plan's count, failed flag and row chunks.  With a
// workspace the kept rows are gathered into one tight buffer; otherwise the
// chunks point into `result`, which `arena` (when given) keeps alive.
gsi_status batch_collect(BatchLaunch &L, gsi_graph *g, std::vector<BatchPlan> &plans, int32_t *result,
                         std::shared_ptr<ResultArena> arena, cudaStream_t st, gsi_stats *stats, BatchWorkspace *ws) {
    const int nq = (int)plans.size();
    for (BatchPlan &p : plans) {
        p.failed = false;
        p.count = 0;
        p.chunks.clear();
        p.arena.reset();
    }
    if (L.all_plain) {
        for (BatchPlan &p : plans)
            if (p.active) p.failed = true;
        return GSI_OK;
    }
    BatchCtl rctl;
    std::memset(&rctl, 0, sizeof rctl);
    std::vector<BatchQuery> bqs((size_t)nq);
    std::vector<BatchRec> recs;
    BatchQuery *d_q = reinterpret_cast<BatchQuery *>(L.ctl + L.o_q);
    if (cudaMemcpyAsync(&rctl, L.ctl + L.o_ctl, sizeof rctl, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(bqs.data(), d_q, sizeof(BatchQuery) * bqs.size(), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        set_error("batch: kernel or readback failed");
        return GSI_ECUDA;
    }
    if (rctl.nrecs) {
        recs.resize(rctl.nrecs);
        if (cudaMemcpyAsync(recs.data(), L.ctl + L.o_recs, sizeof(BatchRec) * recs.size(), cudaMemcpyDeviceToHost,
                            st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            set_error("batch: record readback failed");
            return GSI_ECUDA;
        }
    }
    if (stats) {
        unsigned long long hb[3] = {0, 0, 0};
        if (L.dstats && cudaMemcpy(hb, L.dstats, 24, cudaMemcpyDeviceToHost) != cudaSuccess) hb[0] = hb[1] = hb[2] = 0;
        stats->join_bytes += hb[0];
        stats->batch_bytes += hb[0];
        stats->join_items += hb[1];
        stats->join_bytes_listwise += hb[2];
        stats->tiles += rctl.units;
    }
    // a wait that ran out leaves units undone: every query goes to the plain path
    const bool all_failed = rctl.error != 0;
    for (int i = 0; i < nq; ++i) {
        BatchPlan &p = plans[i];
        if (!p.active) continue;
        p.failed = all_failed || bqs[i].status != 0;
        p.count = bqs[i].count;
    }
    if (ws) {
        // gather every kept query's rows out of the reusable staging area into
        // one tight buffer (each query's rows contiguous), which the batch's
        // results share
        std::vector<unsigned long long> dst(recs.size(), ~0ull);
        std::vector<uint64_t> qrows((size_t)nq, 0), qoff((size_t)nq, 0);
        for (const BatchRec &r : recs)
            if (!plans[r.q].failed) qrows[r.q] += r.rows;
        uint64_t tot = 0;
        for (int i = 0; i < nq; ++i) {
            qoff[i] = tot;
            tot += qrows[i] * (uint64_t)plans[i].k;
        }
        std::vector<uint64_t> fill(qoff);
        for (size_t j = 0; j < recs.size(); ++j) {
            const BatchRec &r = recs[j];
            if (plans[r.q].failed) continue;
            dst[j] = fill[r.q];
            fill[r.q] += r.rows * (uint64_t)plans[r.q].k;
        }
        int32_t *buf = nullptr;
        gsi_status rc = GSI_OK;
        if (tot > 0) {
            unsigned long long *d_dst = reinterpret_cast<unsigned long long *>(L.ctl + L.o_dst);
            if (device_alloc(&buf, tot * 4, st) != cudaSuccess ||
                cudaMemcpyAsync(d_dst, dst.data(), sizeof(unsigned long long) * dst.size(), cudaMemcpyHostToDevice,
                                st) != cudaSuccess) {
                (void)cudaGetLastError();
                set_error("batch: result buffer or gather upload failed");
                rc = GSI_ENOMEM;
            } else {
                const int gblocks = (int)std::min<size_t>(recs.size(), (size_t)L.nsm * 8);
                k_gather<<<gblocks, 256, 0, st>>>(d_q, reinterpret_cast<const BatchRec *>(L.ctl + L.o_recs), d_dst,
                                                  result, buf, (int64_t)recs.size());
                if (stats) {
                    stats->kernels += 1;
                    stats->other_launches += 1;
                }
                if (cudaGetLastError() != cudaSuccess) {
                    set_error("batch: gather launch failed");
                    rc = GSI_ECUDA;
                }
            }
        }
        if (rc == GSI_OK && cudaStreamSynchronize(st) != cudaSuccess) rc = GSI_ECUDA;
        if (rc == GSI_OK && buf) {
            auto shared = std::make_shared<ResultArena>();
            shared->ptr = buf;
            shared->device = g->device;
            shared->stream = st;
            shared->own_stream = true;
            for (int i = 0; i < nq; ++i) {
                BatchPlan &p = plans[i];
                if (!p.active || p.failed || !qrows[i]) continue;
                p.chunks.push_back({buf + qoff[i], qrows[i]});
                p.arena = shared;
            }
        } else if (buf) {
            cudaFreeAsync(buf, st);
        }
        return rc;
    }
    for (const BatchRec &r : recs)
        if (!plans[r.q].failed) plans[r.q].chunks.push_back({result + r.off, r.rows});
    for (int i = 0; i < nq; ++i)
        if (plans[i].active) plans[i].arena = arena;
    return GSI_OK;
}

void batch_release(BatchLaunch &L, cudaStream_t st) {
    if (L.ctl) cudaFreeAsync(L.ctl, st);
    if (L.own_arena.p) block_put(L.device, L.own_arena, st, false);
    if (L.dstats) cudaFreeAsync(L.dstats, st);
    L = BatchLaunch();
}

// One batch launch end to end: setup, control words, kernel, collection.
gsi_status batch_run_device(gsi_graph *g, std::vector<BatchPlan> &plans, const gsi_batch_opts &o,
                            uint64_t budget, cudaStream_t st, gsi_stats *stats, BatchWorkspace *ws) {
    if (plans.empty()) return GSI_OK;
    BatchLaunch L;
    gsi_status rc = batch_setup(L, g, plans, o, budget, st, ws, stats != nullptr, false);
    int32_t *result = nullptr;
    Block blk;
    std::shared_ptr<ResultArena> arena;
    if (rc == GSI_OK && !L.all_plain) {
        if (ws) {
            result = ws->result;
        } else if (block_get(g->device, L.result_bytes, st, &blk) != cudaSuccess) {
            (void)cudaGetLastError();
            set_error("batch: could not reserve the result arena");
            rc = GSI_ENOMEM;
        } else {
            result = static_cast<int32_t *>(blk.p);
            arena = std::make_shared<ResultArena>();     // the last result to go releases it
            arena->ptr = result;
            arena->device = g->device;
            arena->stream = st;
            arena->own_stream = true;
            arena->block = blk.bytes;
        }
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (rc == GSI_OK && stats && !L.all_plain) {
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
    }
    if (rc == GSI_OK) rc = batch_enqueue_ctl(L, result, L.result_bytes, st);
    if (rc == GSI_OK && e0) cudaEventRecord(e0, st);
    if (rc == GSI_OK) rc = batch_enqueue_kernel(L, st);
    if (rc == GSI_OK && e1) cudaEventRecord(e1, st);
    if (rc == GSI_OK) rc = batch_collect(L, g, plans, result, arena, st, stats, ws);
    if (e0) {
        float ms = 0;
        if (rc == GSI_OK) cudaEventElapsedTime(&ms, e0, e1);
        stats->join_ms += ms;
        stats->batch_ms += ms;
        stats->join_launches += L.nitems ? 1 : 0;
        stats->kernels += L.nitems ? 1 : 0;
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
    }
    batch_release(L, st);
    return rc;
}

}  // namespace gsi
