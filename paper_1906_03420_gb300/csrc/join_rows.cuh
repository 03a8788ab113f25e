// The row pass of a join step: short rows joined by one thread each, long
// rows set aside for the candidate-slot tiles.
//
// Most rows of the large steps have one or two candidates in their shortest
// label sub-list (the Alg. 4 bound).  For such a row the slot-tile path pays
// more for the bookkeeping (a bound record, a slot offset, a tile partition,
// staging, a slot-to-row map and W staging slots) than for the join itself.
// Here one thread takes one row from its bound to its survivors in a single
// pass:
//   * a CTA stages NT consecutive rows of M with coalesced loads;
//   * each thread finds its row's shortest label sub-list over the linking
//     edges (the output bound, Alg. 4);
//   * when that bound is at most SHORT_MAX, the thread tests every candidate
//     (bitmap of C(u), set subtraction against the row, membership in the
//     other linking lists: Alg. 3's set operations) and keeps a bit mask of
//     survivors;
//   * otherwise the row, with its bound record (length, linking edge, start)
//     and its place among the step's candidate slots, is appended to a
//     long-row table that the slot tiles process after a grid barrier (a hub
//     row then spreads over many warps, Sec. VI-A's load balancing done by the
//     tiles);
//   * one block-wide scan and one atomic per CTA and batch place the batch's
//     survivors in M', which the CTA writes as one coalesced run
//     (Prealloc-Combine without a second join: each survivor is written
//     once).
//
// Shared work between rows (duplicate removal, Sec. VI-B).  Rows of a step
// reuse few data vertices: consecutive rows of M' often extend the same
// row of M, and hubs recur everywhere.  Two mechanisms keep rows from
// repeating each other's work:
//   * a per-step memo holds, for each data vertex v and each of the first
//     MEMO_EDGES linking edges, where the label(u) sub-list of N(v, l) starts,
//     how long it is and, for a short one, which of its entries are in C(u); a
//     row whose vertex is in the memo skips the list lookup, the label-range
//     search and the bitmap probes (entries carry the step number, so a stale
//     entry is a miss, never a wrong answer);
//   * without a memo, the lanes of a warp whose single-edge rows share the
//     first-edge vertex v (found with __match_any_sync) elect one lane, which
//     locates the sub-list and probes the candidate bitmap C(u) for the whole
//     group once; the other lanes receive the bound and the bitmap mask by
//     shuffle and only add their own set subtraction, as Alg. 5 shares one
//     N(v, l0) fetch among the rows of a block that have the same m_i[u0'].
#pragma once

#include "join_tile.cuh"

namespace gsi {

constexpr int SHORT_MAX = 16;     // rows with at most this many candidates are joined inline

// Rows whose bound exceeds SHORT_MAX, copied (t columns) with their bound
// records, for the slot tiles.  Their candidates are slots of a flat index
// space: row i's begin at F[i], the sum of the earlier rows' lengths.  A CTA
// that sets rows aside reserves their places in the table and in the slot
// space with one atomic add on `ctr`, rows in the low rbits bits and slots
// above them, so that F ascends with the row index and is written with the
// row: no scan over the table, no pass that cuts it into tiles, and no grid
// barriers between them (they cost 14-20 us a step, more than the join of most
// steps).  rbits holds the step's row count, or the table's room where that is
// less: the reservation that leaves the room sees that it does, so a count that
// runs into the slots' bits is always of a step that has failed.  A table that is
// full fails the step with LONG_FULL, and more room helps; slots that do not fit
// the other bits (2^37 of them for the 10^8 rows of a first arena) or a sub-list
// that does not fit a bound record fail it with LONG_NEVER, and it does not.
struct LongTable {
    int32_t *rows;
    uint64_t *F;
    uint32_t *bnd;                // length | linking edge << BOUND_LEN_BITS
    uint32_t *blo;                // start of the shortest sub-list
    uint64_t cap;                 // rows the table holds
    unsigned long long *ctr;
    int rbits;
};

constexpr unsigned LONG_FULL = 1u, LONG_NEVER = 2u;

__host__ __device__ inline int long_row_bits(uint64_t R, uint64_t cap) {
    int b = 1;
    for (uint64_t x = R < cap ? R : cap; x >> b;) ++b;
    return b;
}
// How a reservation of `rows` rows and `slots` slots (below 2^63) on a counter
// that stood at `old` fails: 0 if it does not.
__host__ __device__ __forceinline__ unsigned long_fails(unsigned long long old, uint64_t rows, uint64_t slots, int rbits,
                                                        uint64_t cap) {
    const uint64_t at = old & ((1ull << rbits) - 1ull);
    return (at + rows > cap ? LONG_FULL : 0u) |
           ((old >> rbits) + slots >= 1ull << (64 - rbits) ? LONG_NEVER : 0u);
}

// The long-row table of step t, whose input has R rows, with room for `room`
// rows in the scratch region S: F, rows, bound records.
__device__ __forceinline__ LongTable long_table(uint64_t *S, uint64_t room, int t, uint64_t R, unsigned long long *ctr) {
    LongTable lt;
    lt.cap = room;
    lt.F = S;
    lt.rows = reinterpret_cast<int32_t *>(S + lt.cap);
    lt.bnd = reinterpret_cast<uint32_t *>(lt.rows + lt.cap * (uint64_t)t);
    lt.blo = lt.bnd + lt.cap;
    lt.ctr = ctr;
    lt.rbits = 64 - __clzll((long long)(min(R, lt.cap) | 1));      // long_row_bits, without its loop
    return lt;
}

constexpr int ROW_RPT = 2;        // rows per thread in one batch of the row pass
constexpr int ROW_SURV = 4;       // survivor-list entries per batch row (more are written in rounds)

// Dynamic shared memory of the row pass for CTAs of nt threads: nt * ROW_RPT
// staged rows of t columns, their candidate sub-list starts, then the
// survivor list (values, local row and candidate position).
__host__ __device__ constexpr size_t rows_smem(int nt, int t, int rpt = ROW_RPT) {
    return (size_t)nt * rpt * ((size_t)t * 4 + 4) + (size_t)nt * rpt * ROW_SURV * 6;
}

// Bulk prefetch of [p, p + bytes) into L2 (TMA engine, no registers or
// shared memory involved): the start is rounded up and the size down to 16
// bytes, so the prefetch never reaches past the range.
__device__ __forceinline__ void prefetch_l2(const void *p, uint64_t bytes) {
    const uint64_t a = (uint64_t)reinterpret_cast<uintptr_t>(p);
    const uint64_t end = (a + bytes) & ~15ull;
    for (uint64_t x = (a + 15) & ~15ull; x < end;) {
        const uint32_t chunk = (uint32_t)min(end - x, (uint64_t)1 << 20);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(x), "r"(chunk) : "memory");
        x += chunk;
    }
}

// Copies n int32 from global src to shared dst (16-byte aligned) through L2
// (the rows may have been written by other SMs), spread over NT threads: in
// 16-byte pieces when src is 16-byte aligned, four pieces in flight per
// thread; element by element otherwise.
template <int NT>
__device__ __forceinline__ void stage_rows(int32_t *dst, const int32_t *__restrict__ src, int n) {
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        const int nv = n >> 2;
        const int4 *s4 = reinterpret_cast<const int4 *>(src);
        int4 *d4 = reinterpret_cast<int4 *>(dst);
        int i = threadIdx.x;
        for (; i + 3 * NT < nv; i += 4 * NT) {
            const int4 x0 = __ldcg(s4 + i), x1 = __ldcg(s4 + i + NT), x2 = __ldcg(s4 + i + 2 * NT),
                       x3 = __ldcg(s4 + i + 3 * NT);
            d4[i] = x0;
            d4[i + NT] = x1;
            d4[i + 2 * NT] = x2;
            d4[i + 3 * NT] = x3;
        }
        for (; i < nv; i += NT) d4[i] = __ldcg(s4 + i);
        for (int e = nv * 4 + threadIdx.x; e < n; e += NT) dst[e] = __ldcg(src + e);
    } else {
        for (int e = threadIdx.x; e < n; e += NT) dst[e] = __ldcg(src + e);
    }
}

// Rows that one CTA takes at a time when R rows meet G CTAs: at most NB, and
// as few as make every CTA take the same number of batches (a table of 9,000
// rows is spread over the whole GPU in pieces of 16, instead of over ten CTAs: a
// step of so few rows is bound by the latency of one batch, 12-20 us when its
// threads were all in a few CTAs), in multiples of 8 so that a batch starts on
// 16 bytes whatever its columns.
__device__ __forceinline__ int batch_rows(uint64_t R, unsigned G, int NB) {
    const uint64_t per = (R + G - 1) / G, rounds = (per + NB - 1) / NB;
    return min(NB, max(8, ((int)((per + rounds - 1) / rounds) + 7) & ~7));
}

// Length of the whole linking list N(v, lab[j]) (for the whole-list byte count).
__device__ __forceinline__ uint32_t whole_len(const JoinArgs &a, int j, int32_t v) {
    const uint64_t seg = (uint64_t)(uint32_t)v * (uint64_t)a.s.L + (uint64_t)a.s.lab[j];
    return __ldg(a.off + seg + 1) - __ldg(a.off + seg);
}

// Candidates ci[lo + p], p < len <= 32, that are in C(u): bit p of the result.
__device__ __forceinline__ uint32_t bitmap_mask(const JoinArgs &a, uint32_t lo, uint32_t len) {
    uint32_t mask = 0;
    for (uint32_t p0 = 0; p0 < len; p0 += 4) {
        int32_t w[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = p0 + q < len ? __ldg(a.ci + lo + p0 + q) : -1;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (w[q] >= 0 && ((__ldg(a.cand + (w[q] >> 5)) >> (w[q] & 31)) & 1u)) mask |= 1u << (p0 + q);
    }
    return mask;
}

// Clears the bits of `mask` whose candidate equals a value of the row in a
// column the set subtraction tests (only columns whose query vertex carries
// u's label can hold w; none under homomorphism).
__device__ __forceinline__ uint32_t subtract_row(const JoinArgs &a, const int32_t *row, uint32_t lo, uint32_t mask) {
    const uint32_t inj = a.s.inj;
    if (!inj) return mask;
    for (uint32_t m = mask; m; m &= m - 1) {
        const int p = __ffs(m) - 1;
        const int32_t w = __ldg(a.ci + lo + (uint32_t)p);
        for (uint32_t im = inj; im; im &= im - 1)
            if (row[__ffs(im) - 1] == w) {
                mask &= ~(1u << p);
                break;
            }
    }
    return mask;
}

// One row of the pass: its bound (shortest label sub-list: length *best,
// start *lob, linking edge *jb) and the mask of its survivors among the
// first *best candidates when best <= SHORT_MAX.
template <bool LW = true, bool MEMO = true>
__device__ __forceinline__ uint32_t row_join(const JoinArgs &a, const int32_t *row, bool valid,
                                             uint32_t *best_out, uint32_t *lob_out, int *jb_out,
                                             unsigned long long *abytes, unsigned long long *items,
                                             unsigned long long *lbytes) {
    const int t = a.s.t, d = a.s.d;
    const bool stats = a.stats != nullptr;
    uint32_t mask = 0, best = 0, lob = 0;
    int jb = 0;
    if (valid) {
        uint32_t lo4[MEMO_EDGES], len4[MEMO_EDGES];
        uint64_t lsum = 0;
        uint32_t known = NO_MASK;                     // the best list's mask, if the memo has it
        best = 0xffffffffu;
#pragma unroll
        for (int j = 0; j < MEMO_EDGES; ++j) {
            lo4[j] = 0;
            len4[j] = 0;
            if (j < d) {
                uint32_t m;
                len4[j] = sublist<MEMO>(a, j, row[a.s.col[j]], &lo4[j], &m);
                lsum += len4[j];
                if (len4[j] < best) {
                    best = len4[j];
                    lob = lo4[j];
                    jb = j;
                    known = m;
                }
            }
        }
        for (int j = MEMO_EDGES; j < d; ++j) {
            uint32_t l, m;
            const uint32_t n = sublist<MEMO>(a, j, row[a.s.col[j]], &l, &m);
            lsum += n;
            if (n < best) {
                best = n;
                lob = l;
                jb = j;
                known = m;
            }
        }
        if (stats) {
            if (LW) {
                uint64_t wsum = 0;
                for (int j = 0; j < d; ++j) wsum += whole_len(a, j, row[a.s.col[j]]);
                *lbytes += row_list_bytes(t, d, wsum, best);
            }
            *abytes += row_alg_bytes(t, d, lsum, best);
            if (known != NO_MASK) *abytes -= 8ull * best - 4ull * (unsigned)__popc(known);
            *items += best;
        }
        if (best > 0 && best <= (uint32_t)SHORT_MAX) {
            if (known == NO_MASK) {
                known = bitmap_mask(a, lob, best);
                if (MEMO && a.memo && jb < MEMO_EDGES)
                    a.memo[(uint64_t)jb * (uint64_t)a.memo_n + (uint32_t)row[a.s.col[jb]]] =
                        memo_entry(t, lob, best, known);
            }
            mask = subtract_row(a, row, lob, known);
            // every other linking list must hold the candidate (Alg. 3)
            if (a.isect == ISECT_BSEARCH) {
                if (MEMO) {
#pragma unroll
                    for (int j = 0; j < MEMO_EDGES; ++j)
                        if (mask && j < d && j != jb) mask = contains_mask(a.ci, lob, mask, lo4[j], len4[j]);
                } else {                              // rows of small units: one candidate, seldom two
                    for (uint32_t m = mask; m; m &= m - 1) {
                        const int p = __ffs(m) - 1;
                        const int32_t w = __ldg(a.ci + lob + (uint32_t)p);
                        bool ok = true;
#pragma unroll
                        for (int j = 0; j < MEMO_EDGES; ++j)
                            if (ok && j < d && j != jb) ok = sorted_contains(a.ci + lo4[j], len4[j], w);
                        if (!ok) mask &= ~(1u << p);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < MEMO_EDGES; ++j) {
                    if (!mask || j >= d || j == jb) continue;
                    uint32_t keep = 0;
                    const uint32_t b0 = lo4[j], b1 = lo4[j] + len4[j];
                    if (a.isect == ISECT_MERGE) {
                        // both lists ascend: one pointer into the other list
                        uint32_t q = b0;
                        for (uint32_t m = mask; m && q < b1; m &= m - 1) {
                            const int p = __ffs(m) - 1;
                            const int32_t w = __ldg(a.ci + lob + (uint32_t)p);
                            while (q < b1 && __ldg(a.ci + q) < w) ++q;
                            if (q < b1 && __ldg(a.ci + q) == w) keep |= 1u << p;
                        }
                    } else {
                        // every element of the other list marks its position
                        // among the candidates
                        for (uint32_t q = b0; q < b1; ++q) {
                            const int32_t x = __ldg(a.ci + q);
                            uint32_t l = 0, h = best;
                            while (l < h) {
                                const uint32_t mid = (l + h) >> 1;
                                if (__ldg(a.ci + lob + mid) < x) l = mid + 1;
                                else h = mid;
                            }
                            if (l < best && __ldg(a.ci + lob + l) == x) keep |= 1u << l;
                        }
                    }
                    mask &= keep;
                }
            }
            for (int j = MEMO_EDGES; j < d && mask; ++j) {      // lists without a memo slot: searched whole
                if (j == jb) continue;
                const uint64_t seg = (uint64_t)(uint32_t)row[a.s.col[j]] * (uint64_t)a.s.L + (uint64_t)a.s.lab[j];
                const uint32_t x0 = __ldg(a.off + seg), x1 = __ldg(a.off + seg + 1);
                for (uint32_t m = mask; m; m &= m - 1) {
                    const int p = __ffs(m) - 1;
                    if (!ranked_contains(a.ci, a.cl.cl, x0, x1, (uint32_t)a.s.ulab, __ldg(a.ci + lob + (uint32_t)p)))
                        mask &= ~(1u << p);
                }
            }
        }
    }
    *best_out = best;
    *lob_out = lob;
    *jb_out = jb;
    return mask;
}

// The single-edge rows of one thread (RPT of them, rows q * NT + tid) in
// lockstep, so that each round of loads is issued for all of them at once.
// Sets best[q], lob[q] and mask[q]; rows past nb get best 0.
//
// With a memo (one query's launch), each row looks its vertex up: an entry
// with a mask is all it needs, and large steps meet each vertex many times.
// On a miss it finds the sub-list, probes the bitmap and leaves both there.
// Without one (batches), the lanes of a warp whose rows share the vertex elect
// a leader that does this for the group.
constexpr int ROW_C = 8;          // candidate values of a single-edge group loaded in the first round

template <int NT, int RPT, bool LW = true, bool MEMO = true>
__device__ __forceinline__ void rows_join_single(const JoinArgs &a, const int32_t *rowv, int nb, int lane,
                                                 uint32_t *best, uint32_t *lob, uint32_t *mask,
                                                 unsigned long long *abytes, unsigned long long *items,
                                                 unsigned long long *lbytes) {
    constexpr int C = ROW_C;
    const int t = a.s.t;
    const bool memo = MEMO && a.memo != nullptr;
    int32_t v[RPT];
    bool lead[RPT];
    int leader[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int lr = q * NT + (int)threadIdx.x;
        v[q] = lr < nb ? rowv[lr * t + a.s.col[0]] : -1 - lane;
        leader[q] = memo ? lane : __ffs(__match_any_sync(FULL_MASK, v[q])) - 1;
        lead[q] = lane == leader[q] && lr < nb;
    }
    // memo lookups, with the list offsets beside them (used on a miss)
    uint32_t x0[RPT], x1[RPT];
    uint64_t e[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        e[q] = (lead[q] && memo) ? a.memo[(uint32_t)v[q]] : 0ull;
        const uint64_t seg = (uint64_t)(uint32_t)(lead[q] ? v[q] : 0) * (uint64_t)a.s.L + (uint64_t)a.s.lab[0];
        x0[q] = lead[q] ? __ldg(a.off + seg) : 0u;
        x1[q] = lead[q] ? __ldg(a.off + seg + 1) : 0u;
    }
    bool probe[RPT], store[RPT];
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        best[q] = 0;
        lob[q] = 0;
        mask[q] = 0;
        probe[q] = store[q] = false;
        if (!lead[q]) continue;
        if (MEMO && memo_hit(e[q], t)) {
            lob[q] = (uint32_t)e[q];
            best[q] = memo_len(e[q]);
            mask[q] = memo_mask(e[q]);
            probe[q] = mask[q] == NO_MASK && best[q] <= (uint32_t)SHORT_MAX;
            if (mask[q] == NO_MASK) mask[q] = 0;
        } else {
            uint32_t h;
            label_range(a.cl, x0[q], x1[q], (uint32_t)a.s.ulab, &lob[q], &h);
            best[q] = h - lob[q];
            probe[q] = best[q] <= (uint32_t)SHORT_MAX;
            store[q] = memo && best[q] <= MEMO_LEN_MASK;
        }
    }
    // the first C candidates of every short list to probe, then their bitmap
    // words
    int32_t w[RPT][C];
#pragma unroll
    for (int q = 0; q < RPT; ++q)
#pragma unroll
        for (int p = 0; p < C; ++p)
            w[q][p] = probe[q] && (uint32_t)p < best[q] ? __ldg(a.ci + lob[q] + (uint32_t)p) : -1;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
#pragma unroll
        for (int p = 0; p < C; ++p)
            if (w[q][p] >= 0 && ((__ldg(a.cand + (w[q][p] >> 5)) >> (w[q][p] & 31)) & 1u)) mask[q] |= 1u << p;
        // candidates past the first C
        if (probe[q] && best[q] > (uint32_t)C) mask[q] |= bitmap_mask(a, lob[q] + C, best[q] - C) << C;
        if ((probe[q] && memo) || store[q])
            a.memo[(uint32_t)v[q]] = memo_entry(t, lob[q], best[q], probe[q] ? mask[q] : NO_MASK);
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
        const int lr = q * NT + (int)threadIdx.x;
        const bool valid = lr < nb;
        if (!memo) {
            best[q] = __shfl_sync(FULL_MASK, best[q], leader[q]);
            lob[q] = __shfl_sync(FULL_MASK, lob[q], leader[q]);
            mask[q] = __shfl_sync(FULL_MASK, mask[q], leader[q]);
            if (!valid) best[q] = mask[q] = 0;
        }
        if (mask[q]) mask[q] = subtract_row(a, rowv + lr * t, lob[q], mask[q]);
        if (a.stats) {
            if (LW && valid) *lbytes += row_list_bytes(t, 1, whole_len(a, 0, v[q]), best[q]);
            if (valid) {
                const bool masked = memo && !probe[q] && best[q] <= (uint32_t)SHORT_MAX;
                *abytes += masked ? row_memo_bytes(t, mask[q]) : row_alg_bytes(t, 1, best[q], best[q]);
                *items += best[q];
            }
        }
    }
}

// The row pass over rows [first, R) in batches of nbatch <= NT * RPT rows,
// batch starts `stride` apart (a grid-strided pass: first = blockIdx.x *
// nbatch, stride = gridDim.x * nbatch; one CTA alone: first = 0, stride =
// nbatch).  With a ticket counter (zero before the step) only three quarters of
// the batches go out that way, at least two to a CTA, and the rest on demand:
// rows differ in their lists, and of a step of millions of rows a quarter of
// the time went by while the last CTAs worked alone.  `a` should live in shared
// memory.  Survivors go to out (up to cap rows; `count` is exact), long rows to
// lt; *fail gets LONG_* bits when they do not fit.  MEMO false: the steps have no
// memo (batches).  When a.stats is set, adds this thread's algorithmic bytes
// (rows read, lists located and read; survivors are counted by the caller) to
// *abytes, the same under the whole-list model to *lbytes (only when LW), and its
// candidate slots to *items.
template <int NT, bool DR = true, int RPT = ROW_RPT, bool LW = true, bool MEMO = true>
__device__ void row_pass(const JoinArgs &a, const int32_t *M, uint64_t R, uint64_t first, uint64_t stride, int nbatch,
                         int32_t *__restrict__ out, uint64_t cap, unsigned long long *count, const LongTable &lt,
                         unsigned *fail, unsigned char *smem, unsigned long long *abytes,
                         unsigned long long *items, unsigned long long *lbytes,
                         unsigned long long *ticket = nullptr) {
    constexpr int NW = NT / 32, NB = NT * RPT, CCAP = NB * ROW_SURV;
    __shared__ uint32_t wt[NW];
    __shared__ unsigned long long wts[NW];              // slots of each warp's long rows
    __shared__ unsigned long long base_s, lbase_s, after_s;
    const int t = a.s.t, W1 = t + 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t *rowv = reinterpret_cast<int32_t *>(smem);                  // NB * t
    uint32_t *lobs = reinterpret_cast<uint32_t *>(rowv + NB * t);        // NB
    int32_t *comp_w = reinterpret_cast<int32_t *>(lobs + NB);           // CCAP
    uint16_t *comp_r = reinterpret_cast<uint16_t *>(comp_w + CCAP);     // local row | position << 10
    const bool write = cap > 0;
    // the output loop's fixed lane map: lane = rs * W1 + c writes column c of
    // the rs-th of the warp's rpw rows per round
    const int rpw = 32 / W1, rs = lane / W1, oc = lane - rs * W1;
    const int src_col = a.iperm[oc < W1 ? oc : 0];
    const uint64_t fixed = ticket ? max(2 * stride, R / stride * 3 / 4 * stride) : R;     // rows dealt by stride
    uint64_t next = first + stride;
    for (uint64_t r0 = first; r0 < R; r0 = next, next = after_s) {
        const int nb = (int)min((uint64_t)nbatch, R - r0);
        const int32_t *src = M + r0 * (uint64_t)t;
        if (threadIdx.x == 0 && next < R)             // the next batch's rows, while this one runs
            prefetch_l2(M + next * (uint64_t)t, min((uint64_t)nbatch, R - next) * (uint64_t)t * 4);
        stage_rows<NT>(rowv, src, nb * t);
        __syncthreads();
        // this thread's rows q * NT + tid, q < RPT (a warp's lanes hold
        // consecutive rows)
        uint32_t mask[RPT], best[RPT], lob[RPT];
        int jb[RPT];
        uint32_t n = 0, nl = 0;
        unsigned long long sl = 0;                    // slots of this thread's long rows, then their exclusive prefix
        if (DR && a.s.d == 1 && !a.nodedup) {
            rows_join_single<NT, RPT, LW, MEMO>(a, rowv, nb, lane, best, lob, mask, abytes, items, lbytes);
#pragma unroll
            for (int q = 0; q < RPT; ++q) jb[q] = 0;
        } else {
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int lr = q * NT + (int)threadIdx.x;
                const bool valid = lr < nb;
                mask[q] = row_join<LW, MEMO>(a, rowv + (valid ? lr : 0) * t, valid, &best[q], &lob[q], &jb[q],
                                          abytes, items, lbytes);
                if (!valid) best[q] = 0;
            }
        }
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            n += __popc(mask[q]);
            const bool lng = best[q] > (uint32_t)SHORT_MAX;
            nl += lng;
            sl += lng ? best[q] : 0u;
        }
        // one barrier: warp scans, warp totals through shared memory (wt is
        // written again only after the next batch's staging barrier)
        uint32_t ex, tot;
        unsigned long long stot = 0;
        {
            const uint32_t v = n | (nl << 16);
            uint32_t x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL_MASK, x, o);
                if (lane >= o) x += y;
            }
            const unsigned long long own = sl;
            if (__any_sync(FULL_MASK, nl != 0)) {
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned long long y = __shfl_up_sync(FULL_MASK, sl, o);
                    if (lane >= o) sl += y;
                }
            }
            if (lane == 31) {
                wt[warp] = x;
                wts[warp] = sl;
            }
            __syncthreads();
            uint32_t pre = 0;
            unsigned long long spre = 0;
            tot = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const uint32_t y = wt[w];
                pre += w < warp ? y : 0u;
                tot += y;
            }
            ex = pre + x - v;
            if (tot >> 16) {                          // the batch has long rows
                for (int w = 0; w < NW; ++w) {
                    const unsigned long long y = wts[w];
                    spre += w < warp ? y : 0ull;
                    stot += y;
                }
                sl = spre + sl - own;
            }
        }
        const uint32_t ntot = tot & 0xffffu, ltot = tot >> 16;
        if (threadIdx.x == 0) {                 // read after the next barrier
            after_s = next + stride;
            if (after_s >= fixed && ticket && next < R)
                after_s = fixed + atomicAdd(ticket, 1ull) * (uint64_t)nbatch;
            base_s = ntot ? atomicAdd(count, (unsigned long long)ntot) : 0ull;
            if (ltot) {
                const unsigned long long old = atomicAdd(lt.ctr, (stot << lt.rbits) | (unsigned long long)ltot);
                const unsigned f = long_fails(old, ltot, stot, lt.rbits, lt.cap);
                if (f) atomicOr(fail, f);
                lbase_s = old;
            }
        }
        // long rows to the table
        auto copy_long = [&]() {
            unsigned long long li = (lbase_s & ((1ull << lt.rbits) - 1ull)) + (ex >> 16);
            unsigned long long f = (lbase_s >> lt.rbits) + sl;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                if (best[q] <= (uint32_t)SHORT_MAX) continue;
                const int32_t *row = rowv + (q * NT + (int)threadIdx.x) * t;
                if (best[q] > BOUND_LEN_MASK) {
                    atomicOr(fail, LONG_NEVER);
                } else if (li < lt.cap) {
                    int32_t *dst = lt.rows + li * (uint64_t)t;
                    for (int c = 0; c < t; ++c) dst[c] = row[c];
                    lt.bnd[li] = best[q] | ((uint32_t)jb[q] << BOUND_LEN_BITS);
                    lt.blo[li] = lob[q];
                    lt.F[li] = f;
                }
                ++li;
                f += best[q];
            }
        };
        if (!write || ntot == 0) {
            __syncthreads();
            if (ltot) copy_long();
            __syncthreads();
            continue;
        }
        // survivors in rounds of CCAP rows: list, then one coalesced run (the
        // list needs only this batch's total; the output base arrives with
        // the first round's barrier)
        for (uint32_t rb = 0; rb < ntot; rb += CCAP) {
            const uint32_t re = min(ntot, rb + (uint32_t)CCAP);
            // each thread lists its survivors as (local row, candidate
            // position); the values are then fetched with the loads spread
            // over all threads instead of one serial chain per thread
            uint32_t i = ex & 0xffffu;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int lr = q * NT + (int)threadIdx.x;
                if (rb == 0 && mask[q]) lobs[lr] = lob[q];
                for (uint32_t m = mask[q]; m && i < re; m &= m - 1) {
                    if (i >= rb) comp_r[i - rb] = (uint16_t)(lr | ((__ffs(m) - 1) << 10));
                    ++i;
                }
            }
            __syncthreads();
            if (rb == 0 && ltot) copy_long();
            const uint32_t nr0 = re - rb;
            {   // four loads in flight per thread (shared reads first, then the list loads)
                uint32_t r = threadIdx.x;
                for (; r + 3 * NT < nr0; r += 4 * NT) {
                    uint32_t idx[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t e = comp_r[r + j * NT];
                        idx[j] = lobs[e & 1023u] + (e >> 10);
                    }
                    int32_t v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) v[j] = __ldg(a.ci + idx[j]);
#pragma unroll
                    for (int j = 0; j < 4; ++j) comp_w[r + j * NT] = v[j];
                }
                for (; r < nr0; r += NT) {
                    const uint32_t e = comp_r[r];
                    comp_w[r] = __ldg(a.ci + lobs[e & 1023u] + (e >> 10));
                }
            }
            __syncthreads();
            const uint64_t base = base_s;
            const uint64_t room = cap > base ? cap - base : 0;
            const uint32_t nrow = (uint32_t)min((uint64_t)ntot, room);
            int32_t *dst = out + (base + rb) * (uint64_t)W1;
            const uint32_t nr = nrow > rb ? min(re, nrow) - rb : 0u;
            if (rs < rpw) {
                // four rows per lane per iteration: the shared reads of all
                // four are issued before the first store
                const uint32_t step = (uint32_t)(NW * rpw);
                uint32_t r = (uint32_t)(warp * rpw + rs);
                for (; r + 3 * step < nr; r += 4 * step) {
                    int32_t v[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t rr = r + j * step;
                        v[j] = src_col == t ? comp_w[rr] : rowv[(int)(comp_r[rr] & 1023u) * t + src_col];
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) dst[(uint64_t)(r + j * step) * W1 + oc] = v[j];
                }
                for (; r < nr; r += step) {
                    const int32_t val = src_col == t ? comp_w[r] : rowv[(int)(comp_r[r] & 1023u) * t + src_col];
                    dst[(uint64_t)r * W1 + oc] = val;
                }
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------- long rows
// The slot tiles: warp wi of nw takes an equal, contiguous run of the table's
// slots, in tiles of LW_SLOTS, and works alone: no barrier, no map of the tile
// in shared memory.  The warp finds its first row with one 32-way search of F
// and from then on walks the table.  With a ticket counter (zero before the
// step) and runs long enough to pay for more searches (3 us each), a quarter of
// the slots, three quarters of long runs, is left for pieces a thirty-second as
// long that warps take on demand: slots differ in what they find, and the warps
// had been waiting for the last ones for a quarter of the time.  In each tile its lanes
//   * load the records of the rows that meet the tile (at most LW_ROWS, as
//     every long row has more than SHORT_MAX slots) and stage their columns;
//   * find their slots' rows from one 32-bit mask of row starts per group of
//     32 slots;
//   * load LW_SLOTS / 32 candidates and then as many bitmap words each, all in
//     flight together;
//   * test set subtraction and compact what is left by ballots;
//   * search it in the other lists (label sub-lists, from the step's memo or
//     searched), LW_Q candidates a lane in lockstep, and compact again: most
//     candidates are not in C(u), and searched in their slots' lanes, one after
//     the other, the rest kept few lanes and one load of each in flight (849M
//     slots of rows with three lists took 15.3 ms, 14.0 with a part dealt on
//     demand and 11.4 with both; steps of one list have a variant without it,
//     as its registers cost them 10%).
// One atomic per tile places the survivors, which the warp writes as one
// coalesced run.  What bounds it is the latency of the two rounds of loads
// (candidates, bitmap words) times the warps in flight.  CTA-wide tiles of
// 1,024 slots with five barriers each did 156 slots per ns on the medium graph
// (R-MAT 2^20, 16M edges, 64 labels); with these tiles and the table above,
// eight counting queries there went from 5558 to 4220 us and four large ones
// (2^22, 64M edges) from 22.2 to 18.1 ms.
constexpr int LW_SLOTS = 256;
constexpr int LW_G = LW_SLOTS / 32;
constexpr int LW_ROWS = LW_SLOTS / (SHORT_MAX + 1) + 2;
constexpr int LW_Q = 4;                               // candidates a lane searches for in lockstep
constexpr uint64_t LW_DEAL = 1024;                    // slots a warp from which a part is dealt on demand

// Shared memory of one warp: survivors (value, local row), rows, other lists.
__host__ __device__ constexpr size_t long_warp_smem(int t, int d) {
    return ((size_t)LW_SLOTS * 5 + (size_t)LW_ROWS * ((size_t)t * 4 + (size_t)(d - 1) * 8) + 15) / 16 * 16;
}

// LONG_TAIL (see count_tail): the table's rows are vertices, each standing for
// a.mult[v] rows; no set subtraction and no other lists.
enum { LONG_SINGLE, LONG_MULTI, LONG_TAIL };

template <int MODE, bool MEMO = true>
__device__ inline void long_rows_mode(const JoinArgs &a, const LongTable &lt, uint64_t L, uint64_t total, uint64_t wi,
                                      uint64_t nw, int32_t *__restrict__ out, uint64_t cap, unsigned long long *count,
                                      unsigned char *smem, unsigned long long *ticket = nullptr) {
    const int lane = threadIdx.x & 31;
    constexpr bool TAIL = MODE == LONG_TAIL, MULTI = MODE == LONG_MULTI;
    const int t = TAIL ? 1 : a.s.t, d = MULTI ? a.s.d : 1, dm1 = d - 1, W1 = t + 1;
    int32_t *sw = reinterpret_cast<int32_t *>(smem);
    int32_t *rowv = sw + LW_SLOTS;                                   // LW_ROWS * t
    uint32_t *lst = reinterpret_cast<uint32_t *>(rowv + LW_ROWS * t);   // LW_ROWS * 2 * dm1
    unsigned char *sr = reinterpret_cast<unsigned char *>(lst + LW_ROWS * 2 * dm1);
    // small tables: at least 64 slots a warp, so that the search pays
    const uint64_t per = max((uint64_t)64, ((total + nw - 1) / nw + 31) / 32 * 32);
    const bool deal = ticket && per >= LW_DEAL;
    const bool most = per >= 8 * LW_DEAL;
    const uint64_t run = deal ? max((uint64_t)1, (most ? per : 3 * per) / (4 * LW_SLOTS)) * LW_SLOTS : per;
    const uint64_t piece = max((uint64_t)1, per / (32 * LW_SLOTS)) * LW_SLOTS;
    uint64_t s = wi * run, w1 = min(total, s + run), r = 0;
    bool found_row = false;
    const unsigned le = lanemask_lt() | (1u << lane);
    const int rpw = 32 / W1, rs = lane / W1, oc = lane - rs * W1;
    const int src_col = a.iperm[oc];
    unsigned long long found = 0;                     // counting only: this lane's survivors
    for (;;) {
        if (s >= w1) {
            if (!deal) break;
            unsigned long long k = 0;
            if (lane == 0) k = atomicAdd(ticket, 1ull);
            s = nw * run + __shfl_sync(FULL_MASK, k, 0) * piece;
            if (s >= total) break;
            w1 = min(total, s + piece);
            found_row = false;
        }
        if (!found_row) {                             // the row that holds slot s: the last with F <= s
            found_row = true;
            r = 0;
            for (uint64_t hi = L; hi - r > 1;) {
                const uint64_t step = (hi - r + 31) / 32, p = r + (uint64_t)(lane + 1) * step;
                const int c = __popc(__ballot_sync(FULL_MASK, p < hi && __ldcg(lt.F + p) <= s));
                r += (uint64_t)c * step;
                hi = min(hi, r + step);
            }
        }
        const uint64_t e = min(s + (uint64_t)LW_SLOTS, w1);
        // lane j: the record of row r + j
        uint64_t Fj = ~0ull;
        uint32_t len = 0, lo = 0, jb = 0;
        if (r + (uint64_t)lane < L) {
            Fj = __ldcg(lt.F + r + lane);
            const uint32_t b = __ldcg(lt.bnd + r + lane);
            lo = __ldcg(lt.blo + r + lane);
            len = b & BOUND_LEN_MASK;
            jb = b >> BOUND_LEN_BITS;
        }
        const int nr = __popc(__ballot_sync(FULL_MASK, Fj < e));
        {
            const int32_t *src = lt.rows + r * (uint64_t)t;
            for (int i = lane; i < nr * t; i += 32) rowv[i] = __ldcg(src + i);
        }
        __syncwarp();
        if (MULTI && lane < nr) {
            uint32_t *l = lst + lane * 2 * dm1;
            for (int j = 0; j < d; ++j) {
                if (j == (int)jb) continue;
                uint32_t m;
                l[1] = sublist<MEMO>(a, j, rowv[lane * t + a.s.col[j]], &l[0], &m);
                l += 2;
            }
        }
        // the first slot of the row in the tile, and the list position of the
        // tile's slot 0 (modulo 2^32)
        const int start = (lane < nr && Fj > s) ? (int)(Fj - s) : 0;
        const uint32_t base = lo + (uint32_t)(s - Fj);
        const uint64_t endF = Fj + (uint64_t)len;
        const unsigned long long weight = TAIL && lane < nr ? a.mult[rowv[lane]] : 0ull;
        __syncwarp();
        int32_t w[LW_G];
        int row[LW_G];
        int before = 0;
#pragma unroll
        for (int g = 0; g < LW_G; ++g) {
            const unsigned m = __reduce_or_sync(FULL_MASK, start > 0 && (start >> 5) == g ? 1u << (start & 31) : 0u);
            row[g] = before + __popc(m & le);
            before += __popc(m);
            const uint32_t o = (uint32_t)(g * 32 + lane);
            const uint32_t cix = __shfl_sync(FULL_MASK, base, row[g]) + o;
            w[g] = s + o < e ? __ldg(a.ci + cix) : -1;
        }
        uint32_t bw[LW_G];
#pragma unroll
        for (int g = 0; g < LW_G; ++g) bw[g] = w[g] >= 0 ? __ldg(a.cand + (w[g] >> 5)) : 0u;
        unsigned ns = 0;
#pragma unroll
        for (int g = 0; g < LW_G; ++g) {
            bool ok = w[g] >= 0 && ((bw[g] >> (w[g] & 31)) & 1u);
            if (TAIL) {
                const unsigned long long x = __shfl_sync(FULL_MASK, weight, row[g]);
                found += ok ? x : 0ull;
                continue;
            }
            const int32_t *rv = rowv + row[g] * t;
            for (uint32_t im = a.s.inj; ok && im; im &= im - 1) ok = rv[__ffs(im) - 1] != w[g];
            if (!MULTI && a.count_only) {
                found += ok;
                continue;
            }
            const unsigned b = __ballot_sync(FULL_MASK, ok);
            if (ok) {
                const unsigned i = ns + __popc(b & le) - 1;
                sw[i] = w[g];
                sr[i] = (unsigned char)row[g];
            }
            ns += __popc(b);
        }
        if (MULTI && ns > 0) {
            __syncwarp();
            const unsigned n = ns;
            ns = 0;
            for (unsigned i0 = 0; i0 < n; i0 += 32 * LW_Q) {
                int32_t x[LW_Q];
                uint32_t rr[LW_Q];
                bool ok[LW_Q];
#pragma unroll
                for (int q = 0; q < LW_Q; ++q) {
                    const unsigned i = i0 + (unsigned)(q * 32 + lane);
                    ok[q] = i < n;
                    x[q] = ok[q] ? sw[i] : 0;
                    rr[q] = ok[q] ? sr[i] : 0u;
                }
                for (int j = 0; j < dm1; ++j) {
                    uint32_t at[LW_Q], m[LW_Q], end[LW_Q], left = 0;
#pragma unroll
                    for (int q = 0; q < LW_Q; ++q) {
                        const uint32_t *l = lst + (rr[q] * (uint32_t)dm1 + (uint32_t)j) * 2;
                        at[q] = l[0];
                        m[q] = ok[q] ? l[1] : 0u;
                        end[q] = at[q] + m[q];
                        left |= m[q];
                    }
                    while (left) {                    // lower bounds, in lockstep
                        left = 0;
                        int32_t y[LW_Q];
#pragma unroll
                        for (int q = 0; q < LW_Q; ++q) y[q] = m[q] ? __ldg(a.ci + at[q] + (m[q] >> 1)) : 0;
#pragma unroll
                        for (int q = 0; q < LW_Q; ++q) {
                            const uint32_t h = m[q] >> 1;
                            at[q] += m[q] && y[q] < x[q] ? m[q] - h : 0u;
                            m[q] = h;
                            left |= h;
                        }
                    }
                    int32_t y[LW_Q];
#pragma unroll
                    for (int q = 0; q < LW_Q; ++q) y[q] = ok[q] && at[q] < end[q] ? __ldg(a.ci + at[q]) : -1;
#pragma unroll
                    for (int q = 0; q < LW_Q; ++q) ok[q] = ok[q] && y[q] == x[q];
                }
                if (a.count_only) {
#pragma unroll
                    for (int q = 0; q < LW_Q; ++q) found += ok[q];
                    continue;
                }
                __syncwarp();                         // read: those that stay move to the front
#pragma unroll
                for (int q = 0; q < LW_Q; ++q) {
                    const unsigned b = __ballot_sync(FULL_MASK, ok[q]);
                    if (ok[q]) {
                        const unsigned i = ns + __popc(b & le) - 1;
                        sw[i] = x[q];
                        sr[i] = (unsigned char)rr[q];
                    }
                    ns += __popc(b);
                }
            }
        }
        if (ns) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(count, (unsigned long long)ns);
            at = __shfl_sync(FULL_MASK, at, 0);       // also orders the list before its readers
            __syncwarp();
            const uint64_t room = cap > at ? cap - at : 0;
            const unsigned nrow = (unsigned)min((uint64_t)ns, room);
            int32_t *dst = out + at * (uint64_t)W1;
            if (rs < rpw)
                for (unsigned i = (unsigned)rs; i < nrow; i += (unsigned)rpw)
                    dst[(uint64_t)i * W1 + oc] = src_col == t ? sw[i] : rowv[(int)sr[i] * t + src_col];
        }
        // a last row that ends with the tile is done
        r += (uint64_t)(nr - (__shfl_sync(FULL_MASK, endF, nr - 1) > e ? 1 : 0));
        s = e;
        __syncwarp();                                 // the staged rows are free
    }
    if (TAIL || a.count_only) {
#pragma unroll
        for (int o = 16; o; o >>= 1) found += __shfl_down_sync(FULL_MASK, found, o);
        if (lane == 0 && found) atomicAdd(count, found);
    }
}

template <bool MEMO = true>
__device__ __forceinline__ void long_rows_join(const JoinArgs &a, const LongTable &lt, uint64_t L, uint64_t total,
                                               uint64_t wi, uint64_t nw, int32_t *__restrict__ out, uint64_t cap,
                                               unsigned long long *count, unsigned char *smem,
                                               unsigned long long *ticket = nullptr) {
    if (a.s.d == 1) long_rows_mode<LONG_SINGLE, MEMO>(a, lt, L, total, wi, nw, out, cap, count, smem, ticket);
    else long_rows_mode<LONG_MULTI, MEMO>(a, lt, L, total, wi, nw, out, cap, count, smem, ticket);
}

// --------------------------------------------------------- counting tail
// The last step of a counting query with one linking edge needs no
// enumeration: row m with m[u'] = v has as many survivors as its list has
// entries in C(u), c(v) = |N(v, l) with label(u), in C(u)|, less the values of
// m itself among them.  c(v) of a short list is the population count of its
// memo mask.  For a long one the rows of each vertex are counted (a.mult), the
// first of them puts the vertex in the long table, and the tiles then go once
// over each distinct list and weigh every hit with the vertex's rows, instead
// of once over it for every row.  Rows subtract their own values by a search.
// No survivor is placed, so the pass has no shared memory and no barriers:
// each warp takes TAIL_Q * 32 rows, each lane TAIL_Q of them in lockstep.  It
// is bound by reading the table: 70M rows of 8 columns in 473 us (4.8 TB/s of
// the measured 6.7), where the row pass took 1,795 us; 84M candidates of 92
// distinct hubs that 757,034 rows met cost 6 us instead of 248.
constexpr int TAIL_Q = 4;

template <bool LW>
__device__ __noinline__ void count_tail(const JoinArgs &a, const int32_t *M, uint64_t R, uint64_t wi, uint64_t nw,
                                  const LongTable &lt, unsigned *fail, unsigned long long *count,
                                  unsigned long long *abytes, unsigned long long *items, unsigned long long *lbytes) {
    const int lane = threadIdx.x & 31, t = a.s.t, c0 = a.s.col[0];
    const uint64_t nb = (uint64_t)batch_rows(R, (unsigned)nw, TAIL_Q * 32);
    unsigned long long found = 0;                     // modulo 2^64
    for (uint64_t r0 = wi * nb; r0 < R; r0 += nw * nb) {
        const uint64_t r1 = min(R, r0 + nb);
        int32_t v[TAIL_Q];
        uint64_t e[TAIL_Q];
        uint32_t lo[TAIL_Q], len[TAIL_Q], mask[TAIL_Q];
        // the table may have been written by other SMs in this launch: plain
        // loads, ordered by the grid barrier, not the read-only path
#pragma unroll
        for (int q = 0; q < TAIL_Q; ++q) {
            const uint64_t i = r0 + (uint64_t)(q * 32 + lane);
            v[q] = i < r1 ? M[i * (uint64_t)t + c0] : -1;
        }
#pragma unroll
        for (int q = 0; q < TAIL_Q; ++q) e[q] = v[q] >= 0 ? a.memo[(uint32_t)v[q]] : 0ull;
#pragma unroll
        for (int q = 0; q < TAIL_Q; ++q) {
            lo[q] = (uint32_t)e[q];
            len[q] = memo_len(e[q]);
            mask[q] = memo_mask(e[q]);
            if (v[q] < 0) {
                len[q] = mask[q] = 0;
            } else if (!memo_hit(e[q], t) || (mask[q] == NO_MASK && len[q] <= (uint32_t)SHORT_MAX)) {
                uint32_t h;
                const uint64_t seg = (uint64_t)(uint32_t)v[q] * (uint64_t)a.s.L + (uint64_t)a.s.lab[0];
                label_range(a.cl, __ldg(a.off + seg), __ldg(a.off + seg + 1), (uint32_t)a.s.ulab, &lo[q], &h);
                len[q] = h - lo[q];
                mask[q] = len[q] <= (uint32_t)SHORT_MAX ? bitmap_mask(a, lo[q], len[q]) : NO_MASK;
                if (len[q] <= MEMO_LEN_MASK) a.memo[(uint32_t)v[q]] = memo_entry(t, lo[q], len[q], mask[q]);
                if (a.stats) *abytes += 16ull + (mask[q] != NO_MASK ? 8ull * len[q] : 0ull);
            }
        }
        // the rows' own values among the candidates: long lists are searched
        // for all TAIL_Q rows in lockstep (a hub's rows follow one another, and
        // one search after the other made their warps the step's last by far)
        for (uint32_t im = a.s.inj; im; im &= im - 1) {
            const int c = __ffs(im) - 1;
            int32_t x[TAIL_Q];
            uint32_t n[TAIL_Q], at[TAIL_Q], most = 0;
#pragma unroll
            for (int q = 0; q < TAIL_Q; ++q) {
                const bool lng = len[q] > (uint32_t)SHORT_MAX;
                x[q] = lng || mask[q] ? M[(r0 + (uint64_t)(q * 32 + lane)) * (uint64_t)t + c] : -1;
                n[q] = lng && x[q] >= 0 && ((__ldg(a.cand + (x[q] >> 5)) >> (x[q] & 31)) & 1u) ? len[q] : 0u;
                at[q] = lo[q];
                most = max(most, n[q]);
                if (!lng && x[q] >= 0)
                    for (uint32_t m = mask[q]; m; m &= m - 1)
                        found -= __ldg(a.ci + lo[q] + (uint32_t)(__ffs(m) - 1)) == x[q];
            }
            if (most == 0) continue;
            uint32_t end[TAIL_Q];
#pragma unroll
            for (int q = 0; q < TAIL_Q; ++q) end[q] = lo[q] + n[q];
            while (most) {                            // lower bounds
                most = 0;
                int32_t y[TAIL_Q];
#pragma unroll
                for (int q = 0; q < TAIL_Q; ++q) y[q] = n[q] ? __ldg(a.ci + at[q] + (n[q] >> 1)) : 0;
#pragma unroll
                for (int q = 0; q < TAIL_Q; ++q) {
                    const uint32_t h = n[q] >> 1;
                    at[q] += n[q] && y[q] < x[q] ? n[q] - h : 0u;
                    n[q] = h;
                    most |= h;
                }
            }
#pragma unroll
            for (int q = 0; q < TAIL_Q; ++q)
                if (at[q] < end[q] && __ldg(a.ci + at[q]) == x[q]) --found;
        }
#pragma unroll
        for (int q = 0; q < TAIL_Q; ++q) {
            const bool lng = len[q] > (uint32_t)SHORT_MAX;
            if (!lng) found += __popc(mask[q]);
            if (a.stats && v[q] >= 0) {               // long lists are counted where they are read, once for all their rows
                *abytes += row_memo_bytes(t, 0);
                *items += len[q];
                if (LW) *lbytes += row_list_bytes(t, 1, whole_len(a, 0, v[q]), len[q]);
            }
            const unsigned longs = __ballot_sync(FULL_MASK, lng);
            if (lng) {
                const unsigned peers = __match_any_sync(longs, v[q]);
                if (lane == __ffs(peers) - 1 &&
                    atomicAdd(a.mult + (uint32_t)v[q], (unsigned long long)__popc(peers)) == 0ull) {
                    const unsigned long long old = atomicAdd(lt.ctr, ((unsigned long long)len[q] << lt.rbits) | 1ull);
                    const unsigned long long li = old & ((1ull << lt.rbits) - 1ull), f = old >> lt.rbits;
                    const unsigned bad = long_fails(old, 1, len[q], lt.rbits, lt.cap) |
                                         (len[q] > BOUND_LEN_MASK ? LONG_NEVER : 0u);
                    if (!bad) {
                        lt.rows[li] = v[q];
                        lt.bnd[li] = len[q];
                        lt.blo[li] = lo[q];
                        lt.F[li] = f;
                        if (a.stats) *abytes += 8ull * len[q];
                    } else {
                        atomicOr(fail, bad);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) found += __shfl_down_sync(FULL_MASK, found, o);
    if (lane == 0 && found) atomicAdd(count, found);
}

}  // namespace gsi
