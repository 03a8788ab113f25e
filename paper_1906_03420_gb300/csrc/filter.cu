// Filtering phase (Sec. III-A) and the seed of the intermediate table.
//
// The filter reads the signature table in its label-grouped copy (vertex ids
// of each label in ascending order, groups padded to whole warps), so a warp
// holds 32 vertices of one label and is only visited when some query vertex
// of the call carries that label: the label test of Sec. III-A becomes the
// choice of warps, and the remaining 15 words decide S(v) & S(u) == S(u) for
// the query vertices of that label only.  One call serves every query vertex
// of a query or of a whole batch.  Each verdict becomes a bit of the bitmap
// C(u) (the set form the join probes, Sec. V): lanes whose vertices share a
// bitmap word (consecutive, as ids ascend) OR their bits together and the
// last of them sets them with one atomicOr.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "internal.h"
#include "scan.cuh"

namespace gsi {
namespace {

constexpr int FNT = 256;

// One warp's 32 vertices against the query vertices of their label.
//
// A query vertex has few (edge label, neighbour label) pairs, so most of its
// 15 group words are zero and hold for every vertex: only the words that some
// query vertex of the label uses are read (gmask), and only a query vertex's
// own are compared (qsig[s][0], where the label itself is not needed).  On the
// medium graph (2^20 vertices, 64 labels) a 10-vertex query reads 3-6 words
// instead of 15.
//
// That choice of words pays where a query vertex's own come from the launch's
// parameters.  In a batch (WIDE) they come from memory, hundreds to a label, and
// a branch for each word made their loads wait for one another: there each
// signature is four 16-byte loads and 15 and-nots without branches.  233 queries
// of 7-8 vertices on 410,886 vertices: 219 us with 15 4-byte loads, 277 with the
// branches, 136 so.
template <bool WIDE>
__device__ __forceinline__ void filter_warp(const int32_t *__restrict__ gperm, const uint32_t *__restrict__ gsig,
                                            int64_t np, int64_t p, const uint32_t *qsig, const int32_t *qid, int32_t s0,
                                            int32_t s1, uint32_t gmask, uint32_t *scnt, int32_t nwords,
                                            uint32_t *__restrict__ bitmaps, unsigned long long *__restrict__ counts) {
    const int lane = threadIdx.x & 31;
    const int32_t v = __ldg(gperm + p);
    uint32_t x[GSI_SIG_WORDS - 1];
#pragma unroll
    for (int j = 0; j < GSI_SIG_WORDS - 1; ++j) x[j] = (gmask >> j) & 1u ? __ldg(gsig + (int64_t)j * np + p) : 0u;
    const int32_t word = v >= 0 ? (v >> 5) : -1;
    unsigned run = 0;                                 // lanes sharing my bitmap word, once needed
    for (int32_t s = s0; s < s1; ++s) {
        const uint32_t *q = qsig + (int64_t)s * GSI_SIG_WORDS;
        bool pass = v >= 0;
        if (WIDE) {                                   // a word that is not read (gmask) is zero in q too
            uint32_t miss = 0;
#pragma unroll
            for (int h = 0; h < GSI_SIG_WORDS / 4; ++h) {
                const uint4 y = __ldg(reinterpret_cast<const uint4 *>(q) + h);
                if (h) miss |= y.x & ~x[4 * h - 1];   // word 0 is the mask of the words in use
                miss |= (y.y & ~x[4 * h]) | (y.z & ~x[4 * h + 1]) | (y.w & ~x[4 * h + 2]);
            }
            pass = pass && miss == 0;
        } else {
            const uint32_t qm = q[0];
#pragma unroll
            for (int j = 0; j < GSI_SIG_WORDS - 1; ++j)
                if ((qm >> j) & 1u) {
                    const uint32_t qw = q[j + 1];
                    pass = pass && ((x[j] & qw) == qw);
                }
        }
        const unsigned b = __ballot_sync(FULL_MASK, pass);
        if (!b) continue;
        uint32_t *bm = bitmaps + (int64_t)qid[s] * nwords;
        uint32_t bit = pass ? 1u << (v & 31) : 0u;
        if (__popc(b) <= 4) {                         // few: one atomic each
            if (bit) atomicOr(&bm[word], bit);
        } else {                                      // lanes that share a word OR their bits; the last one sets them
            if (!run) run = __match_any_sync(FULL_MASK, word);
            const int first = __ffs(run) - 1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(FULL_MASK, bit, o);
                if (lane - o >= first) bit |= y;
            }
            if (31 - __clz(run) == lane && bit) atomicOr(&bm[word], bit);
        }
        if (lane == 0) {
            if (scnt) atomicAdd(&scnt[s], (uint32_t)__popc(b));
            else atomicAdd(&counts[qid[s]], (unsigned long long)__popc(b));
        }
    }
}

// meta: qid[nqv] (bitmap / counter index of sorted query vertex s),
// gstart[ngroups + 1] (query vertices of group g), wbeg[ngroups] (first warp
// of the group's label), wcum[ngroups + 1] (prefix of the groups' warps),
// gmask[ngroups] (words that the group's query vertices use).
template <bool WIDE>
__device__ __forceinline__ void filter_body(const int32_t *__restrict__ gperm, const uint32_t *__restrict__ gsig,
                                            int64_t np, const uint32_t *qsig, const int32_t *meta, int32_t ngroups,
                                            int32_t nqv, int32_t shared_counts, int32_t nwords,
                                            uint32_t *__restrict__ bitmaps, unsigned long long *__restrict__ counts,
                                            uint32_t *scnt) {
    const int32_t *qid = meta;
    const int32_t *gstart = qid + nqv;
    const int32_t *wbeg = gstart + ngroups + 1;
    const int32_t *wcum = wbeg + ngroups;
    const int32_t *gmask = wcum + ngroups + 1;
    if (shared_counts)
        for (int32_t s = threadIdx.x; s < nqv; s += FNT) scnt[s] = 0;
    __syncthreads();
    const int64_t total = wcum[ngroups];
    const int64_t stride = (int64_t)gridDim.x * (FNT / 32);
    for (int64_t aw = (int64_t)blockIdx.x * (FNT / 32) + (threadIdx.x >> 5); aw < total; aw += stride) {
        int lo = 0, hi = ngroups - 1;                  // the group whose warps hold aw
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (wcum[mid] <= aw) lo = mid;
            else hi = mid - 1;
        }
        const int64_t p = ((int64_t)wbeg[lo] + (aw - wcum[lo])) * 32 + (threadIdx.x & 31);
        filter_warp<WIDE>(gperm, gsig, np, p, qsig, qid, gstart[lo], gstart[lo + 1], (uint32_t)gmask[lo],
                    shared_counts ? scnt : nullptr, nwords, bitmaps, counts);
    }
    if (shared_counts) {
        __syncthreads();
        for (int32_t s = threadIdx.x; s < nqv; s += FNT)
            if (scnt[s]) atomicAdd(&counts[qid[s]], (unsigned long long)scnt[s]);
    }
}

// A batch's query vertices, from device memory.
__global__ void __launch_bounds__(FNT) k_filter_groups(const int32_t *__restrict__ gperm,
                                                       const uint32_t *__restrict__ gsig, int64_t np,
                                                       const uint32_t *__restrict__ qsig,
                                                       const int32_t *__restrict__ meta, int32_t ngroups,
                                                       int32_t nqv, int32_t shared_counts, int32_t nwords,
                                                       uint32_t *__restrict__ bitmaps,
                                                       unsigned long long *__restrict__ counts) {
    extern __shared__ uint32_t scnt[];
    filter_body<true>(gperm, gsig, np, qsig, meta, ngroups, nqv, shared_counts, nwords, bitmaps, counts, scnt);
}

// One query's, from the launch's own parameters: no buffer to allocate and
// nothing to upload before the kernel (two pageable copies and an allocation
// were 10 us of a single query's host time).
__global__ void __launch_bounds__(FNT) k_filter_query(const int32_t *__restrict__ gperm,
                                                      const uint32_t *__restrict__ gsig, int64_t np,
                                                      const __grid_constant__ FilterInline f, int32_t ngroups,
                                                      int32_t nqv, int32_t nwords, uint32_t *__restrict__ bitmaps,
                                                      unsigned long long *__restrict__ counts) {
    __shared__ uint32_t scnt[GSI_MAX_QUERY_VERTICES];
    filter_body<false>(gperm, gsig, np, f.sig, f.meta, ngroups, nqv, 1, nwords, bitmaps, counts, scnt);
}

struct PopcProducer {
    const uint32_t *bm;
    __device__ uint32_t operator()(int64_t i) const { return __popc(bm[i]); }
};
struct SeedWriter {
    const uint32_t *bm;
    int64_t nwords;
    int32_t *out;
    __device__ void operator()(int64_t i, uint32_t pos) const {
        if (i >= nwords) return;
        uint32_t b = bm[i];
        while (b) {
            int bit = __ffs(b) - 1;
            out[pos++] = (int32_t)(i * 32 + bit);
            b &= b - 1;
        }
    }
};

}  // namespace

void query_signatures(const int32_t *qvlab, int32_t k, const int32_t *qsrc, const int32_t *qdst,
                      const int32_t *qelab, int32_t qm, QuerySig *out, bool hom) {
    out->k = k;
    for (int u = 0; u < k; ++u) {
        for (int w = 0; w < GSI_SIG_WORDS; ++w) out->sig[u][w] = 0;
        out->sig[u][0] = (uint32_t)qvlab[u];
    }
    // a group's first pair sets its first bit, a second one the other
    auto add = [&](int u, int32_t elab, int32_t nlab) {
        const uint32_t g = sig_group(elab, nlab), bit = 1u << sig_bit(g);
        uint32_t &w = out->sig[u][sig_word(g)];
        w |= (w & bit) && !hom ? 2u * bit : bit;
    };
    for (int e = 0; e < qm; ++e) {
        add(qsrc[e], qelab[e], qvlab[qdst[e]]);
        add(qdst[e], qelab[e], qvlab[qsrc[e]]);
    }
}

// Groups the query vertices in sigs (bitmap / counter index = position in
// sigs) by label and uploads their signatures with the group table; a group
// whose label no data vertex carries is dropped (its C(u) stays empty).
gsi_status filter_plan(const gsi_graph *g, const std::vector<const uint32_t *> &sigs, FilterPlan *fp,
                       cudaStream_t st) {
    *fp = FilterPlan();
    const int32_t nqv = (int32_t)sigs.size();
    fp->nqv = nqv;
    fp->bytes = (uint64_t)nqv * (uint64_t)g->nwords * 4ull;
    if (nqv == 0) return GSI_OK;
    std::vector<int32_t> perm((size_t)nqv);
    for (int32_t i = 0; i < nqv; ++i) perm[i] = i;
    std::stable_sort(perm.begin(), perm.end(), [&](int32_t a, int32_t b) { return sigs[a][0] < sigs[b][0]; });
    std::vector<uint32_t> flat;
    std::vector<int32_t> qid, gstart, wbeg, wcum, gmask;
    flat.reserve((size_t)nqv * GSI_SIG_WORDS);
    int64_t warps = 0;
    for (int32_t i = 0; i < nqv;) {
        int32_t j = i;
        while (j < nqv && sigs[perm[j]][0] == sigs[perm[i]][0]) ++j;
        const int32_t r = g->label_rank((int32_t)sigs[perm[i]][0]);
        if (r >= 0 && g->goff[r + 1] > g->goff[r]) {
            gstart.push_back((int32_t)qid.size());
            wbeg.push_back((int32_t)(g->goff[r] / 32));
            wcum.push_back((int32_t)warps);
            warps += (g->goff[r + 1] - g->goff[r]) / 32;
            gmask.push_back(0);
            for (int32_t t = i; t < j; ++t) {
                const uint32_t *sig = sigs[perm[t]];
                uint32_t used = 0;                    // its non-zero words, in the label's place
                for (int w = 1; w < GSI_SIG_WORDS; ++w) used |= sig[w] ? 1u << (w - 1) : 0u;
                qid.push_back(perm[t]);
                flat.push_back(used);
                flat.insert(flat.end(), sig + 1, sig + GSI_SIG_WORDS);
                gmask.back() |= (int32_t)used;
            }
            fp->bytes += (uint64_t)(g->goff[r + 1] - g->goff[r]) * 4ull * (uint64_t)(1 + __builtin_popcount((unsigned)gmask.back()));
        }
        i = j;
    }
    // up to 96 KB of per-CTA counters (set once per device, outside any
    // stream capture)
    {
        static std::once_flag once[64];
        int dev = 0;
        cudaGetDevice(&dev);
        cudaError_t e = cudaSuccess;
        if (dev >= 0 && dev < 64)
            std::call_once(once[dev], [&e]() {
                e = cudaFuncSetAttribute(k_filter_groups, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
            });
        GSI_CUDA_TRY(e);
    }
    fp->ngroups = (int32_t)wbeg.size();
    fp->nq = (int32_t)qid.size();
    fp->warps = warps;
    if (fp->ngroups == 0) return GSI_OK;
    gstart.push_back(fp->nq);
    wcum.push_back((int32_t)warps);
    std::vector<int32_t> meta;
    meta.reserve(qid.size() + gstart.size() + wbeg.size() + wcum.size() + gmask.size());
    meta.insert(meta.end(), qid.begin(), qid.end());
    meta.insert(meta.end(), gstart.begin(), gstart.end());
    meta.insert(meta.end(), wbeg.begin(), wbeg.end());
    meta.insert(meta.end(), wcum.begin(), wcum.end());
    meta.insert(meta.end(), gmask.begin(), gmask.end());
    if (nqv <= GSI_MAX_QUERY_VERTICES) {              // one query: in the launch's parameters
        fp->in.reset(new FilterInline());
        std::memcpy(fp->in->sig, flat.data(), flat.size() * 4);
        std::memcpy(fp->in->meta, meta.data(), meta.size() * 4);
        return GSI_OK;
    }
    const size_t qbytes = flat.size() * 4;
    GSI_CUDA_TRY(device_alloc(&fp->d_q, qbytes + meta.size() * 4, st));
    fp->d_meta = reinterpret_cast<int32_t *>(reinterpret_cast<unsigned char *>(fp->d_q) + qbytes);
    GSI_CUDA_TRY(cudaMemcpyAsync(fp->d_q, flat.data(), qbytes, cudaMemcpyHostToDevice, st));
    GSI_CUDA_TRY(cudaMemcpyAsync(fp->d_meta, meta.data(), meta.size() * 4, cudaMemcpyHostToDevice, st));
    return GSI_OK;
}

// Zeroes the bitmaps and counters, then runs the filter kernel: stream work
// only (no host synchronisation, no allocation), so it can be captured.
gsi_status filter_enqueue(const gsi_graph *g, const FilterPlan &fp, uint32_t *bitmaps, unsigned long long *counts,
                          cudaStream_t st) {
    if (fp.nqv == 0) return GSI_OK;
    const size_t bm_bytes = filter_bitmap_bytes(g, fp.nqv);
    if (reinterpret_cast<unsigned char *>(bitmaps) + bm_bytes == reinterpret_cast<unsigned char *>(counts)) {
        GSI_CUDA_TRY(cudaMemsetAsync(bitmaps, 0, bm_bytes + (size_t)fp.nqv * 8, st));       // one block of the caller's
    } else {
        GSI_CUDA_TRY(cudaMemsetAsync(bitmaps, 0, (size_t)fp.nqv * (size_t)g->nwords * 4, st));
        GSI_CUDA_TRY(cudaMemsetAsync(counts, 0, (size_t)fp.nqv * 8, st));
    }
    if (fp.ngroups == 0) return GSI_OK;
    int64_t blocks = (fp.warps + (FNT / 32) - 1) / (FNT / 32);
    if (blocks > 152 * 8) blocks = 152 * 8;
    if (blocks < 1) blocks = 1;
    if (fp.in) {
        k_filter_query<<<(unsigned)blocks, FNT, 0, st>>>(g->gperm, g->gsig, g->np, *fp.in, fp.ngroups, fp.nq, g->nwords,
                                                         bitmaps, counts);
        GSI_CUDA_TRY(cudaGetLastError());
        return GSI_OK;
    }
    // per-CTA counters in shared memory when they fit (else global atomics)
    const size_t smem = (size_t)fp.nq * 4;
    const int shared_counts = smem <= 96 * 1024 ? 1 : 0;
    k_filter_groups<<<(unsigned)blocks, FNT, shared_counts ? smem : 0, st>>>(
        g->gperm, g->gsig, g->np, fp.d_q, fp.d_meta, fp.ngroups, fp.nq, shared_counts, g->nwords, bitmaps, counts);
    GSI_CUDA_TRY(cudaGetLastError());
    return GSI_OK;
}

void filter_plan_free(FilterPlan &fp, cudaStream_t st) {
    if (fp.d_q) cudaFreeAsync(fp.d_q, st);
    fp = FilterPlan();
}

static gsi_status launch_filter_groups(const gsi_graph *g, const std::vector<const uint32_t *> &sigs,
                                       uint32_t *bitmaps, unsigned long long *counts, cudaStream_t st,
                                       uint64_t *bytes = nullptr) {
    FilterPlan fp;
    gsi_status rc = filter_plan(g, sigs, &fp, st);
    if (bytes) *bytes = fp.bytes;
    if (rc == GSI_OK) rc = filter_enqueue(g, fp, bitmaps, counts, st);
    filter_plan_free(fp, st);
    return rc;
}

gsi_status launch_filter(const gsi_graph *g, const QuerySig &q, uint32_t *bitmaps, unsigned long long *counts,
                         cudaStream_t st, uint64_t *bytes) {
    std::vector<const uint32_t *> sigs;
    for (int u = 0; u < q.k; ++u) sigs.push_back(q.sig[u]);
    return launch_filter_groups(g, sigs, bitmaps, counts, st, bytes);
}

gsi_status launch_filter_batch(const gsi_graph *g, const std::vector<QuerySig> &qs, uint32_t *bitmaps,
                               unsigned long long *counts, cudaStream_t st) {
    std::vector<const uint32_t *> sigs;
    for (const QuerySig &q : qs)
        for (int u = 0; u < q.k; ++u) sigs.push_back(q.sig[u]);
    return launch_filter_groups(g, sigs, bitmaps, counts, st);
}

int64_t seed_scratch_words(const gsi_graph *g) { return scan_blocks(g->nwords) + 1; }

gsi_status launch_seed(const gsi_graph *g, const uint32_t *bitmap, int32_t *out, uint32_t *scratch,
                       cudaStream_t st) {
    GSI_CUDA_TRY(device_scan<uint32_t>(PopcProducer{bitmap}, g->nwords, SeedWriter{bitmap, g->nwords, out}, scratch,
                                       st));
    return GSI_OK;
}

}  // namespace gsi
