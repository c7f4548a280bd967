// Host side of the batched query: launch shapes, shared-memory budgets,
// the fused form's graphs and the autotuned shapes, and the count-width
// dispatch. The kernels are in query_impl.cuh.
#include <algorithm>

#include "query_impl.cuh"

namespace flinng {
namespace {

constexpr size_t kMaxSmem = 227 * 1024;   // dynamic shared memory of a CTA

inline uint32_t pow2_at_least(uint32_t v)
{
    uint32_t p = 1;
    while (p < v) p <<= 1;
    return p;
}

QArgs make_args(flinng_index *ix, const uint32_t *qb, uint32_t nq)
{
    QArgs a{};
    a.qb = qb;
    a.nq = nq;
    a.off = ix->off;
    a.cells = ix->cells;
    a.moff = ix->moff;
    a.mrec = ix->mrec;
    a.mg1 = ix->mg1;
    a.hidx = ix->hidx;
    a.hbm = ix->hbm;
    a.BRw = ix->BRw;
    a.heavy_min = ix->heavy_min;
    a.L = ix->cfg.L;
    a.W = ix->cfg.range_bits;
    a.R = ix->cfg.R;
    a.B = ix->cfg.B;
    a.BR = ix->BR;
    a.t_min = ix->cfg.min_threshold;
    a.avg_cell = uint32_t((ix->n_points + ix->cfg.B - 1) / ix->cfg.B);
    a.gcells = 1;
    a.id_bits = 1;
    while (a.id_bits < 32 && (ix->cfg.capacity - 1) >> a.id_bits) ++a.id_bits;
    return a;
}

// Members that a query walks, by the average length of its tables' lists.
uint64_t expected_members(const flinng_index *ix)
{
    const uint64_t per = (ix->n_points + ix->cfg.B - 1) / ix->cfg.B;
    return ix->n_cells * ix->cfg.L / (ix->nslot * ix->cfg.R) * per;
}

constexpr uint64_t kLightMembers = 600;

// Candidate buffer: room for one full round of members after a compaction
// to k keys; tune->cap overrides the default when large enough. The default
// holds about four times k, so that a flood of equal scores is cut early and
// seldom; its 8 bytes per entry cost resident CTAs (10^4 URL queries, k = 10:
// 1.25 ms with 512 entries, 1.34 with 1,024), and past 2,048 entries (or what two
// rounds of k need) they cost more than the cuts (4,000 configured genomic
// queries, k = 1,024: 61 us with 2,048, 157 with 8,192). Queries of a few
// hundred members flood nothing: the smallest.
void pick_buffer(QArgs &a, int NT, const QueryTuning *tune, size_t extra, size_t *smem_out, int cw, bool light)
{
    a.kp = pow2_at_least(a.k_max > 1 ? a.k_max : 2);
    // the decode appends freely up to cap - (NT + 32), then compacts: that
    // mark must stay above the kp keys a compaction keeps
    const uint32_t cap_min = pow2_at_least(a.kp + uint32_t(NT + 32) + 1);
    const uint32_t most = std::max(2048u, pow2_at_least(2 * a.kp + uint32_t(NT + 32)));
    uint32_t cap = (tune && tune->cap) ? pow2_at_least(tune->cap)
                   : light             ? cap_min
                                       : std::min(most, pow2_at_least(4 * a.kp + uint32_t(NT + 32)));
    if (cap < cap_min) cap = cap_min;
    a.lcap = a.B < kLevelCells ? (a.B + 7) & ~7u : kLevelCells;
    auto bytes = [&](uint32_t c) { return qsmem_bytes(c, a.kp, a.BR, a.lcap, NT, a.L, cw); };
    while (bytes(cap) + extra > kMaxSmem && cap > cap_min) cap >>= 1;
    a.cap = cap;
    const size_t smem = bytes(cap);
    *smem_out = smem;
    // one stop check per level group: the first of about 1,024 members (4 k for
    // larger k), then doubling to 16,384
    const uint32_t per = a.avg_cell ? a.avg_cell : 1u;
    const uint32_t g0 = std::max(1024u, 4 * a.k_max) / per;
    a.gcells = std::min(std::max(g0, 1u), a.lcap);
    a.gmax = std::min(std::max(16384u / per, a.gcells), a.lcap);
    // eight members per lane need cells that fill them
    a.wide = a.R > 1 && a.avg_cell >= 8 ? 1u : 0u;
}

}  // namespace

int query_launch(flinng_index *ix, const uint32_t *qbuckets, uint32_t nq,
                 const uint32_t *k, uint32_t k_max, uint32_t *out_ids,
                 uint16_t *out_scores, const uint32_t *out_row)
{
    return query_launch_counts(ix, qbuckets, nullptr, 0, nq, k, k_max, out_ids, out_scores, out_row);
}

int query_launch_counts(flinng_index *ix, const uint32_t *qbuckets, const uint16_t *counts, uint32_t max_count,
                        uint32_t nq, const uint32_t *k, uint32_t k_max, uint32_t *out_ids, uint16_t *out_scores,
                        const uint32_t *out_row)
{
    if (nq == 0) return FLINNG_OK;
    QArgs a = make_args(ix, qbuckets, nq);
    int cw = int(ix->cw);
    if (counts) {
        // decode from given counts: levels run to the caller's table total
        a.cnt_in = counts;
        a.L = max_count;
        cw = max_count <= 255 ? 1 : 2;
    }
    a.k = k;
    a.k_max = k_max;
    a.out_ids = out_ids;
    a.out_scores = out_scores;
    a.out_row = out_row;
    // CTA size: 512 threads for a batch that is then resident at once, since it
    // waits for its slowest query (80 and 300 queries, sets and vectors: 0.85 times
    // the time of 256 threads), else the smallest that keeps the most threads on
    // an SM (with large B*R shared memory admits only one or two CTAs)
    if (!ix->sms) FL_CUDA(cudaDeviceGetAttribute(&ix->sms, cudaDevAttrMultiProcessorCount, ix->device));
    const uint32_t sms = uint32_t(ix->sms);
    const bool light = !counts && expected_members(ix) < kLightMembers;
    int NT = 256;
    size_t smem = 0;
    uint32_t most = 0;
    for (int nt = 256; nt <= 1024; nt *= 2) {
        pick_buffer(a, nt, nullptr, 0, &smem, cw, light);
        const uint32_t ctas = uint32_t(228 * 1024 / (smem + 1024)), on = std::min(1024u, ctas * nt);
        if (on > most || (nt == 512 && nq <= sms * std::min(ctas, 2u))) {
            most = on;
            NT = nt;
        }
    }
    pick_buffer(a, NT, nullptr, 0, &smem, cw, light);
    // 32 registers a thread for a batch of more than one wave of such CTAs, where
    // shared memory admits them: more queries overlap their chains of loads (4,000
    // given counts of 60,000 reads in 128 tables, k = 10: 172 us with 64 registers,
    // 130 so; a batch resident at once, 1,200 of them, 54 and 60; 16-bit counts,
    // 4,000 queries of 512 tables, 144 and 188)
    const uint32_t sm_threads = NT == 256 && cw == 1 && 228 * 1024 / (smem + 1024) > 4 && nq > 8 * sms ? 2048 : 1024;
    if (smem > kMaxSmem)
        return set_error(FLINNG_ERR_INVALID_ARG,
                         "query: k_max=%u with B*R=%u needs %zu bytes of shared memory (> 227 KB)",
                         k_max, a.BR, smem);
    const void *fn = cw == 1 ? plain_kernel_c1(NT, ix->rw, sm_threads) : plain_kernel_c2(NT, ix->rw, sm_threads);
    FL_TRY(ensure_dyn_smem(fn, smem));
    void *args[] = {&a};
    FL_CUDA(cudaLaunchKernel(fn, dim3(nq), dim3(NT), args, smem, ix->stream));   // one CTA per query
    count_launch();
    return FLINNG_OK;
}

// Everything one fused launch needs: kernel, shape, shared memory and the
// argument blocks (kept in this struct so that a graph node can point at them).
struct FusedPlan {
    QArgs a;
    HArgs h;
    const void *fn;
    int threads;
    size_t smem;
    uint32_t grid;
    void *args[2];
};

// Shared memory of a fused CTA of nt threads; a's buffer sizes and the hash
// region's offset are set. The hash region (query buckets, hash scratch, the
// query slot) is live only before the decode keeps candidates, so it shares the
// candidate buffer with the gather's heavy-table list (the buffer's last 2 nt
// words) when both fit; otherwise it follows the query state.
static size_t fused_smem(const flinng_index *ix, QArgs &a, int nt, const QueryTuning *tune, bool light, size_t *hash_off)
{
    const size_t scratch = ix->cfg.metric == FLINNG_COSINE_SRP ? ix->cfg.dim : ix->P + (ix->P + 31) / 32;
    const size_t hash_bytes = (size_t((ix->cfg.L + 3) & ~3u) * 4 + 16 + scratch * 4 + 15) & ~size_t(15);
    size_t qbytes;
    pick_buffer(a, nt, tune, 0, &qbytes, int(ix->cw), light);
    *hash_off = 0;
    if (hash_bytes + size_t(nt) * 8 <= size_t(a.cap) * 8) return qbytes;
    pick_buffer(a, nt, tune, hash_bytes, &qbytes, int(ix->cw), light);
    *hash_off = qbytes;
    return qbytes + hash_bytes;
}

bool query_fused_fits(const flinng_index *ix, uint32_t k_max)
{
    QArgs a{};
    a.L = ix->cfg.L;
    a.B = ix->cfg.B;
    a.R = ix->cfg.R;
    a.BR = ix->BR;
    a.k_max = k_max;
    size_t off;
    return fused_smem(ix, a, 128, nullptr, true, &off) <= kMaxSmem;
}

static int fused_prepare(flinng_index *ix, const FusedQuery &fq, const uint32_t *k, uint32_t k_max,
                         uint32_t *out_ids, uint16_t *out_scores, const QueryTuning *tune,
                         uint32_t grid_for, FusedPlan *P)
{
    const uint32_t nq = fq.nq;
    if (!ix->sms) FL_CUDA(cudaDeviceGetAttribute(&ix->sms, cudaDevAttrMultiProcessorCount, ix->device));
    const int sms = ix->sms;
    QArgs &a = P->a;
    HArgs &h = P->h;
    a = make_args(ix, nullptr, nq);
    a.k = k;
    a.k_max = k_max;
    a.out_ids = out_ids;
    a.out_scores = out_scores;
    a.out_row = fq.out_row;
    h = HArgs{};
    const bool srp = ix->cfg.metric == FLINNG_COSINE_SRP;
    h.K = ix->cfg.K;
    h.qnext = ix->qnext;
    if (srp) {
        h.x = fq.x;
        h.ldx = fq.ldx;
        h.w = ix->srp_w;
        h.d = ix->cfg.dim;
        h.gamma2 = ix->srp_margin_gamma;
        h.tiny = float(h.d) * ldexpf(1.0f, -146);
        h.gamma64 = ix->srp_gamma64;
        h.stats = ix->stats;
    } else {
        h.q_off = fq.off;
        h.q_el = fq.elems;
        h.nb = ix->P;
        h.da = ix->doph_a;
        h.db = ix->doph_b;
        h.seed = ix->doph_seed;
        h.ba = ix->bucket_a;
        h.bc = ix->bucket_c;
        h.draw = ix->doph_draw;
    }
    const bool light = expected_members(ix) < kLightMembers;
    auto shape = [&](int nt) { P->smem = fused_smem(ix, a, nt, tune, light, &h.hash_off); };
    // CTA size, unless tuned. A batch that is resident at once takes 512 threads:
    // it waits for its slowest query, whose phases scale with its CTA (1 query
    // of the recall-target genomic index: 35 us with 512, 43 with 256, 65 with
    // 128). A larger batch takes 256 when shared memory still admits four such
    // CTAs per SM, so that more queries overlap their phases (10^4 URL queries:
    // 1.24 ms against 1.46 with 512; 1,000 configured genomic queries: 35 us
    // against 45), else 512. Where a query walks few members (the lists of its
    // tables, by their average length, lead to a few hundred) its time is that of
    // barriers and scans, which grow with the CTA: more than two such queries per
    // SM take 256 threads, more than four 128, if that leaves the SM three quarters
    // of its threads (30,000 reads in 16 tables, k = 10, 512 / 256 / 128 threads: 600
    // queries 18.6 / 14.6 / 14.5 us, 4,000 queries 92 / 57 / 46).
    int NT = tune && tune->threads ? int(tune->threads) : 512;
    shape(NT);
    auto fit = [&]() { return uint32_t(228 * 1024 / (P->smem + 1024)); };
    // Threads per SM by registers: with 16-bit counts 1,024 where shared memory
    // (or the batch) fills no more of the SM, since 64 registers then cost nothing
    // (4,000 recall-target queries: 382 -> 363 us; at 2,048 possible threads, 349
    // tables in 2,000 cells, they cost 187 -> 231 us).
    uint32_t sm_threads = srp ? 1024 : 2048;
    const bool both = !srp && ix->cw == 2;
    if (!tune || !tune->threads) {
        const bool small = light && nq > 2 * uint32_t(sms);
        if (both && nq <= uint32_t(sms) * std::min(fit(), 2u)) {
            sm_threads = 1024;
        } else if (small || nq > uint32_t(sms) * std::min(fit(), sm_threads / 512)) {
            shape(256);
            const uint32_t f256 = std::min(fit(), sm_threads / 256);
            if (small && f256 >= 4 && nq > 4 * uint32_t(sms)) {
                shape(128);
                if (8 * std::min(fit(), sm_threads / 128) >= 11 * f256) NT = 128;
                else shape(256);
            }
            if (NT == 512) {
                if (f256 >= 4) NT = 256;
                else shape(512);
            }
        }
    }
    // a shape that asks for too much (the usual one or a tuned one): smaller CTAs
    while (P->smem > kMaxSmem && NT > 128) shape(NT /= 2);
    if (both && fit() * uint32_t(NT) <= 1024) sm_threads = 1024;
    if (P->smem > kMaxSmem)
        return set_error(FLINNG_ERR_INVALID_ARG, "fused query: %zu bytes of shared memory needed (> 227 KB)", P->smem);
    P->fn = ix->cw == 1 ? fused_kernel_c1(NT, ix->rw, srp, sm_threads) : fused_kernel_c2(NT, ix->rw, srp, sm_threads);
    P->threads = NT;
    FL_TRY(ensure_dyn_smem(P->fn, P->smem));
    int per_sm = 0;
    for (uint32_t i = 0; i < ix->n_occ; ++i) {
        const OccEntry &e = ix->occ[i];
        if (e.fn == P->fn && e.threads == NT && e.smem == P->smem) per_sm = e.per_sm;
    }
    if (!per_sm) {
        FL_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, P->fn, NT, P->smem));
        if (per_sm < 1) per_sm = 1;
        const uint32_t slot = ix->n_occ < 8 ? ix->n_occ++ : 7;
        ix->occ[slot] = OccEntry{P->fn, NT, P->smem, per_sm};
    }
    uint32_t want = (tune && tune->ctas_per_sm) ? tune->ctas_per_sm : uint32_t(per_sm);
    if (want > uint32_t(per_sm)) want = per_sm;
    uint64_t grid = uint64_t(sms) * want;
    if (grid > grid_for) grid = grid_for;
    P->grid = uint32_t(grid ? grid : 1);
    // every query has a CTA of its own: no counter to clear and draw from
    if (P->grid == nq && grid_for == nq) h.qnext = nullptr;
    P->args[0] = &P->a;
    P->args[1] = &P->h;
    return FLINNG_OK;
}

int query_fused_launch(flinng_index *ix, const FusedQuery &fq, const uint32_t *k, uint32_t k_max,
                       uint32_t *out_ids, uint16_t *out_scores, const QueryTuning *tune)
{
    if (fq.nq == 0) return FLINNG_OK;
    FusedPlan P;
    FL_TRY(fused_prepare(ix, fq, k, k_max, out_ids, out_scores, tune, fq.nq, &P));
    if (ix->cfg.metric == FLINNG_COSINE_SRP)
        FL_CUDA(cudaMemsetAsync(ix->stats, 0, kStats * sizeof(unsigned long long), ix->stream));
    if (P.h.qnext) FL_CUDA(cudaMemsetAsync(ix->qnext, 0, sizeof(uint32_t), ix->stream));
    FL_CUDA(cudaLaunchKernel(P.fn, dim3(P.grid), dim3(P.threads), P.args, P.smem, ix->stream));
    count_launch();
    return FLINNG_OK;
}

// Graph form: one CUDA graph per batch-size class (nq rounded up to a power
// of two) and per result width, built once and replayed; each call only
// rewrites the kernel node's arguments (query and output pointers, nq).
int query_graph_launch(flinng_index *ix, const FusedQuery &fq, const uint32_t *k, uint32_t k_max,
                       uint32_t *out_ids, uint16_t *out_scores, const QueryTuning *tune)
{
    const uint32_t nq = fq.nq;
    if (nq == 0) return FLINNG_OK;
    uint32_t bucket = 0;
    while ((1u << bucket) < nq) ++bucket;
    FusedPlan P;
    FL_TRY(fused_prepare(ix, fq, k, k_max, out_ids, out_scores, tune, 1u << bucket, &P));
    QueryGraph &g = ix->graphs[bucket];
    cudaKernelNodeParams kp{};
    kp.func = const_cast<void *>(P.fn);
    kp.gridDim = dim3(P.grid);
    kp.blockDim = dim3(P.threads);
    kp.sharedMemBytes = (unsigned)P.smem;
    kp.kernelParams = P.args;
    const bool srp = ix->cfg.metric == FLINNG_COSINE_SRP;
    if (!g.exec || g.fn != P.fn || g.smem != P.smem || g.grid != P.grid) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        if (g.graph) cudaGraphDestroy(g.graph);
        g = QueryGraph{};
        FL_CUDA(cudaGraphCreate(&g.graph, 0));
        cudaGraphNode_t deps[2];
        int ndep = 0;
        cudaMemsetParams mp{};
        mp.dst = ix->qnext;      // query counter
        mp.value = 0;
        mp.elementSize = 4;
        mp.width = 1;
        mp.height = 1;
        FL_CUDA(cudaGraphAddMemsetNode(&deps[ndep++], g.graph, nullptr, 0, &mp));
        if (srp) {
            mp.dst = ix->stats;
            mp.width = 2 * kStats;   // 64-bit counters
            FL_CUDA(cudaGraphAddMemsetNode(&deps[ndep++], g.graph, nullptr, 0, &mp));
        }
        FL_CUDA(cudaGraphAddKernelNode(&g.node, g.graph, deps, ndep, &kp));
        FL_CUDA(cudaGraphInstantiate(&g.exec, g.graph, 0));
        g.fn = P.fn;
        g.smem = P.smem;
        g.grid = P.grid;
    } else {
        FL_CUDA(cudaGraphExecKernelNodeSetParams(g.exec, g.node, &kp));
    }
    FL_CUDA(cudaGraphLaunch(g.exec, ix->stream));
    count_launch();
    return FLINNG_OK;
}

void destroy_graphs(flinng_index *ix)
{
    for (QueryGraph &g : ix->graphs) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        if (g.graph) cudaGraphDestroy(g.graph);
        g = QueryGraph{};
    }
}

int counts_launch(flinng_index *ix, const uint32_t *qbuckets, uint32_t nq,
                  uint16_t *out_counts)
{
    if (nq == 0) return FLINNG_OK;
    QArgs a = make_args(ix, qbuckets, nq);
    a.cap = kQTmax;          // the heavy-table list takes the buffer's last 2 kQTmax words
    a.kp = 2;
    a.out_counts = out_counts;
    const size_t smem = qsmem_bytes(a.cap, a.kp, a.BR, a.lcap, kQTmax, a.L, int(ix->cw));
    const void *fn = ix->cw == 1 ? counts_kernel_c1() : counts_kernel_c2();
    FL_TRY(ensure_dyn_smem(fn, smem));
    void *args[] = {&a};
    FL_CUDA(cudaLaunchKernel(fn, dim3(nq), dim3(kQTmax), args, smem, ix->stream));
    count_launch();
    return FLINNG_OK;
}

const void *plain_kernel_c1(int NT, uint32_t rw, uint32_t sm_threads)
{
    return plain_kernel_t<1>(NT, rw, sm_threads);
}
const void *fused_kernel_c1(int NT, uint32_t rw, bool srp, uint32_t sm_threads)
{
    return fused_kernel_t<1>(NT, rw, srp, sm_threads);
}
const void *counts_kernel_c1() { return (const void *)k_counts<1>; }

}  // namespace flinng
