// Batched query: collision counts, group tests, AND-over-R decode and top-k
// (Sec. 5, Alg. 2 and Alg. 3). One CTA of 128 to 1,024 threads per query.
//
// Alg. 3 walks cells by count (descending, ties by cell id) and emits a point
// when the last of its R cells is reached. That order is the ascending order
// of the key (-score, lastcell, id) with score = the least count among the
// point's R cells and lastcell = the largest cell id among those cells with
// that count; points with score < t_min are never emitted. The kernel
// computes the k smallest keys without the per-point counter array:
//
//  1. counts: cnt[c] += 1 for every cell c in the query's list of each table,
//     in shared memory: bytes when L <= 255, 16-bit words up to L = 4095
//     (count width CW). Tables are taken NT at a time; their lists are
//     flattened over the whole CTA.
//  2. group tests at decreasing thresholds: the cells of repetition 0 are
//     bucketed by count, the highest levels first and only as many cells as
//     the level list holds; level t holds those with count exactly t.
//  3. decode: walk levels t = L, L-1, ..., t_min. A point of score >= t has
//     all R cells at count >= t, in particular its repetition-0 cell, so after
//     level t every point with score >= t has been seen. The members of a
//     level's cells are flattened over the CTA, eight per lane: one 16-byte
//     load of their repetition-1 group ids drops every member whose
//     repetition-1 cell is below the admission bound's score, and only the
//     rest read their full record and get a key from all R group ids (the AND
//     over R). Stop once >= k points of score >= t were seen: no unseen point
//     can precede them.
//  4. top-k: candidates go to one shared buffer. After each group of levels, or
//     when the buffer would overflow, at most 128 of them are ranked against each
//     other, the k best are kept and the k-th key becomes the admission bound. Of
//     more candidates a histogram of their scores gives the k-th best score as
//     the bound; when many share it a radix select over the rest of the keys
//     keeps exactly the k best. At the end the best k are ranked.
//
// The kernels are templates on the count width; query.cu instantiates CW = 1
// and query_c16.cu CW = 2, each in its own translation unit.
#pragma once
#include "doph.cuh"
#include "internal.cuh"

namespace flinng {

constexpr int kQTmax = 256;              // CTA size of the counts kernel
constexpr uint32_t kLevelCells = 2048;   // repetition-0 cells placed at a time, by level
// Compactions of at most this many keys rank them directly, n^2 comparisons and no
// passes over a histogram. With 256 batches of 300 to 1,200 paid for it (60,000
// reads, R3 B300 L256, 900 queries of k = 100: 104.7 us against 85.4); batches of
// up to 150 with 128 to 256 candidates gained 2 us by it (14.6 against 16.6). Of 956
// sizes 128 is 2 % faster in the mean; 64 gave less than 128.
constexpr uint32_t kRankKeys = 128;

// key = (score_max - score) << 48 | lastcell << 32 | id
template <int CW> struct CountWidth;
template <> struct CountWidth<1> {
    static constexpr uint32_t kScoreMax = 255;
    static constexpr uint64_t kKeyBits = (1ull << 56) - 1;
};
template <> struct CountWidth<2> {
    static constexpr uint32_t kScoreMax = 4095;
    static constexpr uint64_t kKeyBits = (1ull << 60) - 1;
};

// cells per chunk of the walk, tables per round of the gather
template <int NT> constexpr uint32_t kChunkCells = 2 * NT;
constexpr uint32_t kWarpQueue = 64;      // filtered members a warp holds back (2 NT words in all)

struct QArgs {
    const uint32_t *qb;
    const uint16_t *cnt_in;   // per-cell counts given by the caller (nq x BR), or null: gather them
    uint32_t nq;
    const uint32_t *k;
    uint32_t k_max;
    const uint32_t *off;
    const uint16_t *cells;
    const uint32_t *moff;
    const uint32_t *mrec;     // repetition-0 member records (RW words each)
    const uint16_t *mg1;      // repetition-1 group ids in the same order (16-byte aligned, padded)
    const uint32_t *hidx;     // per slot: heavy bitmap index or kEmpty32
    const uint32_t *hbm;      // heavy slots' cell bitmaps, BRw words each
    uint32_t L, W, R, B, BR, BRw, t_min;
    uint32_t heavy_min; // a slot is heavy (has a cell bitmap) iff its list holds >= heavy_min cells
    uint32_t gcells;   // cells in the decode's first level group (at least 1); later groups double
    uint32_t gmax;     // up to this many
    uint32_t lcap;     // cells the level list holds
    uint32_t wide;     // 1: cells are large enough for the walk's filter (eight members per lane)
    uint32_t id_bits;  // bits of a point id
    uint32_t avg_cell; // members per repetition-0 cell, rounded up
    uint32_t cap;      // candidate buffer entries (power of two)
    uint32_t kp;       // final sort width: power of two >= k_max
    uint32_t *out_ids;
    uint16_t *out_scores;
    const uint32_t *out_row;  // per query: its row of the outputs, or null (row = query index)
    uint16_t *out_counts;
};

struct QSmem {
    uint64_t *buf;       // cap candidate keys
    uint64_t *keep;      // kp keys (selection output, final sort)
    uint32_t *u;         // 8 scalars: nbuf, nkeep, digit / k-th score, rank / found, whole / count,
                         // heavy tables (gather) / cells of a big level (decode), bound (u[6..7])
    uint32_t *lvl_n;     // nlev: repetition-0 cells per count, then cells at levels >= v
    uint32_t *shist;     // nlev: candidates in buf per score (score_hist)
    uint32_t *rhist;     // 256: radix histogram
    uint32_t *c_pre;     // kChunkCells + 4: exclusive prefix of unit counts, closed by ~0
    uint32_t *c_ms;      // kChunkCells: first member of each cell of a chunk; in the gather, first
                         // cell of each of 2 NT tables' lists
    uint32_t *lvl_cur;   // nlev: placement cursors of the level list (in c_pre and c_ms, which hold
                         // nothing while cells are placed)
    uint32_t *g_hl;      // 2 NT: bitmap indices of the heavy tables of a chunk of tables (the last
                         // words of buf: the gather runs before any candidate is kept)
    uint32_t *wsum;      // NT / 32: block-scan scratch
    uint32_t *q_m;       // kWarpQueue per warp: members that passed the filter; in the gather, the
                         // lengths of the 2 NT tables' lists
    uint16_t *q_c;       // their cells
    uint32_t *cntw;      // count words: 4 byte counts (CW = 1) or 2 16-bit counts (CW = 2) each
    uint16_t *lvl_cells; // lcap
};

// count levels 0..L, rounded up to a multiple of 4
__host__ __device__ inline uint32_t q_nlev(uint32_t L) { return (L + 4) & ~3u; }
// counter words, for whole 32-cell bitmap words
__host__ __device__ inline uint32_t q_count_words(uint32_t BR, int cw) { return (BR + 31) / 32 * (cw == 1 ? 8 : 16); }

__host__ __device__ inline size_t qsmem_bytes(uint32_t cap, uint32_t kp, uint32_t BR, uint32_t lcap, int NT,
                                              uint32_t L, int cw)
{
    const uint32_t ch = 2 * NT, chunk = 2 * ch + 4;      // kChunkCells; c_pre and c_ms
    size_t b = size_t(cap) * 8 + size_t(kp) * 8 + 8 * 4 + 2 * size_t(q_nlev(L)) * 4 + 256 * 4 +
               size_t(chunk > q_nlev(L) ? chunk : q_nlev(L)) * 4 + (NT / 32) * 4 + size_t(NT / 32) * kWarpQueue * 6;
    b = (b + 15) & ~size_t(15);
    b += size_t(q_count_words(BR, cw)) * 4 + size_t(lcap) * 2;
    return (b + 15) & ~size_t(15);
}

template <int NT, int CW>
__device__ inline QSmem carve_q(unsigned char *sm, uint32_t cap, uint32_t kp, uint32_t BR, uint32_t L)
{
    QSmem s;
    const uint32_t nlev = q_nlev(L);
    s.buf = (uint64_t *)sm;
    s.keep = s.buf + cap;
    s.u = (uint32_t *)(s.keep + kp);
    s.lvl_n = s.u + 8;
    s.shist = s.lvl_n + nlev;
    s.rhist = s.shist + nlev;
    s.c_pre = s.rhist + 256;
    s.c_ms = s.c_pre + kChunkCells<NT> + 4;
    s.lvl_cur = s.c_pre;
    s.g_hl = reinterpret_cast<uint32_t *>(s.buf + cap) - 2 * NT;   // needs cap >= NT
    s.wsum = s.c_pre + (2 * kChunkCells<NT> + 4 > nlev ? 2 * kChunkCells<NT> + 4 : nlev);
    s.q_m = s.wsum + NT / 32;
    s.q_c = reinterpret_cast<uint16_t *>(s.q_m + NT / 32 * kWarpQueue);
    size_t o = (size_t)((unsigned char *)(s.q_c + NT / 32 * kWarpQueue) - sm);
    o = (o + 15) & ~size_t(15);
    s.cntw = (uint32_t *)(sm + o);
    s.lvl_cells = (uint16_t *)(s.cntw + q_count_words(BR, CW));
    return s;
}

template <int CW>
__device__ __forceinline__ uint32_t cnt_at(const QSmem &s, uint32_t c)
{
    if constexpr (CW == 1) return reinterpret_cast<const uint8_t *>(s.cntw)[c];
    else return reinterpret_cast<const uint16_t *>(s.cntw)[c];
}

namespace {

// Member record of repetition 0: word 0 = point id, words 1.. = the group
// ids of repetitions 1..R-1, two 16-bit ids per word.
template <int RW>
__device__ inline void load_record(const uint32_t *__restrict__ rec, uint32_t m, uint32_t w[RW])
{
    if constexpr (RW == 1) {
        w[0] = __ldg(rec + m);
    } else if constexpr (RW == 2) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(rec) + m);
        w[0] = v.x; w[1] = v.y;
    } else if constexpr (RW == 4) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(rec) + m);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(rec) + 2 * size_t(m));
        const uint4 u = __ldg(reinterpret_cast<const uint4 *>(rec) + 2 * size_t(m) + 1);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
        w[4] = u.x; w[5] = u.y; w[6] = u.z; w[7] = u.w;
    }
}

// Exclusive block scan of one value per thread; returns the prefix and
// writes the total to *total (all threads). Contains __syncthreads.
template <int NT>
__device__ uint32_t block_excl_scan(uint32_t v, uint32_t *wsum, uint32_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) {
        const uint32_t t = wsum[w];
        before += (w < warp) ? t : 0u;
        all += t;
    }
    __syncthreads();
    *total = all;
    return before + x - v;
}

// Largest i in [lo, n) with pre[i] <= j (pre ascending, pre[lo] <= j).
__device__ inline uint32_t find_seg(const uint32_t *pre, uint32_t n, uint32_t j, uint32_t lo = 0)
{
    uint32_t hi = n;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (pre[mid] <= j) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Radix select over keys[0..n), given the kk-th key's score: exactly kk keys
// satisfy (key & mask) <= prefix on return (keys are unique, kk <= n). above:
// keys of a better score. Only the 48 bits below the score are searched.
template <int NT, int CW>
__device__ void block_select(const uint64_t *keys, uint32_t n, uint32_t kk, uint32_t score, uint32_t above,
                             uint32_t id_bits, const QSmem &s, uint64_t &prefix_out, uint64_t &mask_out)
{
    const int tid = threadIdx.x, lane = tid & 31;
    uint64_t prefix = uint64_t(CountWidth<CW>::kScoreMax - score) << 48, mask = ~0ull << 48;
    uint32_t rem = kk - above;
    for (int i = tid; i < 256; i += NT) s.rhist[i] = 0u;
    __syncthreads();
    for (int shift = 40; shift >= 0; shift -= 8) {
        if (shift < 32 && uint32_t(shift) >= id_bits) {     // all zeros
            mask |= uint64_t(0xFF) << shift;
            continue;
        }
        // keys share their leading digits: aggregate per warp before the
        // shared-memory atomic (one per distinct digit per warp)
        for (uint32_t ib = tid & ~31u; ib < n; ib += NT) {
            const uint32_t i = ib + lane;
            bool in = false;
            uint32_t dg = 256;
            if (i < n) {
                const uint64_t v = keys[i];
                in = (v & mask) == prefix;
                dg = in ? uint32_t((v >> shift) & 0xFF) : 256u;
            }
            const uint32_t grp = __match_any_sync(0xffffffffu, dg);
            if (in && lane == __ffs(grp) - 1) atomicAdd(&s.rhist[dg], __popc(grp));
        }
        __syncthreads();
        if (tid < 32) {
            uint32_t h[8], sum = 0;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                h[j] = s.rhist[lane * 8 + j];
                s.rhist[lane * 8 + j] = 0u;       // for the next digit
                sum += h[j];
            }
            uint32_t incl = sum;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            uint32_t run = incl - sum;
            if (run < rem && rem <= incl) {       // exactly one lane holds the digit
                uint32_t d = 0, hd = 0;
                bool found = false;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    if (!found) {
                        if (run + h[j] >= rem) {
                            d = lane * 8 + j;
                            hd = h[j];
                            found = true;
                        } else {
                            run += h[j];
                        }
                    }
                }
                s.u[2] = d;
                s.u[3] = rem - run;               // rank inside the digit's bucket
                s.u[4] = (hd == rem - run) ? 1u : 0u;   // the bucket is taken whole
            }
        }
        __syncthreads();
        const uint32_t d = s.u[2];
        rem = s.u[3];
        const bool whole = s.u[4] != 0;           // written again only after the next digit's barrier
        prefix |= uint64_t(d) << shift;
        mask |= uint64_t(0xFF) << shift;
        if (whole) break;
    }
    __syncthreads();
    prefix_out = prefix;
    mask_out = mask;
}

// Candidates of buf[0..n) per score, of scores in [lo, hi] (the others are not
// counted). Contains __syncthreads.
template <int NT, int CW>
__device__ void score_hist(const QSmem &s, uint32_t n, uint32_t lo, uint32_t hi)
{
    constexpr uint32_t kScoreMax = CountWidth<CW>::kScoreMax;
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t v = lo + threadIdx.x; v <= hi; v += NT) s.shist[v] = 0u;
    __syncthreads();
    for (uint32_t ib = threadIdx.x & ~31u; ib < n; ib += NT) {
        const uint32_t i = ib + lane;
        const uint32_t score = i < n ? kScoreMax - uint32_t(s.buf[i] >> 48) : 0u;
        const bool in = i < n && score >= lo;
        const uint32_t any = __ballot_sync(0xffffffffu, in);
        if (!any) continue;
        // candidates mostly tie: one addition for those that share the first one's score
        const uint32_t lead = __ffs(any) - 1, first = __shfl_sync(0xffffffffu, score, lead);
        const uint32_t same = __ballot_sync(0xffffffffu, in && score == first);
        if (lane == lead) atomicAdd(&s.shist[first], __popc(same));
        else if (in && score != first) atomicAdd(&s.shist[score], 1u);
    }
    __syncthreads();
}

// The kk-th best candidate's score, from the score histogram (scores in [lo,
// hi]), by one warp; all threads get it. False if there are fewer than kk. *m
// receives the number of candidates of at least that score. Contains
// __syncthreads.
__device__ inline bool kth_score_of(const QSmem &s, uint32_t lo, uint32_t hi, uint32_t kk, uint32_t *score, uint32_t *m)
{
    if (threadIdx.x < 32) {
        const uint32_t lane = threadIdx.x, nl = hi - lo + 1, per = (nl + 31) / 32;
        uint32_t local = 0;
        for (uint32_t i = 0; i < per; ++i) {
            const uint32_t pos = lane * per + i;         // the pos-th level below hi
            if (pos < nl) local += s.shist[hi - pos];
        }
        uint32_t incl = local;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= uint32_t(d)) incl += y;
        }
        uint32_t run = incl - local;
        if (lane == 31) s.u[3] = incl >= kk ? 1u : 0u;
        if (run < kk && kk <= incl) {                    // at most one lane holds the level
            uint32_t pos = lane * per;
            for (;; ++pos) {
                run += s.shist[hi - pos];
                if (run >= kk) break;
            }
            s.u[2] = hi - pos;
            s.u[4] = run;
        }
    }
    __syncthreads();
    const bool found = s.u[3] != 0u;
    if (found) {
        *score = s.u[2];
        *m = s.u[4];
    }
    __syncthreads();
    return found;
}

// The nk lowest of list[0..n) to keep[0..nk) in order: the keys are distinct, so
// a key's rank is the number of smaller keys, counted by four lanes.
template <int NT>
__device__ __forceinline__ void rank_keys(const uint64_t *list, uint32_t n, uint32_t nk, uint64_t *keep)
{
    const uint32_t part = threadIdx.x & 3;
    for (uint32_t ib = 0; ib < n; ib += NT / 4) {          // uniform: whole warps shuffle
        const uint32_t i = ib + (threadIdx.x >> 2);
        const uint64_t x = i < n ? list[i] : 0ull;
        uint32_t r = 0;
        for (uint32_t j = part; j < n; j += 4) r += list[j] < x ? 1u : 0u;
        r += __shfl_xor_sync(0xffffffffu, r, 1);
        r += __shfl_xor_sync(0xffffffffu, r, 2);
        if (part == 0 && i < n && r < nk) keep[r] = x;
    }
}

// The kk best of buf[0..nbuf), at most kRankKeys of them, to keep[0..kk) in order;
// returns the kk-th. Contains __syncthreads.
template <int NT>
__device__ __forceinline__ uint64_t rank_keep(const QSmem &s, uint32_t nbuf, uint32_t kk)
{
    rank_keys<NT>(s.buf, nbuf, kk, s.keep);
    __syncthreads();
    return s.keep[kk - 1];
}

// buf[0..kk) = keep[0..kk). Contains __syncthreads.
template <int NT>
__device__ __forceinline__ void take_kept(const QSmem &s, uint32_t kk)
{
    for (uint32_t i = threadIdx.x; i < kk; i += NT) s.buf[i] = s.keep[i];
    if (threadIdx.x == 0) s.u[0] = kk;
    __syncthreads();
}

// Keep the kk best of buf[0..nbuf) in buf[0..kk); score: the kk-th best's, m:
// candidates of at least it (kth_score_of, whose histogram is read). Returns
// the new admission bound: the largest kept key (later keys above it can never
// enter the top kk).
template <int NT, int CW>
__device__ uint64_t block_compact(const QArgs &a, const QSmem &s, uint32_t nbuf, uint32_t kk, uint32_t score, uint32_t m)
{
    const int lane = threadIdx.x & 31;
    const uint32_t above = m - s.shist[score];
    uint64_t prefix, mask;
    block_select<NT, CW>(s.buf, nbuf, kk, score, above, a.id_bits, s, prefix, mask);
    if (threadIdx.x == 0) s.u[1] = 0u;
    __syncthreads();
    for (uint32_t ib = threadIdx.x & ~31u; ib < nbuf; ib += NT) {
        const uint32_t i = ib + lane;
        const uint64_t v = i < nbuf ? s.buf[i] : kKeyNone;
        const bool take = i < nbuf && (v & mask) <= prefix;
        const uint32_t wm = __ballot_sync(0xffffffffu, take);
        if (wm) {
            uint32_t base = 0;
            if (lane == __ffs(wm) - 1) base = atomicAdd(&s.u[1], __popc(wm));
            base = __shfl_sync(0xffffffffu, base, __ffs(wm) - 1);
            if (take) s.keep[base + __popc(wm & ((1u << lane) - 1u))] = v;
        }
    }
    __syncthreads();
    uint64_t mx = 0;
    for (uint32_t i = threadIdx.x; i < kk; i += NT) {
        const uint64_t v = s.keep[i];
        s.buf[i] = v;
        mx = v > mx ? v : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t y = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = y > mx ? y : mx;
    }
    // u[6..7]: one 64-bit word (8-byte aligned: u follows the 64-bit keep array)
    if (threadIdx.x == 0) {
        s.u[0] = kk;
        s.u[6] = 0u;
        s.u[7] = 0u;
    }
    __syncthreads();
    if (lane == 0 && mx) {
        atomicMax(reinterpret_cast<unsigned long long *>(&s.u[6]), (unsigned long long)mx);
    }
    __syncthreads();
    const uint64_t bound = *reinterpret_cast<const unsigned long long *>(&s.u[6]);
    __syncthreads();
    return bound;
}

// Carry-save adder on 32 bit lanes: a + b + c = sum + 2 carry in every lane.
__device__ __forceinline__ void csa(uint32_t &carry, uint32_t &sum, uint32_t a, uint32_t b, uint32_t c)
{
    const uint32_t u = a ^ b;
    sum = u ^ c;
    carry = (a & b) | (u & c);
}

// Rows of an 8 x 32 bit matrix to its columns as bytes: pl[p] holds bit p of 32
// cells' counts, out[j] the counts of cells 4j .. 4j+3 as packed bytes. Three
// butterfly stages transpose each 8 x 8 block (byte j of row r then holds cell
// 8j + r), two 4 x 4 byte transposes put the cells in order: about 80
// operations, against 240 for spreading every plane's bits by multiplication.
__device__ __forceinline__ void planes_to_bytes(uint32_t (&pl)[8], uint32_t (&out)[8])
{
    constexpr uint32_t kMask[3] = {0x55555555u, 0x33333333u, 0x0F0F0F0Fu};
#pragma unroll
    for (int st = 0; st < 3; ++st) {
        const int d = 1 << st;
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            if (p & d) continue;
            const uint32_t t = ((pl[p] >> d) ^ pl[p + d]) & kMask[st];
            pl[p + d] ^= t;
            pl[p] ^= t << d;
        }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {              // rows 4h .. 4h + 3: cells 8j + 4h ..
        const uint32_t x0 = __byte_perm(pl[4 * h], pl[4 * h + 1], 0x5140);
        const uint32_t x1 = __byte_perm(pl[4 * h], pl[4 * h + 1], 0x7362);
        const uint32_t y0 = __byte_perm(pl[4 * h + 2], pl[4 * h + 3], 0x5140);
        const uint32_t y1 = __byte_perm(pl[4 * h + 2], pl[4 * h + 3], 0x7362);
        out[0 + h] = __byte_perm(x0, y0, 0x5410);
        out[2 + h] = __byte_perm(x0, y0, 0x7632);
        out[4 + h] = __byte_perm(x1, y1, 0x5410);
        out[6 + h] = __byte_perm(x1, y1, 0x7632);
    }
}

// Per-cell collision counts of one query (Sec. 5), up to 2 NT tables at a time (a
// thread's two offset pairs are in flight together).
// Tables whose bucket is heavy contribute their cell bitmap: each thread owns
// one bitmap word position (32 cells) and sums it over the heavy tables in
// bit-sliced form, then adds the sums to its counter words without atomics. The
// other tables' lists are flattened over the CTA in units of eight aligned
// cells, one 16-byte load per lane, and counted with shared-memory atomics: a
// list of the usual few dozen cells costs a few loads in flight together, not
// a chain of 2-byte loads with a search per cell. Expects s.u[5] == 0 (the
// heavy table count, zeroed with the query state) and leaves it 0. Contains
// __syncthreads.
template <int NT, int CW>
__device__ void gather_counts(const QArgs &a, const QSmem &s, const uint32_t *qb)
{
    const int tid = threadIdx.x;
    constexpr uint32_t kTab = 2 * NT;
    for (uint32_t l0 = 0; l0 < a.L; l0 += kTab) {
        // one table per thread while that covers them (32 tables on 16 threads
        // took 600 cycles more than on 32)
        const uint32_t nl = min(kTab, a.L - l0), tpt = nl <= uint32_t(NT) ? 1u : 2u;
        uint32_t o0[2] = {0u, 0u}, o1[2] = {0u, 0u}, units[2];
        uint64_t slot[2];
#pragma unroll
        for (uint32_t i = 0; i < 2; ++i) {
            const uint32_t l = l0 + tid * tpt + i;
            if (i < tpt && l < a.L) {
                slot[i] = (uint64_t(l) << a.W) | qb[l];
                o0[i] = a.off[slot[i]];
                o1[i] = a.off[slot[i] + 1];
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            // the list's length decides whether the slot is heavy, so the
            // bitmap index (another random DRAM access) is read for heavy
            // slots only
            if (o1[i] - o0[i] >= a.heavy_min) {
                s.g_hl[atomicAdd(&s.u[5], 1u)] = a.hidx[slot[i]];
                o1[i] = o0[i];
            }
            units[i] = o1[i] > o0[i] ? ((o1[i] - 1) >> 3) - (o0[i] >> 3) + 1 : 0u;
        }
        if (tid == 0) s.c_pre[NT * tpt] = ~0u;   // ends every forward search of c_pre
        uint32_t total;
        const uint32_t pre = block_excl_scan<NT>(units[0] + units[1], s.wsum, &total);
#pragma unroll
        for (uint32_t i = 0; i < 2; ++i) {
            if (i >= tpt) break;
            s.c_pre[tid * tpt + i] = pre + (i ? units[0] : 0u);
            s.c_ms[tid * tpt + i] = o0[i];
            s.q_m[tid * tpt + i] = o1[i] - o0[i];
        }
        __syncthreads();
        const uint32_t nh = s.u[5];
        if (nh > 0) {
            constexpr uint32_t kSub = 248;                // tables per pass: counts below 256, 8 bit planes
            for (uint32_t w = tid; w < a.BRw; w += NT) {
                for (uint32_t i1 = 0; i1 < nh; i1 += kSub) {
                    const uint32_t i2 = min(nh, i1 + kSub);
                    // bit-sliced counters of the word's 32 cells: pl[p] holds bit p
                    // of every cell's count. Eight bitmap words at a time (loaded
                    // together) go through a carry-save adder tree into planes 0..2;
                    // the weight-8 carry ripples into the planes above.
                    uint32_t pl[8];
#pragma unroll
                    for (int p = 0; p < 8; ++p) pl[p] = 0u;
                    for (uint32_t i0 = i1; i0 < i2; i0 += 8) {
                        uint32_t x[8];
#pragma unroll
                        for (int v = 0; v < 8; ++v)
                            x[v] = i0 + v < i2 ? __ldg(a.hbm + size_t(s.g_hl[i0 + v]) * a.BRw + w) : 0u;
                        uint32_t t0, t1, f0, f1, e;
                        csa(t0, pl[0], pl[0], x[0], x[1]);
                        csa(t1, pl[0], pl[0], x[2], x[3]);
                        csa(f0, pl[1], pl[1], t0, t1);
                        csa(t0, pl[0], pl[0], x[4], x[5]);
                        csa(t1, pl[0], pl[0], x[6], x[7]);
                        csa(f1, pl[1], pl[1], t0, t1);
                        csa(e, pl[2], pl[2], f0, f1);
#pragma unroll
                        for (int p = 3; p < 8; ++p) {
                            const uint32_t c = pl[p] & e;
                            pl[p] ^= e;
                            e = c;
                        }
                    }
                    // back to packed counters; a pass adds at most 248 to a cell.
                    // cntw is padded to whole 32-cell words (q_count_words).
                    uint32_t by[8];
                    planes_to_bytes(pl, by);
                    if constexpr (CW == 1) {
                        uint4 *cw = reinterpret_cast<uint4 *>(s.cntw + w * 8);
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            uint4 v = cw[j];
                            v.x += by[4 * j];
                            v.y += by[4 * j + 1];
                            v.z += by[4 * j + 2];
                            v.w += by[4 * j + 3];
                            cw[j] = v;
                        }
                    } else {
                        uint4 *cw = reinterpret_cast<uint4 *>(s.cntw + w * 16);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            uint4 v = cw[j];
                            v.x += __byte_perm(by[2 * j], 0u, 0x4140);
                            v.y += __byte_perm(by[2 * j], 0u, 0x4342);
                            v.z += __byte_perm(by[2 * j + 1], 0u, 0x4140);
                            v.w += __byte_perm(by[2 * j + 1], 0u, 0x4342);
                            cw[j] = v;
                        }
                    }
                }
            }
            __syncthreads();
        }
        // each warp counts a contiguous slice of the flattened units, so a lane's
        // table index moves forward by a few tables per step (c_pre is total
        // past the last table and ~0 at the end, which ends the search)
        const uint32_t per = ((total + NT / 32 - 1) / (NT / 32) + 31) & ~31u;
        const uint32_t eb = min(uint32_t(tid >> 5) * per, total);
        const uint32_t ee = min(eb + per, total);
        uint32_t e = eb + (tid & 31);
        uint32_t t = e < ee ? find_seg(s.c_pre, nl, e) : 0u;
        for (; e < ee; e += 32) {
            for (int step = 0; s.c_pre[t + 1] <= e; ++step) {
                if (step == 4) {
                    t = find_seg(s.c_pre, nl, e, t + 1);
                    break;
                }
                ++t;
            }
            const uint32_t beg = s.c_ms[t], u = (beg >> 3) + (e - s.c_pre[t]), m0 = u << 3;
            const uint32_t lo = beg > m0 ? beg - m0 : 0u, hi = min(beg + s.q_m[t] - m0, 8u);
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(a.cells) + u);
            const uint32_t cv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (uint32_t i = 0; i < 8; ++i) {
                if (i < lo || i >= hi) continue;       // another list's cells, or past the array's end
                const uint32_t c = (cv[i / 2] >> (16 * (i & 1))) & 0xFFFFu;
                if constexpr (CW == 1) atomicAdd(&s.cntw[c >> 2], 1u << ((c & 3) * 8));
                else atomicAdd(&s.cntw[c >> 1], 1u << ((c & 1) * 16));
            }
        }
        // every thread read nh before the heavy section's barrier (or nh was 0)
        if (tid == 0) s.u[5] = 0u;
        __syncthreads();
    }
}

// Per-cell counts given by the caller (e.g. the sum of table shards' counts)
// packed into the shared counters; values above L (here the caller's total
// table count) are clamped to L. Contains __syncthreads.
template <int NT, int CW>
__device__ void load_counts(const QArgs &a, const QSmem &s, const uint16_t *cnt)
{
    constexpr uint32_t kPer = CW == 1 ? 4u : 2u;
    const uint32_t nwords = q_count_words(a.BR, CW);
    uint32_t done = 0;                       // counter words taken eight counts at a time
    if (a.BR % 8 == 0 && reinterpret_cast<uintptr_t>(cnt) % 16 == 0) {
        const uint32_t lim = a.L | (a.L << 16);
        for (uint32_t i = threadIdx.x; i < a.BR / 8; i += NT) {
            uint4 v = __ldg(reinterpret_cast<const uint4 *>(cnt) + i);
            v.x = __vminu2(v.x, lim);
            v.y = __vminu2(v.y, lim);
            v.z = __vminu2(v.z, lim);
            v.w = __vminu2(v.w, lim);
            if constexpr (CW == 2) {
                *reinterpret_cast<uint4 *>(s.cntw + i * 4) = v;
            } else {
                *reinterpret_cast<uint2 *>(s.cntw + i * 2) =
                    make_uint2(__byte_perm(v.x, v.y, 0x6420), __byte_perm(v.z, v.w, 0x6420));
            }
        }
        done = a.BR / kPer;
    }
    for (uint32_t i = done + threadIdx.x; i < nwords; i += NT) {
        uint32_t wv = 0;
#pragma unroll
        for (uint32_t j = 0; j < kPer; ++j) {
            const uint32_t c = i * kPer + j;
            const uint32_t v = c < a.BR ? min(uint32_t(cnt[c]), a.L) : 0u;
            wv |= v << (j * (CW == 1 ? 8u : 16u));
        }
        s.cntw[i] = wv;
    }
    __syncthreads();
}

template <int NT, int CW>
__device__ inline void zero_query_state(const QArgs &a, const QSmem &s)
{
    const int tid = threadIdx.x;
    const uint32_t nwords = q_count_words(a.BR, CW);
    for (uint32_t i = tid; i < nwords; i += NT) s.cntw[i] = 0u;
    const uint32_t nlev = q_nlev(a.L);
    for (uint32_t i = tid; i < nlev; i += NT) {
        s.lvl_n[i] = 0u;
    }
    if (tid < 8) s.u[tid] = 0u;
}

// Calls f(cell, count) for this thread's repetition-0 cells with count >= lo,
// a 32-bit counter word (four or two cells) per access.
template <int NT, int CW, class Fn>
__device__ __forceinline__ void for_level_cells(const QArgs &a, const QSmem &s, uint32_t lo, Fn f)
{
    constexpr uint32_t kPer = CW == 1 ? 4u : 2u, kBits = CW == 1 ? 8u : 16u;
    const uint32_t nw = (a.B + kPer - 1) / kPer;
    for (uint32_t w = threadIdx.x; w < nw; w += NT) {
        const uint32_t x = s.cntw[w];
        if (x == 0u) continue;                 // lo >= 1
#pragma unroll
        for (uint32_t j = 0; j < kPer; ++j) {
            const uint32_t v = (x >> (j * kBits)) & ((1u << kBits) - 1u), b = w * kPer + j;
            if (v >= lo && b < a.B) f(b, v);   // the last word may hold cells of repetition 1
        }
    }
}

// Score of an admission bound: lower scores cannot enter (0 for kKeyBits).
template <int CW>
__device__ __forceinline__ uint32_t bound_score(uint64_t bound)
{
    return CountWidth<CW>::kScoreMax - uint32_t(bound >> 48);
}

// Room for n candidates in the buffer, for a warp (uniform): the first place, or
// ~0 where the buffer is too full. There are no reservations: a warp reads the
// fill first and appends at most 32 keys while it is at or below hwm. Once the
// fill passes hwm every warp appends at most once more, so hwm = cap - (NT + 32)
// cannot overflow.
__device__ __forceinline__ uint32_t append_at(const QSmem &s, uint32_t n, uint32_t hwm)
{
    uint32_t at = kEmpty32;
    if ((threadIdx.x & 31) == 0 && *reinterpret_cast<volatile uint32_t *>(&s.u[0]) <= hwm) at = atomicAdd(&s.u[0], n);
    return __shfl_sync(0xffffffffu, at, 0);
}

// Key of the member with record w in repetition-0 cell `cell`; kKeyNone if its
// score is below smin. No branches: the walk's lanes stay together.
template <int RW, int CW>
__device__ __forceinline__ uint64_t member_key(const QArgs &a, const QSmem &s, const uint32_t (&w)[RW], uint32_t cell,
                                               uint32_t smin)
{
    uint32_t score = cnt_at<CW>(s, cell), last = cell;       // repetition 0: the cell itself, at its level
#pragma unroll
    for (int r = 1; r < 2 * RW - 1; ++r) {
        if (r >= int(a.R)) break;
        const uint32_t g = (w[1 + (r - 1) / 2] >> (16 * ((r - 1) & 1))) & 0xFFFFu;
        const uint32_t c = uint32_t(r) * a.B + g;
        const uint32_t v = cnt_at<CW>(s, c);
        last = v <= score ? c : last;
        score = min(score, v);
    }
    const uint64_t key = (uint64_t(CountWidth<CW>::kScoreMax - score) << 48) | (uint64_t(last) << 32) | w[0];
    return score >= smin ? key : kKeyNone;
}

// The walk's end: true if every warp reached its slice's end; else (a warp paused
// at the buffer's mark) the block compacts and the warps resume.
template <int NT, int CW>
__device__ __forceinline__ bool walk_done(const QArgs &a, const QSmem &s, uint32_t kq, uint32_t hwm, uint32_t smin,
                                          uint32_t hi_level, uint64_t &bound)
{
    __syncthreads();
    const uint32_t nb0 = s.u[0];   // same value in every thread (read after the barrier)
    if (nb0 <= hwm) return true;
    if (nb0 <= kRankKeys) {
        bound = rank_keep<NT>(s, nb0, kq);              // hwm >= kq: there are kq
        take_kept<NT>(s, kq);
    } else {
        uint32_t score, n;
        score_hist<NT, CW>(s, nb0, smin, hi_level);
        kth_score_of(s, smin, hi_level, kq, &score, &n);
        bound = block_compact<NT, CW>(a, s, nb0, kq, score, n);
    }
    return false;
}

// The members of a chunk's cells (c_pre, c_ms; ncc cells whose ids are
// cell_of[0..ncc), M members in all), decoded into candidate keys, every record
// read: U members per lane and step, their loads in flight together. Each warp
// walks its own contiguous slice, so its cell index only moves forward.
template <int NT, int RW, int CW, int U>
__device__ void walk_all(const QArgs &a, const QSmem &s, const uint16_t *cell_of, uint32_t M, uint32_t ncc, uint32_t kq,
                         uint32_t hi_level, uint64_t &bound)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t per = ((M + NT / 32 - 1) / (NT / 32) + 31) & ~31u;
    uint32_t jb = min(uint32_t(tid >> 5) * per, M);   // this warp's cursor (warp-uniform)
    const uint32_t je = min(jb + per, M);
    // the cell holding member jb (warp-uniform; the largest such index is never an empty cell)
    uint32_t cur = jb < je ? find_seg(s.c_pre, ncc, jb) : 0u;
    const uint32_t hwm = a.cap - uint32_t(NT + 32);
    for (;;) {
        const uint32_t smin = max(a.t_min, bound_score<CW>(bound));
        while (jb < je) {
            // lanes to cells: one warp-uniform pass over the cell boundaries
            // inside this step; c_pre is M past the chunk's last cell and ~0 at
            // the array's end, so the pass stops at the step's last member
            const uint32_t last_j = min(jb + 32u * U, je) - 1u;
            uint32_t my[U];
#pragma unroll
            for (int u = 0; u < U; ++u) my[u] = cur;
            uint32_t k = cur + 1, bnd = s.c_pre[k];
            while (bnd <= last_j) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (jb + uint32_t(u) * 32 + lane >= bnd) my[u] = k;
                bnd = s.c_pre[++k];
            }
            uint32_t w[U][RW], cell[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint32_t j = jb + uint32_t(u) * 32 + lane;
                cell[u] = 0;
#pragma unroll
                for (int i = 0; i < RW; ++i) w[u][i] = 0u;
                if (j < je) {
                    cell[u] = cell_of[my[u]];
                    load_record<RW>(a.mrec, s.c_ms[my[u]] + (j - s.c_pre[my[u]]), w[u]);
                }
            }
            // the keys are made again for the few that are wanted, rather than held
            // (one member per lane, in flight: 125 us with the key held, 110 so)
            const uint32_t below = (1u << lane) - 1u;
            uint32_t wm[U], total = 0;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const uint64_t key = member_key<RW, CW>(a, s, w[u], cell[u], smin);
                wm[u] = __ballot_sync(0xffffffffu, jb + uint32_t(u) * 32 + lane < je && key <= bound);
                total += __popc(wm[u]);
            }
            int did = U;
            if (total) {
                // in one go where they are at most 32
                uint32_t at = total <= 32u ? append_at(s, total, hwm) : 0u;
                if (at == kEmpty32) did = 0;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (u >= did || !wm[u]) continue;
                    if (total > 32u) at = append_at(s, __popc(wm[u]), hwm);
                    if (at == kEmpty32) {
                        did = u;
                        continue;
                    }
                    if ((wm[u] >> lane) & 1u)
                        s.buf[at + __popc(wm[u] & below)] = member_key<RW, CW>(a, s, w[u], cell[u], smin);
                    at += __popc(wm[u]);
                }
            }
            if (did < U) {                     // paused: the step's rest after the compaction
                jb += 32u * did;
                if (did && jb < je) cur = find_seg(s.c_pre, ncc, jb);
                break;
            }
            jb += 32 * U;
            cur = k - 1;                       // the cell holding member last_j
        }
        if (walk_done<NT, CW>(a, s, kq, hwm, smin, hi_level, bound)) return;
    }
}

// The same through the repetition-1 groups: a unit is eight consecutive members,
// aligned. A lane reads the repetition-1 groups of its unit's members with one
// 16-byte load and drops those whose repetition-1 cell is below the admission
// bound; of the thousands of members a query walks almost all go there, at 2
// bytes and about five instructions each instead of a record of 8 to 32 bytes
// and a key. Those that pass are queued and decoded 32 at a time. M: units.
template <int NT, int RW, int CW>
__device__ void walk_filtered(const QArgs &a, const QSmem &s, const uint16_t *cell_of, uint32_t M, uint32_t ncc,
                              uint32_t kq, uint32_t hi_level, uint64_t &bound)
{
    const int tid = threadIdx.x, lane = tid & 31;
    // Few units are still spread over all warps, since each warp's chain of
    // loads is what a small chunk waits for.
    const uint32_t per = ((M + NT / 32 - 1) / (NT / 32) + 7) & ~7u;
    uint32_t jb = min(uint32_t(tid >> 5) * per, M);
    const uint32_t je = min(jb + per, M);
    uint32_t cur = jb < je ? find_seg(s.c_pre, ncc, jb) : 0u;
    const uint32_t hwm = a.cap - uint32_t(NT + 32);
    uint32_t *qm = s.q_m + (tid >> 5) * kWarpQueue;
    uint16_t *qc = s.q_c + (tid >> 5) * kWarpQueue;
    uint32_t qn = 0;                             // queued members (warp-uniform)
    uint32_t pend = 0u, m0 = 0u, my_cell = 0u;   // this lane's members m0 + bit still to queue
    for (;;) {
        const uint32_t smin = max(a.t_min, bound_score<CW>(bound));
        for (;;) {
            const bool more = __any_sync(0xffffffffu, pend != 0u);
            if (!more && qn < 32u && jb < je) {
                const uint32_t last_j = min(jb + 32u, je) - 1u, j = jb + lane;
                uint32_t my = cur, k = cur + 1, bnd = s.c_pre[k];
                while (bnd <= last_j) {
                    if (j >= bnd) my = k;
                    bnd = s.c_pre[++k];
                }
                cur = k - 1;   // the cell holding unit last_j
                jb += 32;
                if (j < je) {
                    const uint32_t ms = s.c_ms[my];
                    const uint32_t u = (ms >> 3) + (j - s.c_pre[my]);
                    my_cell = cell_of[my];
                    m0 = u << 3;
                    // members of neighbouring cells and the zeroed padding share
                    // the unit: valid group ids, masked out
                    const uint32_t me = __ldg(a.moff + my_cell + 1);
                    const uint4 g = __ldg(reinterpret_cast<const uint4 *>(a.mg1) + u);
                    const uint32_t lo = ms > m0 ? ms - m0 : 0u, hi = min(me - m0, 8u);
                    pend = ((1u << hi) - 1u) & ~((1u << lo) - 1u);
                    const uint32_t gw[4] = {g.x, g.y, g.z, g.w};
                    uint32_t ok = 0u;
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        ok |= (cnt_at<CW>(s, a.B + ((gw[i / 2] >> (16 * (i & 1))) & 0xFFFFu)) >= smin ? 1u : 0u) << i;
                    pend &= ok;
                }
            }
            if (qn < 32u && __any_sync(0xffffffffu, pend != 0u)) {
                // the members that passed go to the queue, as many as fit; the
                // others wait in pend, so that 32 are always decoded together
                const uint32_t np = __popc(pend);
                uint32_t x = np;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
                    if (lane >= d) x += y;
                }
                uint32_t at = qn + x - np;
                for (; pend && at < kWarpQueue; pend &= pend - 1u, ++at) {
                    qm[at] = m0 + __ffs(pend) - 1;
                    qc[at] = uint16_t(my_cell);
                }
                qn = min(qn + __shfl_sync(0xffffffffu, x, 31), kWarpQueue);
                __syncwarp();
                continue;
            }
            if (qn < 32u && jb < je) continue;      // nothing passed: the next step
            if (qn == 0u) break;
            // the queue's last members, one per lane
            const uint32_t qb = qn > 32u ? qn - 32u : 0u;
            const bool has = qb + lane < qn;
            uint32_t w[RW], cell = 0;
#pragma unroll
            for (int i = 0; i < RW; ++i) w[i] = 0u;
            if (has) {
                cell = qc[qb + lane];
                load_record<RW>(a.mrec, qm[qb + lane], w);
            }
            const uint64_t key = member_key<RW, CW>(a, s, w, cell, smin);
            const bool want = has && key <= bound;
            const uint32_t wm = __ballot_sync(0xffffffffu, want);
            if (wm) {
                const uint32_t at = append_at(s, __popc(wm), hwm);
                if (at == kEmpty32) break;
                if (want) s.buf[at + __popc(wm & ((1u << lane) - 1u))] = key;
            }
            qn = qb;
            __syncwarp();              // entries read before they are written again
        }
        if (walk_done<NT, CW>(a, s, kq, hwm, smin, hi_level, bound)) return;
    }
}

// Group tests, AND-over-R decode and top-k of query q, from the counts in
// shared memory; writes row q of the outputs.
template <int NT, int RW, int CW, int U>
__device__ void decode_topk(const QArgs &a, const QSmem &s, uint32_t q, uint32_t kq)
{
    constexpr uint32_t kScoreMax = CountWidth<CW>::kScoreMax;
    const int tid = threadIdx.x, lane = tid & 31;
    bool in_order = false;               // keep holds the kq best, in order
    uint32_t kth_score = 0, kth_n = 0;   // score of the kq-th best at the last check, candidates of at least it
    if (kq > 0) {
        // group tests of repetition 0: cells per count level
        for_level_cells<NT, CW>(a, s, a.t_min, [&](uint32_t, uint32_t v) { atomicAdd(&s.lvl_n[v], 1u); });
        __syncthreads();
        // lvl_n[v] becomes the number of cells at levels >= v, lvl_cur[v] those at
        // levels above v: thread i takes the i-th run of consecutive levels from L
        // down to t_min
        {
            const uint32_t nl = a.L - a.t_min + 1, per = (nl + NT - 1) / NT;
            uint32_t local = 0;
            for (uint32_t i = 0; i < per; ++i) {
                const uint32_t pos = uint32_t(tid) * per + i;
                if (pos < nl) local += s.lvl_n[a.L - pos];
            }
            uint32_t total, run = block_excl_scan<NT>(local, s.wsum, &total);
            for (uint32_t i = 0; i < per; ++i) {
                const uint32_t pos = uint32_t(tid) * per + i;
                if (pos < nl) {
                    s.lvl_cur[a.L - pos] = run;
                    run += s.lvl_n[a.L - pos];
                    s.lvl_n[a.L - pos] = run;
                }
            }
        }
        __syncthreads();
        // decode, level by level. After level t every point of score >= t has
        // been seen (its repetition-0 cell has count >= t), so the walk stops
        // once the kq-th best candidate scores >= t: no later point can enter.
        uint64_t bound = CountWidth<CW>::kKeyBits;   // admission: key <= bound
        // Levels are placed in the level list a segment at a time: as many whole
        // levels, from t down, as the list holds (most queries stop within the
        // first segment, so the list need not hold all B cells and the lower
        // levels are never placed). A single level larger than the list is
        // placed a range of lcap cell ids at a time. Within a segment levels are
        // taken in groups of whole levels, at most glim cells: small at first,
        // to get a bound early, then doubling. lvl_n[v] (cells at levels >= v) is
        // non-increasing in v, so both extents are binary searches, not walks
        // over the (mostly empty) levels.
        const uint32_t all = s.lvl_n[a.t_min];
        // lowest level in [lo, hi] with at most lim cells at or above it (hi if none)
        auto extent = [&](int lo, int hi, uint32_t lim) {
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (s.lvl_n[mid] <= lim) hi = mid;
                else lo = mid + 1;
            }
            return lo;
        };
        int t = int(a.L);
        // the highest level with a cell, where the levels are many
        if (a.L > 64u && s.lvl_n[t] == 0u) t = extent(int(a.t_min), t, 0u) - 1;
        const uint32_t hi_level = uint32_t(t);                       // no point scores more
        int seg_lo = t + 1;
        uint32_t seg_base = 0, glim = a.gcells;
        // the first group is four times as large where k is large and an early bound
        // helps little: the filter drops most members without one, or the walk that
        // reads all records has several in flight and, with few tables, scores mostly
        // tie (60,000 reads in 128 tables, 600 queries, k = 100: 68 us with the small
        // group, 53 with the large one; 512 tables, two shards: 64 and 73; 2,000
        // embeddings in 64 tables, k = 10: 131 and 158)
        if (kq >= 32u && ((U > 1 && a.R > 1 && a.L < 256u) || (a.wide && all * 2u < a.B))) glim = min(glim * 4u, a.gmax);
        while (t >= int(a.t_min)) {
            const uint32_t above = t < int(a.L) ? s.lvl_n[t + 1] : 0u;   // cells at levels above t
            if (above == all) break;                                     // none left
            const bool big = s.lvl_n[t] - above > a.lcap;
            int t_end = t;
            if (!big) {
                if (t < seg_lo) {
                    seg_lo = all - above <= a.lcap ? int(a.t_min) : extent(int(a.t_min), t, above + a.lcap);
                    seg_base = above;
                    if (above) {                   // nothing walked yet: lvl_cur is there already, t < L otherwise
                        for (int v = seg_lo + tid; v <= t; v += NT) s.lvl_cur[v] = s.lvl_n[v + 1] - seg_base;
                        __syncthreads();
                    }
                    for_level_cells<NT, CW>(a, s, uint32_t(seg_lo), [&](uint32_t b, uint32_t v) {
                        if (v <= uint32_t(t)) s.lvl_cells[atomicAdd(&s.lvl_cur[v], 1u)] = uint16_t(b);
                    });
                    __syncthreads();
                }
                t_end = all - above <= glim ? seg_lo : extent(seg_lo, t, above + glim);
            }
            // a group's cells, in one part or, for a big level, in ranges of cell ids
            for (uint32_t b0 = 0; b0 < (big ? a.B : 1u); b0 += a.lcap) {
                uint32_t first = above - seg_base, nc = s.lvl_n[t_end] - above;
                if (big) {
                    // a cursor of its own (u[5], free here): the words of lvl_cur are
                    // those of c_pre, which is written below as soon as the count is
                    // read, its closing word ahead of a barrier
                    first = 0;
                    if (tid == 0) s.u[5] = 0u;
                    __syncthreads();
                    for (uint32_t b = b0 + tid; b < min(b0 + a.lcap, a.B); b += NT)
                        if (cnt_at<CW>(s, b) == uint32_t(t)) s.lvl_cells[atomicAdd(&s.u[5], 1u)] = uint16_t(b);
                    __syncthreads();
                    nc = s.u[5];
                    __syncthreads();        // read by all before the next range's zero
                }
                // the filter pays while fewer than half the members pass it (a quarter
                // where the other walk has two records in flight): about the share of
                // cells that reach the admission bound (any repetition's counts are
                // alike). 1,528 queries of 568,482 URL sets in 17 tables, whose scores
                // mostly tie, one record in flight: 378 us, 500 with the line at a
                // quarter. It has a second load in its chain, so a chunk that the other
                // walk reads in two steps goes there.
                const bool wide = a.wide && s.lvl_n[max(a.t_min, bound_score<CW>(bound))] * 2u * U < a.B &&
                                  min(nc, uint32_t(2 * NT)) * a.avg_cell > 2u * U * NT;
                // cells per thread: two where there are more than one for each, since cells
                // of a few members make small chunks
                const uint32_t per = nc <= uint32_t(NT) ? 1u : 2u;
                for (uint32_t c0 = 0; c0 < nc; c0 += 2 * NT) {
                    uint32_t ms[2], units[2];
#pragma unroll
                    for (uint32_t i = 0; i < 2; ++i) {
                        const uint32_t ci = c0 + tid * per + i;
                        ms[i] = units[i] = 0;
                        if (i < per && ci < nc) {
                            const uint32_t b = s.lvl_cells[first + ci];
                            // a member's score is at most its repetition-0 cell's level:
                            // members of cells below the bound's score cannot enter
                            if (cnt_at<CW>(s, b) >= bound_score<CW>(bound)) {
                                ms[i] = a.moff[b];
                                units[i] = a.moff[b + 1];
                            }
                        }
                    }
#pragma unroll
                    for (uint32_t i = 0; i < 2; ++i) {
                        const uint32_t me = units[i];
                        units[i] = me - ms[i];
                        if (wide && units[i]) units[i] = ((me - 1) >> 3) - (ms[i] >> 3) + 1;
                    }
                    if (tid == 0) s.c_pre[NT * per] = ~0u;   // ends every forward search of c_pre
                    uint32_t M;
                    const uint32_t pre = block_excl_scan<NT>(units[0] + units[1], s.wsum, &M);
                    s.c_pre[tid * per] = pre;
                    s.c_ms[tid * per] = ms[0];
                    if (per == 2) {
                        s.c_pre[tid * 2 + 1] = pre + units[0];
                        s.c_ms[tid * 2 + 1] = ms[1];
                    }
                    const uint32_t ncc = min(uint32_t(2 * NT), nc - c0);
                    __syncthreads();
                    const uint16_t *cell_of = s.lvl_cells + first + c0;
                    if (wide) walk_filtered<NT, RW, CW>(a, s, cell_of, M, ncc, kq, hi_level, bound);
                    else walk_all<NT, RW, CW, U>(a, s, cell_of, M, ncc, kq, hi_level, bound);
                }
            }
            // the buffer's fill is final after the walk's last barrier (no cells: as at
            // the last check); every level >= t_end is complete, so points of score >=
            // t_end are all seen
            const uint32_t nb = s.u[0];
            if (nb >= kq && nb <= kRankKeys) {
                bound = rank_keep<NT>(s, nb, kq);
                kth_score = bound_score<CW>(bound);
                if (kth_score >= uint32_t(t_end) || s.lvl_n[t_end] == all) {
                    in_order = true;
                    break;
                }
                if (nb != kq) take_kept<NT>(s, kq);
            } else if (nb >= kq) {
                const uint32_t lo = max(a.t_min, bound_score<CW>(bound));
                score_hist<NT, CW>(s, nb, lo, hi_level);
                kth_score_of(s, lo, hi_level, kq, &kth_score, &kth_n);
                if (kth_n > max(2 * kq, 64u)) {
                    // many candidates tie: bound by the kq-th key, not by its score
                    bound = block_compact<NT, CW>(a, s, nb, kq, kth_score, kth_n);
                } else if (kth_score > bound_score<CW>(bound)) {
                    bound = (uint64_t(kScoreMax - kth_score) << 48) | 0xFFFFFFFFFFFFull;
                }
                if (kth_score >= uint32_t(t_end)) break;
            }
            t = t_end - 1;
            glim = min(glim * 2, a.gmax);
        }
    }
    __syncthreads();
    // final top-k, in order
    uint32_t nbuf = s.u[0];
    const uint32_t nk = nbuf < kq ? nbuf : kq;
    uint64_t *list = s.buf;
    if (!in_order && nbuf > kq) {
        // the last check saw every candidate
        if (kth_n <= min(256u, uint32_t(NT))) {
            // those of at least the kq-th score are few more than kq: collected
            // in the chunk scratch, free now
            list = reinterpret_cast<uint64_t *>(s.c_pre);
            if (tid == 0) s.u[1] = 0u;
            __syncthreads();
            for (uint32_t ib = tid & ~31u; ib < nbuf; ib += NT) {
                const uint32_t i = ib + lane;
                const uint64_t v = i < nbuf ? s.buf[i] : kKeyNone;
                const bool take = i < nbuf && kScoreMax - uint32_t(v >> 48) >= kth_score;
                const uint32_t wm = __ballot_sync(0xffffffffu, take);
                if (wm) {
                    uint32_t base = 0;
                    if (lane == __ffs(wm) - 1) base = atomicAdd(&s.u[1], __popc(wm));
                    base = __shfl_sync(0xffffffffu, base, __ffs(wm) - 1);
                    if (take) list[base + __popc(wm & ((1u << lane) - 1u))] = v;
                }
            }
            __syncthreads();
            nbuf = kth_n;
        } else {
            block_compact<NT, CW>(a, s, nbuf, kq, kth_score, kth_n);
            nbuf = kq;
        }
    }
    if (in_order) {
    } else if (nbuf <= uint32_t(NT)) {
        rank_keys<NT>(list, nbuf, nk, s.keep);
        __syncthreads();
    } else {
        for (uint32_t i = tid; i < a.kp; i += NT) s.keep[i] = (i < nk) ? s.buf[i] : kKeyNone;
        __syncthreads();
        for (uint32_t k2 = 2; k2 <= a.kp; k2 <<= 1) {
            for (uint32_t j = k2 >> 1; j > 0; j >>= 1) {
                for (uint32_t i = tid; i < a.kp; i += NT) {
                    const uint32_t l = i ^ j;
                    if (l > i) {
                        const uint64_t x = s.keep[i], y = s.keep[l];
                        const bool up = (i & k2) == 0;
                        if ((x > y) == up) {
                            s.keep[i] = y;
                            s.keep[l] = x;
                        }
                    }
                }
                __syncthreads();
            }
        }
    }
    const size_t row = a.out_row ? size_t(a.out_row[q]) : size_t(q);
    for (uint32_t i = tid; i < a.k_max; i += NT) {
        const uint64_t key = (i < nk) ? s.keep[i] : kKeyNone;
        const bool ok = key != kKeyNone;
        a.out_ids[row * a.k_max + i] = ok ? uint32_t(key & 0xFFFFFFFFu) : 0xFFFFFFFFu;
        if (a.out_scores)
            a.out_scores[row * a.k_max + i] = ok ? uint16_t(kScoreMax - uint32_t(key >> 48)) : uint16_t(0);
    }
    __syncthreads();
}

// FT: threads per SM that its registers allow.
template <int NT, int RW, int CW, int FT>
__global__ void __launch_bounds__(NT, FT / NT)
k_query(QArgs a)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const QSmem s = carve_q<NT, CW>(sm, a.cap, a.kp, a.BR, a.L);
    for (uint32_t q = blockIdx.x; q < a.nq; q += gridDim.x) {
        uint32_t kq = a.k ? a.k[q] : a.k_max;
        if (kq > a.k_max) kq = a.k_max;
        zero_query_state<NT, CW>(a, s);
        __syncthreads();
        if (kq > 0) {
            if (a.cnt_in) load_counts<NT, CW>(a, s, a.cnt_in + size_t(q) * a.BR);
            else gather_counts<NT, CW>(a, s, a.qb + size_t(q) * a.L);
        }
        decode_topk<NT, RW, CW, FT == 1024 ? 2 : 1>(a, s, q, kq);
    }
}

// ---------------------------------------------------------------- fused form
//
// One launch for the whole batch: each CTA hashes its query in shared memory
// (DOPH over the query's set, or the L*K sign projections of its vector),
// then runs the same gather / decode / top-k. The grid is persistent: CTAs
// loop over queries. The hashing follows the same definitions as the hash
// kernels (hash.cu), the bucket results are identical.

struct HArgs {
    // Jaccard
    const uint64_t *q_off;
    const uint32_t *q_el;
    uint32_t nb, da, db;
    uint64_t seed;
    const uint64_t *ba;
    const uint64_t *bc;
    const uint16_t *draw;     // densification draws
    // cosine
    const float *x;
    uint64_t ldx;
    const float *w;
    uint32_t d;
    float gamma2, tiny;
    double gamma64;
    unsigned long long *stats;
    uint32_t *qnext;    // next query to hand out (zeroed before each launch), or null: one per CTA
    uint32_t K;
    size_t hash_off;    // byte offset of the hash region in shared memory (0: inside the
                        // candidate buffer, which is free until the decode)
};

// DOPH of query q into qb[0..L) (shared memory). Contains __syncthreads.
template <int NT>
__device__ void cta_doph(const QArgs &a, const HArgs &h, uint32_t q, uint32_t *qb, uint32_t *val)
{
    const int tid = threadIdx.x;
    const uint32_t nb = h.nb;
    uint32_t *occ = val + nb;
    for (uint32_t k = tid; k < nb; k += NT) val[k] = kEmpty32;
    for (uint32_t k = tid; k < (nb + 31) / 32; k += NT) occ[k] = 0u;
    __syncthreads();
    const uint64_t beg = h.q_off[q], end = h.q_off[q + 1];
    for (uint64_t t = beg + tid; t < end; t += NT) {
        const uint32_t pe = h.da * __ldg(h.q_el + t) + h.db;
        const uint32_t bin = __umulhi(pe, nb);
        atomicMin(&val[bin], pe);
        atomicOr(&occ[bin >> 5], 1u << (bin & 31));
    }
    __syncthreads();
    if (end > beg) {
        for (uint32_t k = tid; k < nb; k += NT)
            if (!((occ[k >> 5] >> (k & 31)) & 1u)) val[k] = val[doph_source(k, nb, h.seed, h.draw, occ)];
    }
    __syncthreads();
    for (uint32_t l = tid; l < a.L; l += NT) {
        uint64_t hh = h.bc[l];
        for (uint32_t j = 0; j < h.K; ++j) hh += h.ba[l * h.K + j] * uint64_t(val[l * h.K + j]);
        qb[l] = uint32_t(hh >> (64 - a.W));
    }
    __syncthreads();
}

// Exact sign of sum_t a_t b_t for fp32 inputs, by one warp: fixed-point
// digits of 32 bits from 2^-384 upward, summed over lanes in int64.
__device__ int warp_exact_sign(const float *xa, const float *wb, uint32_t d, int lane)
{
    constexpr int kLimbs = 24;
    long long acc[kLimbs + 2];
    for (int i = 0; i < kLimbs + 2; ++i) acc[i] = 0;
    for (uint32_t t = lane; t < d; t += 32) {
        const double v = double(xa[t]) * double(wb[t]);
        const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
        const int ex = int((bits >> 52) & 0x7FF);
        unsigned long long man = bits & ((1ull << 52) - 1);
        if (ex == 0 && man == 0) continue;
        int lsb;
        if (ex == 0) {
            lsb = 1 - 1075;
        } else {
            man |= 1ull << 52;
            lsb = ex - 1075;
        }
        const int pos = lsb + 384;
        const int qd = pos >> 5, r = pos & 31;
        const unsigned long long d0 = (man << r) & 0xffffffffull;
        const unsigned long long d1 = (r == 0 ? (man >> 32) : (man >> (32 - r))) & 0xffffffffull;
        const unsigned long long d2 = (r == 0) ? 0ull : (man >> (64 - r));
        const long long sg = (bits >> 63) ? -1 : 1;
        acc[qd] += sg * (long long)d0;
        acc[qd + 1] += sg * (long long)d1;
        acc[qd + 2] += sg * (long long)d2;
    }
    for (int i = 0; i < kLimbs + 2; ++i) {
        long long v = acc[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        acc[i] = v;
    }
    acc[kLimbs - 1] += acc[kLimbs] * 4294967296ll;
    for (int i = 0; i < kLimbs - 1; ++i) {
        const long long c = acc[i] >> 32;
        acc[i] -= c * 4294967296ll;
        acc[i + 1] += c;
    }
    if (acc[kLimbs - 1] != 0) return acc[kLimbs - 1] > 0 ? 1 : -1;
    for (int i = kLimbs - 2; i >= 0; --i)
        if (acc[i] != 0) return 1;
    return 0;
}

// SRP codes of query q into qb[0..L): one warp per projection, fp32 with a
// rigorous error bound, fp64 re-check, exact accumulator last. Contains
// __syncthreads.
template <int NT>
__device__ void cta_srp(const QArgs &a, const HArgs &h, uint32_t q, uint32_t *qb, float *xs)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float *xq = h.x + size_t(q) * h.ldx;
    for (uint32_t t = tid; t < h.d; t += NT) xs[t] = xq[t];
    for (uint32_t l = tid; l < a.L; l += NT) qb[l] = 0u;
    __syncthreads();
    const uint32_t P = a.L * h.K;
    for (uint32_t j = warp; j < P; j += (NT / 32)) {
        const float *wj = h.w + size_t(j) * h.d;
        float p = 0.f, sa = 0.f;
        for (uint32_t t = lane; t < h.d; t += 32) {
            const float wv = __ldg(wj + t), xv = xs[t];
            p = fmaf(wv, xv, p);
            sa = fmaf(fabsf(wv), fabsf(xv), sa);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            p += __shfl_xor_sync(0xffffffffu, p, o);
            sa += __shfl_xor_sync(0xffffffffu, sa, o);
        }
        p = __shfl_sync(0xffffffffu, p, 0);
        sa = __shfl_sync(0xffffffffu, sa, 0);
        bool positive;
        if (fabsf(p) > fmaf(h.gamma2, sa, h.tiny)) {
            positive = p > 0.f;
        } else {
            double p64 = 0.0, s64 = 0.0;
            for (uint32_t t = lane; t < h.d; t += 32) {
                const double prod = double(wj[t]) * double(xs[t]);
                p64 += prod;
                s64 += fabs(prod);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                p64 += __shfl_xor_sync(0xffffffffu, p64, o);
                s64 += __shfl_xor_sync(0xffffffffu, s64, o);
            }
            p64 = __shfl_sync(0xffffffffu, p64, 0);
            s64 = __shfl_sync(0xffffffffu, s64, 0);
            if (fabs(p64) > h.gamma64 * s64) {
                positive = p64 > 0.0;
            } else {
                positive = warp_exact_sign(xs, wj, h.d, lane) > 0;
                if (lane == 0) atomicAdd(&h.stats[1], 1ull);
            }
            if (lane == 0) {
                atomicAdd(&h.stats[0], 1ull);
                atomicAdd(&h.stats[2], 1ull);
                if (positive != (p > 0.f)) atomicAdd(&h.stats[4], 1ull);
            }
        }
        if (lane == 0 && positive) atomicOr(&qb[j / h.K], 1u << (j % h.K));
    }
    __syncthreads();
}

// Bound by latency and instruction issue, not by DRAM: at the recall-target
// genomic shape a query's 8,000 cycles of hashing, 20,000 of gathering and
// 60,000 of decoding are chains of dependent L2 and DRAM loads and barriers, which
// four to eight resident CTAs per SM overlap (32 registers a thread; with 16-bit
// counts also 64, where shared memory admits no more than 1,024 threads anyway). Default launch shapes, same
// box, before the walk's filter, the gather's 16-byte units and the score
// histogram, and after: 1,000 genomic queries 197 -> 121 us, 10^4 URL queries
// 2.66 -> 1.54 ms, the plain form's 10^4 embedding queries 2.95 -> 1.49 ms.
template <int NT, int RW, int HASH, int CW, int FT>
__global__ void __launch_bounds__(NT, FT / NT)
k_query_fused(QArgs a, HArgs h)
{
    extern __shared__ __align__(16) unsigned char sm[];
    const QSmem s = carve_q<NT, CW>(sm, a.cap, a.kp, a.BR, a.L);
    uint32_t *qb = reinterpret_cast<uint32_t *>(sm + h.hash_off);
    uint32_t *qslot = qb + ((a.L + 3) & ~3u);
    uint32_t *hs = qslot + 4;
    // queries are handed out one at a time from a counter (zeroed before the
    // launch), so CTAs that drew cheap queries take more of them
    for (uint32_t q = blockIdx.x;;) {
        if (h.qnext) {
            if (threadIdx.x == 0) qslot[0] = atomicAdd(h.qnext, 1u);
            __syncthreads();
            q = qslot[0];
        }
        if (q >= a.nq) break;
        uint32_t kq = a.k ? a.k[q] : a.k_max;
        if (kq > a.k_max) kq = a.k_max;
        zero_query_state<NT, CW>(a, s);
        if (kq > 0) {
            if constexpr (HASH == 1) cta_doph<NT>(a, h, q, qb, hs);
            else cta_srp<NT>(a, h, q, qb, reinterpret_cast<float *>(hs));
            gather_counts<NT, CW>(a, s, qb);
        } else {
            __syncthreads();
        }
        decode_topk<NT, RW, CW, HASH == 1 && FT == 1024 ? 2 : 1>(a, s, q, kq);
        if (!h.qnext) break;
    }
}

// Bound by the gather's latency and the counts written, 2 B*R bytes a query (256
// tables, 12,288 cells, 512 queries: 20.7 us with 2-byte stores; two shards'
// counts, their sum and the decode 67.6 us, 62.8 with eight counts per access).
template <int CW>
__global__ void __launch_bounds__(kQTmax, 2048 / kQTmax)
k_counts(QArgs a)
{
    constexpr int NT = kQTmax;
    extern __shared__ __align__(16) unsigned char sm[];
    const QSmem s = carve_q<NT, CW>(sm, a.cap, a.kp, a.BR, a.L);
    const int tid = threadIdx.x;
    const uint32_t nwords = q_count_words(a.BR, CW);
    for (uint32_t q = blockIdx.x; q < a.nq; q += gridDim.x) {
        for (uint32_t i = tid; i < nwords; i += NT) s.cntw[i] = 0u;
        if (tid < 8) s.u[tid] = 0u;
        __syncthreads();
        gather_counts<NT, CW>(a, s, a.qb + size_t(q) * a.L);
        uint16_t *out = a.out_counts + size_t(q) * a.BR;
        if (a.BR % 8 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0) {
            // eight counts per store
            for (uint32_t i = tid; i < a.BR / 8; i += NT) {
                uint4 v;
                if constexpr (CW == 2) {
                    v = *reinterpret_cast<const uint4 *>(s.cntw + i * 4);
                } else {
                    const uint2 b = *reinterpret_cast<const uint2 *>(s.cntw + i * 2);
                    v = make_uint4(__byte_perm(b.x, 0u, 0x4140), __byte_perm(b.x, 0u, 0x4342),
                                   __byte_perm(b.y, 0u, 0x4140), __byte_perm(b.y, 0u, 0x4342));
                }
                reinterpret_cast<uint4 *>(out)[i] = v;
            }
        } else {
            for (uint32_t c = tid; c < a.BR; c += NT) out[c] = uint16_t(cnt_at<CW>(s, c));
        }
        __syncthreads();
    }
}

// Kernel entry points of one count width, by CTA size and record width.
template <int CW>
const void *plain_kernel_t(int NT, uint32_t rw, uint32_t sm_threads)
{
#define FL_PLAIN(N, FT) \
    switch (rw) { \
    case 1: return (const void *)k_query<N, 1, CW, FT>; \
    case 2: return (const void *)k_query<N, 2, CW, FT>; \
    case 4: return (const void *)k_query<N, 4, CW, FT>; \
    default: return (const void *)k_query<N, 8, CW, FT>; \
    }
    if (NT == 1024) { FL_PLAIN(1024, 1024) }
    if (NT == 512) { FL_PLAIN(512, 1024) }
    if (sm_threads == 2048) { FL_PLAIN(256, 2048) }
    FL_PLAIN(256, 1024)
#undef FL_PLAIN
}

// sm_threads: the threads per SM that the kernel's registers allow: 1,024 (64
// registers) or 2,048 (32). The SRP hash needs the former; with 8-bit counts the
// latter is compiled alone.
template <int CW>
const void *fused_kernel_t(int NT, uint32_t rw, bool srp, uint32_t sm_threads)
{
#define FL_FUSED(N, H, FT) \
    switch (rw) { \
    case 1: return (const void *)k_query_fused<N, 1, H, CW, FT>; \
    case 2: return (const void *)k_query_fused<N, 2, H, CW, FT>; \
    case 4: return (const void *)k_query_fused<N, 4, H, CW, FT>; \
    default: return (const void *)k_query_fused<N, 8, H, CW, FT>; \
    }
#define FL_FUSED_N(H, FT) \
    if (NT == 128) { FL_FUSED(128, H, FT) } \
    if (NT == 512) { FL_FUSED(512, H, FT) } \
    FL_FUSED(256, H, FT)
    if (srp) { FL_FUSED_N(2, 1024) }
    if constexpr (CW == 2) {
        if (sm_threads == 1024) { FL_FUSED_N(1, 1024) }
    }
    FL_FUSED_N(1, 2048)
#undef FL_FUSED_N
#undef FL_FUSED
}

}  // namespace

// Per count width: the plain, fused and counts kernels (query.cu: CW = 1,
// query_c16.cu: CW = 2).
const void *plain_kernel_c1(int NT, uint32_t rw, uint32_t sm_threads);
const void *fused_kernel_c1(int NT, uint32_t rw, bool srp, uint32_t sm_threads);
const void *counts_kernel_c1();
const void *plain_kernel_c2(int NT, uint32_t rw, uint32_t sm_threads);
const void *fused_kernel_c2(int NT, uint32_t rw, bool srp, uint32_t sm_threads);
const void *counts_kernel_c2();

}  // namespace flinng
