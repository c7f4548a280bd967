// The reverse index of a build from scratch (Sec. 5), by partitioning.
//
// Every (point, table) entry of the batch puts the point's R cells into the
// list of slot (table, bucket); a list holds each cell once, sorted. The
// general path (build.cu) sorts by whole slots with global atomics and
// 2-byte scattered writes, and runs five passes over all L * 2^W slots. Here a
// table's entries are first partitioned by the top C bits of their bucket,
// 2^C partitions of about a thousand points, and everything else happens on
// one partition at a time in shared memory:
//
//  1. k_transpose: buckets n x L -> L x n, so that a table's entries are
//     contiguous.
//  2. k_part_count, a scan, k_part_scatter: the entries of each (table,
//     partition) in one run, packed as (low bucket bits, point id), reordered
//     in shared memory so that the writes are runs too.
//  3. k_part_fine, a CTA per partition: counts per bucket, the points' cells by
//     bucket in shared memory, each list sorted and deduplicated there (a
//     thread, a warp or the CTA per list, by its length), then the lists
//     written compactly to the build scratch, their offsets within the
//     partition to the offset array and the partition's total.
//  4. Partitions too large for shared memory (a bucket that many points
//     share): k_big_count, k_big_starts and k_big_scatter group the partition's
//     points by bucket in global memory, kBigChunk entries a CTA; k_big_lists (a
//     warp per list), k_big_hot (a CTA per list of more than kHotPoints points)
//     and k_big_wide (kBigChunk points a CTA, then k_big_wide_list) build each
//     list through a bitmap over the B*R cells, k_big_scan makes their offsets.
//     Chunks, because a single CTA on the half million points of one bucket is
//     what the others would wait for.
//  5. A scan of the partitions' totals, and k_part_finish: final offsets, the
//     heavy slots' list and bitmap rows, and the lists moved to their place.
//
// Bound by the passes over the entries and slots (about 12 bytes per entry and
// list cell, 8 per slot) and by the lists' sorts in shared memory. Measured,
// general path -> this one, whole build with hashing: recall-target genomic
// index (100,000 reads, 512 tables, 67 M slots, 154 M cells) 5.08 -> 1.88 ms, of
// which k_part_fine 0.87, k_part_finish 0.24, k_doph 0.20; URL index (10^6 sets,
// 64 tables, 136 M cells, buckets of up to half the points) 23.6 -> 3.3 ms, where
// the general path's warp per slot walked the hot buckets alone.
#include <algorithm>

#include "internal.cuh"
#include "trace.h"

namespace flinng {
namespace {

constexpr int kT = 256;                    // threads of the partition kernels
constexpr uint32_t kTile = 4096;           // entries per CTA of the count and scatter passes
constexpr uint32_t kPartPoints = 1024;     // points per partition aimed at
constexpr uint32_t kFinePoints = 1536;     // most points of a partition sorted in shared memory
constexpr uint32_t kMaxC = 11;             // coarse bits
constexpr uint32_t kMaxLow = 12;           // bucket bits within a partition
constexpr uint32_t kThreadList = 16;       // cells a single thread sorts
constexpr uint32_t kWarpList = 128;        // cells a warp sorts
constexpr uint32_t kHotPoints = 512;       // points of a list that one warp still handles
constexpr uint32_t kBigChunk = 8192;       // entries of a big partition, points of a wide list per CTA

// Exclusive prefix of v over the CTA of NT threads; total in *total.
template <int NT>
__device__ uint32_t excl_scan(uint32_t v, uint32_t *wsum, uint32_t *total)
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

// The R cells of a point from its row of group ids (RP of them, one load).
template <int RP>
__device__ __forceinline__ void point_cells(const uint16_t *__restrict__ gid, uint32_t id, uint32_t R, uint32_t B,
                                            uint32_t c[RP])
{
    uint32_t w[RP / 2];
    if constexpr (RP == 2) {
        w[0] = __ldg(reinterpret_cast<const uint32_t *>(gid) + id);
    } else if constexpr (RP == 4) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(gid) + id);
        w[0] = v.x;
        w[1] = v.y;
    } else {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(gid) + id);
        w[0] = v.x;
        w[1] = v.y;
        w[2] = v.z;
        w[3] = v.w;
    }
#pragma unroll
    for (int r = 0; r < RP; ++r) c[r] = uint32_t(r) * B + ((w[r / 2] >> (16 * (r & 1))) & 0xFFFFu);
    (void)R;
}

__global__ void __launch_bounds__(256) k_transpose(const uint32_t *__restrict__ in, uint64_t n, uint32_t L,
                                                   uint32_t *__restrict__ out)
{
    __shared__ uint32_t t[32][33];
    const uint32_t tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const uint64_t x0 = uint64_t(blockIdx.x) * 32;
    const uint32_t l0 = blockIdx.y * 32;
#pragma unroll
    for (uint32_t j = ty; j < 32; j += 8)
        if (x0 + j < n && l0 + tx < L) t[j][tx] = in[(x0 + j) * L + l0 + tx];
    __syncthreads();
#pragma unroll
    for (uint32_t j = ty; j < 32; j += 8)
        if (x0 + tx < n && l0 + j < L) out[uint64_t(l0 + j) * n + x0 + tx] = t[tx][j];
}

// Entries per (table, partition). Grid: tiles x tables.
__global__ void __launch_bounds__(kT) k_part_count(const uint32_t *__restrict__ bt, uint64_t n, uint32_t C,
                                                   uint32_t low, uint32_t *__restrict__ pcnt)
{
    extern __shared__ uint32_t hist[];
    const uint32_t np = 1u << C, l = blockIdx.y;
    for (uint32_t d = threadIdx.x; d < np; d += kT) hist[d] = 0u;
    __syncthreads();
    const uint64_t x0 = uint64_t(blockIdx.x) * kTile;
    const uint32_t m = uint32_t(n - x0 < kTile ? n - x0 : kTile);
    const uint32_t *col = bt + uint64_t(l) * n + x0;
    for (uint32_t i = threadIdx.x; i < m; i += kT) atomicAdd(&hist[col[i] >> low], 1u);
    __syncthreads();
    for (uint32_t d = threadIdx.x; d < np; d += kT)
        if (hist[d]) atomicAdd(&pcnt[(uint64_t(l) << C) + d], hist[d]);
}

// Entries moved to their partition: part[...] = low bucket bits << idbits | id.
// pcur starts as the partitions' bases; a tile takes its run of each with one
// atomic (the order of the runs does not matter: lists are sorted later).
__global__ void __launch_bounds__(kT) k_part_scatter(const uint32_t *__restrict__ bt, uint64_t n, uint32_t C,
                                                     uint32_t low, uint32_t idbits, uint32_t *__restrict__ pcur,
                                                     uint32_t *__restrict__ part)
{
    extern __shared__ uint32_t sm[];
    const uint32_t np = 1u << C, l = blockIdx.y, tid = threadIdx.x;
    uint32_t *start = sm, *gbase = start + np, *key = gbase + np, *wsum = key + kTile;
    uint16_t *dig = reinterpret_cast<uint16_t *>(wsum + kT / 32);
    for (uint32_t d = tid; d < np; d += kT) start[d] = 0u;
    __syncthreads();
    const uint64_t x0 = uint64_t(blockIdx.x) * kTile;
    const uint32_t m = uint32_t(n - x0 < kTile ? n - x0 : kTile);
    const uint32_t *col = bt + uint64_t(l) * n + x0;
    constexpr int kPer = kTile / kT;
    uint32_t b[kPer];
    uint16_t rk[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) b[i] = tid + i * kT < m ? col[tid + i * kT] : 0u;
#pragma unroll
    for (int i = 0; i < kPer; ++i)
        if (tid + i * kT < m) rk[i] = uint16_t(atomicAdd(&start[b[i] >> low], 1u));
    __syncthreads();
    const uint32_t per = (np + kT - 1) / kT;
    uint32_t sum = 0, total;
    for (uint32_t j = 0; j < per; ++j) {
        const uint32_t d = tid * per + j;
        if (d < np) {
            const uint32_t c = start[d];
            gbase[d] = c ? atomicAdd(&pcur[(uint64_t(l) << C) + d], c) : 0u;
            sum += c;
        }
    }
    uint32_t run = excl_scan<kT>(sum, wsum, &total);
    for (uint32_t j = 0; j < per; ++j) {
        const uint32_t d = tid * per + j;
        if (d < np) {
            const uint32_t c = start[d];
            start[d] = run;
            run += c;
        }
    }
    __syncthreads();
    const uint32_t lmask = (1u << low) - 1u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const uint32_t t = tid + i * kT;
        if (t >= m) continue;
        const uint32_t d = b[i] >> low, at = start[d] + rk[i];
        key[at] = ((b[i] & lmask) << idbits) | uint32_t(x0 + t);     // idbits + low <= 32
        dig[at] = uint16_t(d);
    }
    __syncthreads();
    for (uint32_t j = tid; j < m; j += kT) {
        const uint32_t d = dig[j];
        part[gbase[d] + (j - start[d])] = key[j];
    }
}

// Batcher's odd-even merge sort of N registers (N a power of two).
template <int N>
__device__ __forceinline__ void net_sort(uint32_t (&v)[N])
{
#pragma unroll
    for (int p = 1; p < N; p *= 2) {
#pragma unroll
        for (int k = p; k >= 1; k /= 2) {
#pragma unroll
            for (int j = 0; j < N; ++j) {
                // pairs (j, j + k) within one 2p block, taken from j = k mod p in steps of 2k
                const int j0 = k % p;
                if (j < j0 || ((j - j0) / k) % 2 != 0 || j + k >= N || j / (2 * p) != (j + k) / (2 * p)) continue;
                const uint32_t lo = min(v[j], v[j + k]);
                v[j + k] = max(v[j], v[j + k]);
                v[j] = lo;
            }
        }
    }
}

// A list of len <= N cells sorted and deduplicated in place by one thread.
template <int N>
__device__ __forceinline__ uint32_t thread_sort_unique(uint16_t *list, uint32_t len)
{
    uint32_t v[N];
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = uint32_t(i) < len ? uint32_t(list[i]) : 0xFFFFFFFFu;
    net_sort<N>(v);
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (v[i] != 0xFFFFFFFFu && (i == 0 || v[i] != v[i > 0 ? i - 1 : 0])) list[m++] = uint16_t(v[i]);
    return m;
}

// Exclusive prefix over the CTA of nb values, four consecutive ones per thread
// and round: get(b, v) reads values b .. b + 3 (nb of them or fewer), put(b, pre,
// v) receives their prefixes. With nb a power of two of at least four both move
// all four at once. Returns the total. Contains __syncthreads; a round is read
// before it is written.
template <class Get, class Put>
__device__ uint32_t scan_buckets(uint32_t nb, uint32_t *wsum, Get get, Put put)
{
    uint32_t base = 0;
    for (uint32_t b0 = 0; b0 < nb; b0 += 4 * kT) {
        const uint32_t b = b0 + threadIdx.x * 4;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (b < nb) v = get(b);
        uint32_t total;
        uint4 pre;
        pre.x = base + excl_scan<kT>(v.x + v.y + v.z + v.w, wsum, &total);
        pre.y = pre.x + v.x;
        pre.z = pre.y + v.y;
        pre.w = pre.z + v.z;
        if (b < nb) put(b, pre, v);
        base += total;
    }
    return base;
}

__device__ __forceinline__ uint2 pack16x4(const uint4 &v) { return make_uint2(v.x | v.y << 16, v.z | v.w << 16); }

// A list of len <= 32 K cells sorted by one warp in registers and
// deduplicated in place; returns the distinct cells.
template <int K>
__device__ uint32_t warp_sort_unique(uint16_t *list, uint32_t len)
{
    const int lane = threadIdx.x & 31;
    uint32_t v[K];
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = uint32_t(k * 32 + lane) < len ? uint32_t(list[k * 32 + lane]) : 0xFFFFFFFFu;
#pragma unroll
    for (int k2 = 2; k2 <= 32 * K; k2 <<= 1) {
#pragma unroll
        for (int j = k2 >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const int p = k ^ (j >> 5);
                    if (p > k) {
                        const bool up = ((k * 32) & k2) == 0;
                        const uint32_t lo = min(v[k], v[p]), hi = max(v[k], v[p]);
                        v[k] = up ? lo : hi;
                        v[p] = up ? hi : lo;
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k) {
                    const uint32_t o = __shfl_xor_sync(0xffffffffu, v[k], j);
                    const bool up = ((k * 32 + lane) & k2) == 0, lower = (lane & j) == 0;
                    v[k] = (lower == up) ? min(v[k], o) : max(v[k], o);
                }
            }
        }
    }
    uint32_t out = 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        uint32_t prev = __shfl_up_sync(0xffffffffu, v[k], 1);
        if (k > 0) {
            const uint32_t last = __shfl_sync(0xffffffffu, v[k > 0 ? k - 1 : 0], 31);
            if (lane == 0) prev = last;
        }
        const bool keep = v[k] != 0xFFFFFFFFu && ((k == 0 && lane == 0) || v[k] != prev);
        const uint32_t m = __ballot_sync(0xffffffffu, keep);
        if (keep) list[out + __popc(m & ((1u << lane) - 1u))] = uint16_t(v[k]);
        out += __popc(m);
    }
    __syncwarp();
    return out;
}

struct FineArgs {
    const uint32_t *part;
    const uint32_t *pbase;     // partitions + 1: first entry of each
    const uint16_t *gid;
    uint32_t R, B, BRw, low, idbits;
    uint32_t *noff;            // per slot: offset within its partition
    uint16_t *tmp;             // lists of partition p from pbase[p] R on
    uint32_t *ptot;            // per partition: its list cells
    uint32_t *big;             // partitions of more than kFinePoints points
    uint32_t *nbig;
    uint2 *chunks;             // their chunks {partition, first entry of the chunk within it}
    uint32_t *nchunks;
};

__host__ __device__ inline size_t fine_smem(uint32_t low, uint32_t R, uint32_t BRw)
{
    const size_t nb = size_t(1) << low;
    const size_t nb4 = nb < 4 ? 4 : nb;                // the scans move four buckets at a time
    return nb4 * 4 + (size_t(BRw) + 3) / 4 * 16 + 64 + size_t(kFinePoints) * R * 4 + (nb4 + 4) * 2 + nb4 * 2 +
           kFinePoints * 2;
}

// Bound by issue and shared-memory latency over the lists: per list of two or
// more points a sort, nothing per empty bucket but the vectorised scans and the
// offset written.
template <int RP>
__global__ void __launch_bounds__(kT) k_part_fine(FineArgs a)
{
    extern __shared__ __align__(16) unsigned char raw[];
    const uint32_t nb = 1u << a.low, nb4 = max(nb, 4u), tid = threadIdx.x, lane = tid & 31, R = a.R;
    // every array below starts at a multiple of 8 bytes (cnt of 16)
    uint32_t *cnt = reinterpret_cast<uint32_t *>(raw);            // nb4: cells per bucket, later list offsets
    uint32_t *bm = cnt + nb4;                                     // BRw
    uint32_t *wsum = bm + (a.BRw + 3) / 4 * 4;                    // 8
    uint32_t *nwl = wsum + 8;                                     // lists for threads, warps, the CTA; next warp list
    uint16_t *cells = reinterpret_cast<uint16_t *>(nwl + 4);      // kFinePoints R
    uint16_t *owner = cells + kFinePoints * R;                    // their buckets
    uint16_t *start = owner + kFinePoints * R;                    // nb4 + 1
    uint16_t *dlen = start + nb4 + 4;                             // nb4: distinct cells
    // worklists of buckets with two points or more: for threads from the front
    // and for warps from the back of the first half, for the CTA in the second
    uint16_t *wl = dlen + nb4, *wc = wl + kFinePoints / 2;
    const uint64_t p = blockIdx.x;
    const uint32_t e0 = a.pbase[p], E = a.pbase[p + 1] - e0;
    uint32_t *noff = a.noff + (p << a.low);
    if (E == 0) {
        for (uint32_t b = tid; b < nb; b += kT) noff[b] = 0u;
        if (tid == 0) a.ptot[p] = 0u;
        return;
    }
    if (E > kFinePoints) {
        for (uint32_t b = tid; b < nb; b += kT) noff[b] = 0u;      // k_big_count adds up here
        if (tid == 0) {
            a.big[atomicAdd(a.nbig, 1u)] = uint32_t(p);
            uint32_t at = atomicAdd(a.nchunks, (E + kBigChunk - 1) / kBigChunk);
            for (uint32_t t = 0; t < E; t += kBigChunk) a.chunks[at++] = make_uint2(uint32_t(p), t);
        }
        return;
    }
    constexpr int kPer = kFinePoints / kT;
    const uint32_t idmask = (1u << a.idbits) - 1u;                // idbits < 32 (R >= 2)
    uint32_t e[kPer];
    uint16_t rk[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) e[i] = tid + i * kT < E ? a.part[e0 + tid + i * kT] : 0u;
    for (uint32_t b = tid * 4; b < nb4; b += 4 * kT) *reinterpret_cast<uint4 *>(cnt + b) = make_uint4(0u, 0u, 0u, 0u);
    if (tid < 4) nwl[tid] = 0u;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i)
        if (tid + i * kT < E) rk[i] = uint16_t(atomicAdd(&cnt[e[i] >> a.idbits], R));
    __syncthreads();
    const uint32_t total = scan_buckets(
        nb4, wsum, [&](uint32_t b) { return *reinterpret_cast<const uint4 *>(cnt + b); },
        [&](uint32_t b, const uint4 &pre, const uint4 &v) {
            *reinterpret_cast<uint2 *>(start + b) = pack16x4(pre);
            *reinterpret_cast<uint2 *>(dlen + b) = pack16x4(v);
        });
    if (tid == 0) start[nb4] = uint16_t(total);           // start[nb .. nb4) are the total already
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        if (tid + i * kT >= E) continue;
        const uint32_t b = e[i] >> a.idbits, s0 = start[b], len = dlen[b], at = s0 + rk[i];
        uint32_t c[RP];
        point_cells<RP>(a.gid, e[i] & idmask, R, a.B, c);
#pragma unroll
        for (int r = 0; r < RP; ++r)
            if (r < int(R)) {
                cells[at + r] = uint16_t(c[r]);
                owner[at + r] = uint16_t(b);
            }
        // a bucket's first point lists it, unless it is the only one: its cells
        // ascend with the repetition
        if (rk[i] == 0 && len > R) {
            if (len <= kThreadList) wl[atomicAdd(&nwl[0], 1u)] = uint16_t(b);
            else if (len <= kWarpList) wl[kFinePoints / 2 - 1 - atomicAdd(&nwl[1], 1u)] = uint16_t(b);
            else wc[atomicAdd(&nwl[2], 1u)] = uint16_t(b);
        }
    }
    __syncthreads();
    // sorted, distinct lists in place
    const uint32_t nt = nwl[0], nw = nwl[1], nc = nwl[2];
    for (uint32_t i = tid; i < nt; i += kT) {
        const uint32_t b = wl[i], len = dlen[b];
        uint16_t *list = cells + start[b];
        dlen[b] = uint16_t(len <= 8 ? thread_sort_unique<8>(list, len) : thread_sort_unique<16>(list, len));
    }
    __syncwarp();
    for (;;) {
        uint32_t i = lane == 0 ? atomicAdd(&nwl[3], 1u) : 0u;
        i = __shfl_sync(0xffffffffu, i, 0);
        if (i >= nw) break;
        const uint32_t b = wl[kFinePoints / 2 - 1 - i], len = dlen[b];
        uint16_t *list = cells + start[b];
        const uint32_t m = len <= 32 ? warp_sort_unique<1>(list, len)
                           : len <= 64 ? warp_sort_unique<2>(list, len) : warp_sort_unique<4>(list, len);
        if (lane == 0) dlen[b] = uint16_t(m);
        __syncwarp();
    }
    for (uint32_t i = 0; i < nc; ++i) {                 // the CTA: through a bitmap over the cells
        const uint32_t b = wc[i], s0 = start[b], len = start[b + 1] - s0;
        for (uint32_t w = tid; w < a.BRw; w += kT) bm[w] = 0u;
        __syncthreads();
        for (uint32_t t = tid; t < len; t += kT) atomicOr(&bm[cells[s0 + t] >> 5], 1u << (cells[s0 + t] & 31));
        __syncthreads();
        const uint32_t wper = (a.BRw + kT - 1) / kT;
        uint32_t bits = 0, m;
        for (uint32_t j = 0; j < wper; ++j)
            if (tid * wper + j < a.BRw) bits += __popc(bm[tid * wper + j]);
        uint32_t at = s0 + excl_scan<kT>(bits, wsum, &m);
        for (uint32_t j = 0; j < wper; ++j) {
            const uint32_t w = tid * wper + j;
            if (w >= a.BRw) break;
            for (uint32_t x = bm[w]; x; x &= x - 1) cells[at++] = uint16_t(w * 32 + __ffs(x) - 1);
        }
        if (tid == 0) dlen[b] = uint16_t(m);
        __syncthreads();
    }
    __syncthreads();
    // offsets within the partition, then the lists behind one another
    const uint32_t kept = scan_buckets(
        nb4, wsum,
        [&](uint32_t b) {
            const uint2 v = *reinterpret_cast<const uint2 *>(dlen + b);
            return make_uint4(v.x & 0xFFFFu, v.x >> 16, v.y & 0xFFFFu, v.y >> 16);
        },
        [&](uint32_t b, const uint4 &pre, const uint4 &) {
            *reinterpret_cast<uint4 *>(cnt + b) = pre;
            if (nb >= 4) {
                *reinterpret_cast<uint4 *>(noff + b) = pre;
            } else {
                noff[0] = pre.x;
                if (nb > 1) noff[1] = pre.y;
            }
        });
    if (tid == 0) a.ptot[p] = kept;
    __syncthreads();
    uint16_t *out = a.tmp + uint64_t(e0) * R;
    for (uint32_t q = tid; q < total; q += kT) {
        const uint32_t b = owner[q], j = q - start[b];
        if (j < dlen[b]) out[cnt[b] + j] = cells[q];
    }
}

// Points per slot of the big partitions (added up in noff), a chunk per CTA.
__global__ void __launch_bounds__(kT) k_big_count(FineArgs a)
{
    extern __shared__ uint32_t cur[];                 // nb
    const uint32_t nb = 1u << a.low, tid = threadIdx.x, nch = *a.nchunks;
    for (uint32_t i = blockIdx.x; i < nch; i += gridDim.x) {
        const uint2 ch = a.chunks[i];
        const uint32_t e0 = a.pbase[ch.x] + ch.y, m = min(kBigChunk, a.pbase[ch.x + 1] - e0);
        for (uint32_t b = tid; b < nb; b += kT) cur[b] = 0u;
        __syncthreads();
        constexpr int kU = 8;                         // entries in flight per thread
        for (uint32_t t0 = tid; t0 < m; t0 += kT * kU) {
            uint32_t v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) v[u] = t0 + u * kT < m ? a.part[e0 + t0 + u * kT] : 0u;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (t0 + u * kT < m) atomicAdd(&cur[v[u] >> a.idbits], 1u);
        }
        __syncthreads();
        uint32_t *noff = a.noff + (uint64_t(ch.x) << a.low);
        for (uint32_t b = tid; b < nb; b += kT)
            if (cur[b]) atomicAdd(&noff[b], cur[b]);
        __syncthreads();
    }
}

struct BigLists {
    uint32_t *sstart;          // per slot of the big partitions: its first entry in part2
    uint32_t *scur;            // and its scatter cursor
    uint32_t *hot;             // slots of more than kHotPoints points
    uint2 *wide;               // of more than kBigChunk: {slot, points}
    uint2 *wchunk;             // chunks of the wide slots {wide index, first point}
    uint32_t *n;               // counts of hot, wide, wchunk
};

// First entry and cursor of every slot of a big partition; hot and wide slots
// listed.
__global__ void __launch_bounds__(kT) k_big_starts(FineArgs a, BigLists g)
{
    __shared__ uint32_t wsum[kT / 32];
    const uint32_t nb = 1u << a.low, tid = threadIdx.x, nbig = *a.nbig, per = (nb + kT - 1) / kT;
    for (uint32_t i = blockIdx.x; i < nbig; i += gridDim.x) {
        const uint64_t p = a.big[i], slot0 = p << a.low;
        uint32_t sum = 0, total;
        for (uint32_t j = 0; j < per; ++j)
            if (tid * per + j < nb) sum += a.noff[slot0 + tid * per + j];
        uint32_t run = a.pbase[p] + excl_scan<kT>(sum, wsum, &total);
        for (uint32_t j = 0; j < per; ++j) {
            const uint32_t b = tid * per + j;
            if (b >= nb) break;
            const uint32_t c = a.noff[slot0 + b];
            g.sstart[slot0 + b] = g.scur[slot0 + b] = run;
            if (c > kBigChunk) {
                const uint32_t w = atomicAdd(&g.n[1], 1u);
                g.wide[w] = make_uint2(uint32_t(slot0 + b), c);
                uint32_t at = atomicAdd(&g.n[2], (c + kBigChunk - 1) / kBigChunk);
                for (uint32_t t = 0; t < c; t += kBigChunk) g.wchunk[at++] = make_uint2(w, t);
            } else if (c > kHotPoints) {
                g.hot[atomicAdd(&g.n[0], 1u)] = uint32_t(slot0 + b);
            }
            run += c;
        }
    }
}

// The big partitions' points grouped by bucket in part2, a chunk per CTA: its
// run of each bucket reserved with one atomic, places within it drawn in shared
// memory, one atomic for the lanes of a bucket.
__global__ void __launch_bounds__(kT) k_big_scatter(FineArgs a, BigLists g, uint32_t *__restrict__ part2)
{
    extern __shared__ uint32_t cur[];                 // nb
    const uint32_t nb = 1u << a.low, tid = threadIdx.x, lane = tid & 31, nch = *a.nchunks;
    const uint32_t idmask = (1u << a.idbits) - 1u;
    for (uint32_t i = blockIdx.x; i < nch; i += gridDim.x) {
        const uint2 ch = a.chunks[i];
        const uint32_t e0 = a.pbase[ch.x] + ch.y, m = min(kBigChunk, a.pbase[ch.x + 1] - e0);
        for (uint32_t b = tid; b < nb; b += kT) cur[b] = 0u;
        __syncthreads();
        constexpr int kU = 8;
        for (uint32_t t0 = tid; t0 < m; t0 += kT * kU) {
            uint32_t v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) v[u] = t0 + u * kT < m ? a.part[e0 + t0 + u * kT] : 0u;
#pragma unroll
            for (int u = 0; u < kU; ++u)
                if (t0 + u * kT < m) atomicAdd(&cur[v[u] >> a.idbits], 1u);
        }
        __syncthreads();
        uint32_t *scur = g.scur + (uint64_t(ch.x) << a.low);
        for (uint32_t b = tid; b < nb; b += kT)
            if (cur[b]) cur[b] = atomicAdd(&scur[b], cur[b]);
        __syncthreads();
        for (uint32_t t0 = tid - lane; t0 < m; t0 += kT * kU) {
            uint32_t v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const uint32_t t = t0 + lane + u * kT;
                v[u] = t < m ? a.part[e0 + t] : 0u;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const bool in = t0 + lane + u * kT < m;
                const uint32_t b = in ? v[u] >> a.idbits : 0xFFFFFFFFu;
                const uint32_t same = __match_any_sync(0xffffffffu, b);
                const uint32_t lead = __ffs(same) - 1;
                uint32_t at = 0;
                if (in && lane == lead) at = atomicAdd(&cur[b], __popc(same));
                at = __shfl_sync(0xffffffffu, at, lead) + __popc(same & ((1u << lane) - 1u));
                if (in) part2[at] = v[u] & idmask;
            }
        }
        __syncthreads();
    }
}

// Cells of list words: the set bits of the bitmap bm (BRw words, one per lane
// at a time) written ascending at out; returns their number. One warp.
__device__ uint32_t warp_bitmap_list(const uint32_t *bm, uint32_t BRw, uint16_t *out)
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t written = 0;
    for (uint32_t w0 = 0; w0 < BRw; w0 += 32) {
        uint32_t bits = w0 + lane < BRw ? bm[w0 + lane] : 0u;
        const uint32_t c = __popc(bits);
        uint32_t incl = c;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= uint32_t(d)) incl += y;
        }
        uint32_t at = written + incl - c;
        for (; bits; bits &= bits - 1) out[at++] = uint16_t((w0 + lane) * 32 + __ffs(bits) - 1);
        written += __shfl_sync(0xffffffffu, incl, 31);
    }
    return written;
}

// A warp per slot of the big partitions (those of up to kHotPoints points):
// its list at tmp[sstart R], its length in noff.
template <int RP>
__global__ void __launch_bounds__(kT) k_big_lists(FineArgs a, const uint32_t *__restrict__ part2,
                                                  const uint32_t *__restrict__ sstart)
{
    extern __shared__ uint32_t bm_all[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, R = a.R;
    uint32_t *bm = bm_all + warp * a.BRw;
    const uint64_t items = uint64_t(*a.nbig) << a.low;
    for (uint64_t i = uint64_t(blockIdx.x) * (kT / 32) + warp; i < items; i += uint64_t(gridDim.x) * (kT / 32)) {
        const uint64_t slot = (uint64_t(a.big[i >> a.low]) << a.low) + (i & ((1u << a.low) - 1u));
        const uint32_t m = a.noff[slot];
        if (m == 0 || m > kHotPoints) continue;
        const uint32_t s0 = sstart[slot];
        uint16_t *out = a.tmp + uint64_t(s0) * R;
        if (m * R <= 32u) {                  // few cells: sorted in registers, no bitmap to clear and read
            if (lane < m) {
                uint32_t c[RP];
                point_cells<RP>(a.gid, part2[s0 + lane], R, a.B, c);
#pragma unroll
                for (int r = 0; r < RP; ++r)
                    if (r < int(R)) out[lane * R + r] = uint16_t(c[r]);
            }
            __syncwarp();
            const uint32_t len = warp_sort_unique<1>(out, m * R);
            if (lane == 0) a.noff[slot] = len;
            continue;
        }
        for (uint32_t w = lane; w < a.BRw; w += 32) bm[w] = 0u;
        __syncwarp();
        for (uint32_t t = lane; t < m; t += 32) {
            uint32_t c[RP];
            point_cells<RP>(a.gid, part2[s0 + t], R, a.B, c);
#pragma unroll
            for (int r = 0; r < RP; ++r)
                if (r < int(R)) atomicOr(&bm[c[r] >> 5], 1u << (c[r] & 31));
        }
        __syncwarp();
        const uint32_t len = warp_bitmap_list(bm, a.BRw, out);
        if (lane == 0) a.noff[slot] = len;
        __syncwarp();
    }
}

// The cells of points part2[s0 .. s0 + m) set in the CTA's bitmap bm.
template <int RP>
__device__ __forceinline__ void set_cells(const FineArgs &a, const uint32_t *__restrict__ part2, uint32_t s0, uint32_t m,
                                          uint32_t *bm)
{
    constexpr int kU = 4;                             // points in flight per thread
    for (uint32_t t0 = threadIdx.x; t0 < m; t0 += kT * kU) {
        uint32_t id[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) id[u] = t0 + u * kT < m ? part2[s0 + t0 + u * kT] : 0u;
        uint32_t c[kU][RP];
#pragma unroll
        for (int u = 0; u < kU; ++u) point_cells<RP>(a.gid, id[u], a.R, a.B, c[u]);
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            if (t0 + u * kT >= m) break;
#pragma unroll
            for (int r = 0; r < RP; ++r)
                if (r < int(a.R)) atomicOr(&bm[c[u][r] >> 5], 1u << (c[u][r] & 31));
        }
    }
}

// The set bits of a bitmap (BRw words) as an ascending list at out, by the CTA:
// prefixes per word (pre: BRw words of shared memory), then a warp per word, a
// lane per bit, so that a word's cells are one coalesced store. Returns their
// number. Contains __syncthreads.
__device__ __forceinline__ uint32_t cta_bitmap_list(const uint32_t *bm, uint32_t BRw, uint32_t *wsum, uint32_t *pre,
                                                    uint16_t *out)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31, per = (BRw + kT - 1) / kT;
    uint32_t bits = 0, len;
    for (uint32_t j = 0; j < per; ++j)
        if (tid * per + j < BRw) bits += __popc(bm[tid * per + j]);
    uint32_t at = excl_scan<kT>(bits, wsum, &len);
    for (uint32_t j = 0; j < per; ++j) {
        const uint32_t w = tid * per + j;
        if (w >= BRw) break;
        pre[w] = at;
        at += __popc(bm[w]);
    }
    __syncthreads();
    for (uint32_t w = tid >> 5; w < BRw; w += kT / 32) {
        const uint32_t x = bm[w];
        if ((x >> lane) & 1u) out[pre[w] + __popc(x & ((1u << lane) - 1u))] = uint16_t(w * 32 + lane);
    }
    return len;
}

// A CTA per hot slot; eight of them per SM overlap their chains of loads and
// barriers.
template <int RP>
__global__ void __launch_bounds__(kT)
k_big_hot(FineArgs a, const uint32_t *__restrict__ part2, BigLists g)
{
    extern __shared__ uint32_t bm[];                  // BRw, then as many prefixes
    __shared__ uint32_t wsum[kT / 32];
    const uint32_t nh = g.n[0];
    for (uint32_t i = blockIdx.x; i < nh; i += gridDim.x) {
        const uint32_t slot = g.hot[i], s0 = g.sstart[slot];
        for (uint32_t w = threadIdx.x; w < a.BRw; w += kT) bm[w] = 0u;
        __syncthreads();
        set_cells<RP>(a, part2, s0, a.noff[slot], bm);
        __syncthreads();
        const uint32_t len = cta_bitmap_list(bm, a.BRw, wsum, bm + a.BRw, a.tmp + uint64_t(s0) * a.R);
        if (threadIdx.x == 0) a.noff[slot] = len;
        __syncthreads();
    }
}

// A chunk of a wide slot per CTA: its cells OR'ed into the slot's row of wbm
// (zeroed).
template <int RP>
__global__ void __launch_bounds__(kT)
k_big_wide(FineArgs a, const uint32_t *__restrict__ part2, BigLists g, uint32_t *__restrict__ wbm)
{
    extern __shared__ uint32_t bm[];                  // BRw
    const uint32_t nch = g.n[2];
    for (uint32_t i = blockIdx.x; i < nch; i += gridDim.x) {
        const uint2 ch = g.wchunk[i], ws = g.wide[ch.x];
        for (uint32_t w = threadIdx.x; w < a.BRw; w += kT) bm[w] = 0u;
        __syncthreads();
        set_cells<RP>(a, part2, g.sstart[ws.x] + ch.y, min(kBigChunk, ws.y - ch.y), bm);
        __syncthreads();
        for (uint32_t w = threadIdx.x; w < a.BRw; w += kT)
            if (bm[w]) atomicOr(&wbm[uint64_t(ch.x) * a.BRw + w], bm[w]);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kT) k_big_wide_list(FineArgs a, BigLists g, const uint32_t *__restrict__ wbm)
{
    extern __shared__ uint32_t bm[];                  // BRw, then as many prefixes
    __shared__ uint32_t wsum[kT / 32];
    const uint32_t nw = g.n[1];
    for (uint32_t i = blockIdx.x; i < nw; i += gridDim.x) {
        const uint32_t slot = g.wide[i].x;
        for (uint32_t w = threadIdx.x; w < a.BRw; w += kT) bm[w] = wbm[uint64_t(i) * a.BRw + w];
        __syncthreads();
        const uint32_t len = cta_bitmap_list(bm, a.BRw, wsum, bm + a.BRw, a.tmp + uint64_t(g.sstart[slot]) * a.R);
        if (threadIdx.x == 0) a.noff[slot] = len;
        __syncthreads();
    }
}

// List lengths of a big partition's slots -> offsets within it, and its total.
__global__ void __launch_bounds__(kT) k_big_scan(FineArgs a)
{
    __shared__ uint32_t wsum[kT / 32];
    const uint32_t nb = 1u << a.low, tid = threadIdx.x, nbig = *a.nbig, per = (nb + kT - 1) / kT;
    for (uint32_t i = blockIdx.x; i < nbig; i += gridDim.x) {
        const uint64_t p = a.big[i];
        uint32_t *noff = a.noff + (p << a.low);
        uint32_t sum = 0, total;
        for (uint32_t j = 0; j < per; ++j)
            if (tid * per + j < nb) sum += noff[tid * per + j];
        uint32_t run = excl_scan<kT>(sum, wsum, &total);
        for (uint32_t j = 0; j < per; ++j) {
            const uint32_t b = tid * per + j;
            if (b >= nb) break;
            const uint32_t c = noff[b];
            noff[b] = run;
            run += c;
        }
        if (tid == 0) a.ptot[p] = total;
        __syncthreads();
    }
}

// n cells from src to dst (anywhere, not overlapping) by lanes t of nt: 16-byte
// stores at dst's alignment, each from two aligned 16-byte loads of src shifted
// by their distance. Reads up to 15 bytes past src's end (kCellPad).
template <int Q>
__device__ __forceinline__ uint4 shifted(const uint4 &x, const uint4 &y, bool half)
{
    const uint32_t w[9] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w, 0u};
    uint4 o;
    o.x = half ? __funnelshift_r(w[Q], w[Q + 1], 16) : w[Q];
    o.y = half ? __funnelshift_r(w[Q + 1], w[Q + 2], 16) : w[Q + 1];
    o.z = half ? __funnelshift_r(w[Q + 2], w[Q + 3], 16) : w[Q + 2];
    o.w = half ? __funnelshift_r(w[Q + 3], w[Q + 4], 16) : w[Q + 3];
    return o;
}

__device__ __forceinline__ void copy_cells(uint16_t *__restrict__ dst, const uint16_t *__restrict__ src, uint32_t n,
                                           uint32_t t, uint32_t nt)
{
    const uint32_t head = min(n, uint32_t((16u - (reinterpret_cast<uintptr_t>(dst) & 15u)) & 15u) / 2);
    const uint32_t body = (n - head) / 8, tail = head + body * 8;
    if (t < head) dst[t] = src[t];
    if (tail + t < n && t < 8) dst[tail + t] = src[tail + t];
    const uint32_t by = uint32_t(reinterpret_cast<uintptr_t>(src + head) & 15u);
    const uint4 *s4 = reinterpret_cast<const uint4 *>(reinterpret_cast<uintptr_t>(src + head) - by);
    uint4 *d4 = reinterpret_cast<uint4 *>(dst + head);
    const bool half = (by & 2u) != 0u;
    for (uint32_t i = t; i < body; i += nt) {
        const uint4 x = s4[i], y = by ? s4[i + 1] : x;
        switch (by >> 2) {                       // uniform over the copy
        case 0: d4[i] = shifted<0>(x, y, half); break;
        case 1: d4[i] = shifted<1>(x, y, half); break;
        case 2: d4[i] = shifted<2>(x, y, half); break;
        default: d4[i] = shifted<3>(x, y, half); break;
        }
    }
}

// A CTA per partition: its slots' final offsets and bitmap rows, its lists to
// their place. Bound by memory: 1.4 GB in 237 us at the recall-target index (385
// us with 2-byte copies).
__global__ void __launch_bounds__(kT) k_part_finish(FineArgs a, uint64_t nparts, const uint32_t *__restrict__ tbase,
                                                    const uint32_t *__restrict__ sstart, uint32_t heavy_min,
                                                    uint32_t *__restrict__ hidx, uint32_t *__restrict__ list,
                                                    uint32_t *__restrict__ nheavy, uint16_t *__restrict__ cells)
{
    const uint32_t nb = 1u << a.low, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t p = blockIdx.x;
    const uint32_t base = tbase[p], total = tbase[p + 1] - base;
    const uint32_t e0 = a.pbase[p], E = a.pbase[p + 1] - e0;
    const uint64_t slot0 = p << a.low;
    uint32_t *noff = a.noff + slot0;
    for (uint32_t b0 = 0; b0 < nb; b0 += 4 * kT) {
        const uint32_t b = b0 + tid * 4;
        uint32_t o[5] = {0u, 0u, 0u, 0u, 0u};
        if (b + 4 <= nb) {
            const uint4 v = *reinterpret_cast<const uint4 *>(noff + b);
            o[0] = v.x;
            o[1] = v.y;
            o[2] = v.z;
            o[3] = v.w;
            o[4] = b + 4 < nb ? noff[b + 4] : total;
        } else {
            for (uint32_t j = 0; j < 5; ++j) o[j] = b + j < nb ? noff[b + j] : total;
        }
        __syncthreads();                    // all offsets of this stretch read before any is rewritten
        uint32_t h[4];
#pragma unroll
        for (uint32_t j = 0; j < 4; ++j) {
            const bool heavy = b + j < nb && o[j + 1] - o[j] >= heavy_min;
            const uint32_t m = __ballot_sync(0xffffffffu, heavy);
            h[j] = kEmpty32;
            if (m) {
                uint32_t at = 0;
                const uint32_t lead = __ffs(m) - 1;
                if (lane == lead) at = atomicAdd(nheavy, __popc(m));
                at = __shfl_sync(0xffffffffu, at, lead) + __popc(m & ((1u << lane) - 1u));
                if (heavy) {
                    h[j] = at;
                    list[at] = uint32_t(slot0 + b + j);
                }
            }
        }
        if (b + 4 <= nb) {
            *reinterpret_cast<uint4 *>(noff + b) = make_uint4(base + o[0], base + o[1], base + o[2], base + o[3]);
            *reinterpret_cast<uint4 *>(hidx + slot0 + b) = make_uint4(h[0], h[1], h[2], h[3]);
        } else {
            for (uint32_t j = 0; j < 4; ++j)
                if (b + j < nb) {
                    noff[b + j] = base + o[j];
                    hidx[slot0 + b + j] = h[j];
                }
        }
    }
    if (p + 1 == nparts && tid == 0) noff[nb] = base + total;
    if (E <= kFinePoints) {
        copy_cells(cells + base, a.tmp + uint64_t(e0) * a.R, total, tid, kT);
    } else {
        __syncthreads();                    // the final offsets, read back by the warps
        for (uint32_t b = warp; b < nb; b += kT / 32) {
            const uint32_t o0 = noff[b], o1 = b + 1 < nb ? noff[b + 1] : base + total;
            if (o0 == o1) continue;
            copy_cells(cells + o0, a.tmp + uint64_t(sstart[slot0 + b]) * a.R, o1 - o0, lane, 32);
        }
    }
}

struct PartPlan {
    uint32_t C, low, idbits;
    uint64_t parts;
};

// Coarse bits: partitions of about kPartPoints points, so that nearly all fit
// kFinePoints and four to six CTAs an SM, and at most 2^kMaxLow buckets, so that
// the counters of a sparse table (20,000 points in 2^17 buckets) fit too. False where the packed entry would not fit 32 bits or a partition
// would hold too many buckets (W > 23).
bool plan_for(const flinng_index *ix, uint64_t n, PartPlan *pl)
{
    const uint32_t W = ix->cfg.range_bits;
    uint32_t C = 0;
    while (C < kMaxC && C < W && (n >> C) > kPartPoints) ++C;
    if (W > kMaxLow && C < W - kMaxLow) C = W - kMaxLow;
    uint32_t idbits = 1;
    while (idbits < 32 && (n - 1) >> idbits) ++idbits;
    *pl = PartPlan{C, W - C, idbits, uint64_t(ix->cfg.L) << C};
    return C <= kMaxC && pl->low + idbits <= 32;
}

}  // namespace

// Step 1 for n new points: bt (room for L x n words; may be anything but buckets)
// receives the transposed buckets, pcur (L << C words) the entries of each
// (table, top C bucket bits).
int partition_count(flinng_index *ix, const uint32_t *buckets, uint64_t n, uint32_t C, uint32_t *bt, uint32_t *pcur)
{
    const cudaStream_t st = ix->stream;
    const uint32_t L = ix->cfg.L, low = ix->cfg.range_bits - C;
    FL_CUDA(cudaMemsetAsync(pcur, 0, (uint64_t(L) << C) * sizeof(uint32_t), st));
    k_transpose<<<dim3(unsigned((n + 31) / 32), (L + 31) / 32), 256, 0, st>>>(buckets, n, L, bt);
    count_launch();
    FL_CUDA(cudaGetLastError());
    k_part_count<<<dim3(unsigned((n + kTile - 1) / kTile), L), kT, sizeof(uint32_t) << C, st>>>(bt, n, C, low, pcur);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

// Step 2, after it: part (n x L entries) grouped by partition, with the groups'
// bases in pbase (L << C of them, the total last); bt is dead afterwards.
int partition_scatter(flinng_index *ix, uint64_t n, uint32_t C, uint32_t idbits, const uint32_t *bt, uint32_t *part,
                      uint32_t *pbase, uint32_t *pcur, void *scan_ws)
{
    const cudaStream_t st = ix->stream;
    const uint32_t L = ix->cfg.L, low = ix->cfg.range_bits - C;
    const uint64_t parts = uint64_t(L) << C;
    FL_TRY(scan_exclusive(pcur, pbase, parts, scan_ws, st));
    FL_CUDA(cudaMemcpyAsync(pcur, pbase, parts * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st));
    const size_t ssm = (sizeof(uint32_t) * 2 << C) + kTile * 6 + (kT / 32) * 4;
    FL_TRY(ensure_dyn_smem((const void *)k_part_scatter, ssm));
    k_part_scatter<<<dim3(unsigned((n + kTile - 1) / kTile), L), kT, ssm, st>>>(bt, n, C, low, idbits, pcur, part);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

// The build scratch and the list array double as the pass buffers (four
// bytes per entry), which takes R >= 2; the general path of build.cu covers
// the rest. heavy_min >= 32 and the list in shared memory bound R and B*R no
// further.
bool part_build_applies(const flinng_index *ix, uint64_t n)
{
    PartPlan pl;
    return ix->cfg.R >= 2 && n > 0 && plan_for(ix, n, &pl);
}

size_t part_workspace_bytes(const flinng_index *ix, uint64_t n)
{
    PartPlan pl;
    if (!plan_for(ix, n, &pl)) return 0;
    const uint64_t entries = n * ix->cfg.L, ch = 2 * (entries / kFinePoints) + 1, wide = entries / kBigChunk + 1;
    return 4 * carve_bytes<uint32_t>(pl.parts + 1) + carve_bytes<uint2>(ch) + carve_bytes<uint32_t>(entries / kHotPoints + 1) +
           3 * carve_bytes<uint2>(wide) + carve_bytes<uint32_t>(wide * ix->BRw) +
           carve_bytes<uint32_t>(entries * ix->cfg.R / ix->heavy_min + 2) + carve_bytes<uint32_t>(8) +
           carve_bytes<char>(scan_workspace_bytes(pl.parts + 1));
}

// buckets: n x L, overwritten (its space takes the partitioned entries).
// Fills off, hidx, cells and the list of heavy slots; *list_out and *count_out
// (device) receive that list and its length. Does not wait.
int part_build(flinng_index *ix, uint32_t *buckets, uint64_t n, void *ws, uint32_t **list_out, uint32_t **count_out)
{
    const cudaStream_t st = ix->stream;
    const uint32_t R = ix->cfg.R, L = ix->cfg.L;
    PartPlan pl;
    if (!plan_for(ix, n, &pl)) return set_error(FLINNG_ERR_INVALID_ARG, "internal: partitioned build");
    const uint64_t entries = n * L;
    Carver c(ws, ~size_t(0));
    uint32_t *pbase = c.take<uint32_t>(pl.parts + 1);
    uint32_t *pcur = c.take<uint32_t>(pl.parts + 1);       // counts, cursors, then the partitions' totals
    uint32_t *tbase = c.take<uint32_t>(pl.parts + 1);
    uint32_t *big = c.take<uint32_t>(pl.parts + 1);
    // a big partition of E > kFinePoints entries has at most 2 E / kFinePoints
    // chunks, a wide slot of c > kBigChunk points at most 2 c / kBigChunk
    const uint64_t nch = 2 * (entries / kFinePoints) + 1, nwide = entries / kBigChunk + 1;
    uint2 *chunks = c.take<uint2>(nch);
    BigLists g{};
    g.hot = c.take<uint32_t>(entries / kHotPoints + 1);
    g.wide = c.take<uint2>(nwide);
    g.wchunk = c.take<uint2>(2 * nwide);
    uint32_t *wbm = c.take<uint32_t>(nwide * ix->BRw);
    uint32_t *list = c.take<uint32_t>(entries * R / ix->heavy_min + 2);
    uint32_t *cnt = c.take<uint32_t>(8);                   // big partitions, chunks, heavy slots; hot, wide slots, their chunks
    void *scan_ws = c.take<char>(scan_workspace_bytes(pl.parts + 1));
    // L x n buckets, later the big partitions' points by bucket, in the list
    // array (2 R bytes per entry), which receives the lists only at the end
    uint32_t *bt = reinterpret_cast<uint32_t *>(ix->cells);
    uint32_t *part = buckets;
    FL_CUDA(cudaMemsetAsync(cnt, 0, 8 * sizeof(uint32_t), st));
    FL_CUDA(cudaMemsetAsync(wbm, 0, nwide * ix->BRw * sizeof(uint32_t), st));
    FL_TRY(partition_count(ix, buckets, n, pl.C, bt, pcur));
    FL_TRY(partition_scatter(ix, n, pl.C, pl.idbits, bt, part, pbase, pcur, scan_ws));
    FineArgs a{};
    a.part = part;
    a.pbase = pbase;
    a.gid = ix->gid;
    a.R = R;
    a.B = ix->cfg.B;
    a.BRw = ix->BRw;
    a.low = pl.low;
    a.idbits = pl.idbits;
    a.noff = ix->slot_b;
    a.tmp = ix->cells_tmp;
    a.ptot = pcur;
    a.big = big;
    a.nbig = cnt;
    a.chunks = chunks;
    a.nchunks = cnt + 1;
    uint32_t *part2 = bt;
    g.sstart = ix->slot_a;
    g.scur = ix->hidx;          // rewritten as a whole at the end
    g.n = cnt + 4;
    const size_t fsm = fine_smem(pl.low, R, ix->BRw), gsm = sizeof(uint32_t) << pl.low;
    const size_t lsm = size_t(kT / 32) * ix->BRw * 4, hsm = size_t(ix->BRw) * 4;
#define FL_RP(call) \
    do { \
        if (ix->rp == 2) { constexpr int RP = 2; call; } \
        else if (ix->rp == 4) { constexpr int RP = 4; call; } \
        else { constexpr int RP = 8; call; } \
        count_launch(); \
        FL_CUDA(cudaGetLastError()); \
    } while (0)
    FL_TRY(ensure_dyn_smem(ix->rp == 2 ? (const void *)k_part_fine<2> : ix->rp == 4 ? (const void *)k_part_fine<4>
                                                                                     : (const void *)k_part_fine<8>, fsm));
    FL_RP((k_part_fine<RP><<<(unsigned)pl.parts, kT, fsm, st>>>(a)));
    k_big_count<<<152 * 8, kT, gsm, st>>>(a);
    count_launch();
    FL_CUDA(cudaGetLastError());
    k_big_starts<<<152 * 8, kT, 0, st>>>(a, g);
    count_launch();
    FL_CUDA(cudaGetLastError());
    k_big_scatter<<<152 * 8, kT, gsm, st>>>(a, g, part2);
    count_launch();
    FL_CUDA(cudaGetLastError());
    FL_TRY(ensure_dyn_smem(ix->rp == 2 ? (const void *)k_big_lists<2> : ix->rp == 4 ? (const void *)k_big_lists<4>
                                                                                     : (const void *)k_big_lists<8>, lsm));
    // k_big_lists first: it tells the hot slots by their number of points, which
    // the others replace with the length of the list
    FL_RP((k_big_lists<RP><<<152 * 8, kT, lsm, st>>>(a, part2, g.sstart)));
    FL_RP((k_big_hot<RP><<<152 * 8, kT, 2 * hsm, st>>>(a, part2, g)));
    FL_RP((k_big_wide<RP><<<152 * 8, kT, hsm, st>>>(a, part2, g, wbm)));
    k_big_wide_list<<<152 * 8, kT, 2 * hsm, st>>>(a, g, wbm);
    count_launch();
    FL_CUDA(cudaGetLastError());
    k_big_scan<<<152 * 8, kT, 0, st>>>(a);
    count_launch();
    FL_CUDA(cudaGetLastError());
    FL_TRY(scan_exclusive(pcur, tbase, pl.parts, scan_ws, st));
    k_part_finish<<<(unsigned)pl.parts, kT, 0, st>>>(a, pl.parts, tbase, g.sstart, ix->heavy_min, ix->hidx, list, cnt + 2,
                                                     ix->cells);
    count_launch();
    FL_CUDA(cudaGetLastError());
#undef FL_RP
    *list_out = list;
    *count_out = cnt + 2;
    return FLINNG_OK;
}

}  // namespace flinng
