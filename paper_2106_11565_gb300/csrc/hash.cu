// LSH hashing of points and queries (Sec. 3.2, Sec. 5: the L shared hash
// functions, each the concatenation of K base hashes).
//
// Cosine: sign random projections. bit j of table l = (w_{lK+j} . x > 0),
// table bucket = the K bits, bit j at position j. The sign is exact: an FP32
// tile GEMM (a warp per projection for a few rows) computes p~ and a rigorous
// bound on |p~ - p|; the few projections whose |p~| does not clear the bound
// are recomputed in fp64 (fp32 x fp32 products are exact in fp64) and, if still
// ambiguous, summed exactly in a fixed-point long accumulator.
//
// Jaccard: densified one-permutation MinHash. pi(e) = a e + b mod 2^32,
// nb = L*K bins of the 32-bit range, bin value = min pi(e) in the bin; an
// empty bin copies the value of the first originally non-empty bin among
// j = splitmix64(seed ^ (i << 32 | attempt)) mod nb, attempt = 1, 2, ...
// (4096 tries, then the next non-empty bin cyclically). Table l combines its
// K values as ((sum_j a_{l,j} v_{lK+j} + c_l) mod 2^64) >> (64 - W).
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "internal.cuh"
#include "doph.cuh"
#include "srp_rows.cuh"

namespace flinng {

namespace {

// ------------------------------------------------------------------ SRP

constexpr int kBN = 64, kBK = 16;
constexpr int kFold = 2;                     // k-tiles per accumulation chain
constexpr int kSrpChunkRows = 1 << 14;
constexpr int kGemvPer = 8;                  // rows a warp takes at a time

__device__ __forceinline__ void ffma2(unsigned long long &d, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

__device__ __forceinline__ void fadd2(unsigned long long &d, unsigned long long a)
{
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(d) : "l"(a));
}

__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ void unpack2(unsigned long long v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// BM x 64 projections per CTA of 2 BM threads, 8 x 4 each, two rows per packed
// FMA; the next k-tile's loads are in flight while this one is multiplied.
//
// The sums run in chains of kFold k-tiles (32 products), each folded into a
// total, so that |p~ - p| <= [g(32) + g(m)(1 + g(32))] sum |w_i x_i| with m =
// ceil(d / 32), and sum |w_i x_i| <= ||w|| ||x||: the margin needs the rows'
// norms (the x side's squares are summed as its tiles pass by) instead of a
// second FMA per product, and at d = 4096 it is a twentieth of one chain's.
// Bound by the FP32 pipe (packed FMAs take two of its cycles) and, at this size,
// by 256 CTAs on 304 places. 2,000 rows x 1,024 projections x d = 4096: 784 us
// with the second sum and one chain, which left 1.1 % of the signs to an fp64
// re-check of 942 us; 491 us and 59 us now.
template <int BM, bool VEC>
__global__ void __launch_bounds__(2 * BM, 512 / (2 * BM))
k_srp_fp32(const float *__restrict__ X, uint64_t ldx, uint64_t n, const float *__restrict__ Wm,
           const float *__restrict__ wnorm, uint32_t P, uint32_t d, uint32_t L, uint32_t K, float c_norm, float tiny,
           uint32_t *__restrict__ codes, float *__restrict__ proj, unsigned long long *__restrict__ rlist,
           unsigned long long *__restrict__ rcount)
{
    constexpr int NT = 2 * BM, kNB = kBN * kBK / 4 / NT;      // float4 loads of W per thread and tile
    __shared__ __align__(16) float As[2][kBK][BM + 4];
    __shared__ __align__(16) float Bs[2][kBK][kBN + 4];
    __shared__ float xn[BM];
    const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
    const uint64_t row0 = uint64_t(blockIdx.x) * BM;
    const uint32_t col0 = blockIdx.y * kBN;
    // this thread's loads: rows lr, lr + BM / 2 of x and row lr of W, k 4 lk .. + 3
    const int lk = tid & 3, lr = tid >> 2;
    const float *xr[2];
    bool xin[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const uint64_t r = row0 + lr + e * (BM / 2);
        xin[e] = r < n;
        xr[e] = X + (xin[e] ? r : 0) * ldx;
    }
    const float *wr[kNB];
    bool win[kNB];
#pragma unroll
    for (int e = 0; e < kNB; ++e) {
        const uint32_t c = col0 + lr + e * (NT / 4);
        win[e] = c < P;
        wr[e] = Wm + uint64_t(win[e] ? c : 0) * d;
    }
    unsigned long long tot[4][4], acc[4][4];       // [row pair][column]
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) tot[i][j] = acc[i][j] = 0ull;
    float ss[2] = {0.f, 0.f};
    bool any[2] = {false, false};
    float4 ra[2], rb[kNB];
    auto load = [&](uint32_t k0) {
#pragma unroll
        for (int e = 0; e < 2; ++e) ra[e] = load4<VEC>(xr[e], k0 + 4 * lk, d, xin[e]);
#pragma unroll
        for (int e = 0; e < kNB; ++e) rb[e] = load4<VEC>(wr[e], k0 + 4 * lk, d, win[e]);
    };
    auto stage = [&](int b) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float4 v = ra[e];
            const int r = lr + e * (BM / 2);
            As[b][4 * lk][r] = v.x;
            As[b][4 * lk + 1][r] = v.y;
            As[b][4 * lk + 2][r] = v.z;
            As[b][4 * lk + 3][r] = v.w;
            ss[e] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, ss[e]))));
            any[e] |= v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f;
        }
#pragma unroll
        for (int e = 0; e < kNB; ++e) {
            const float4 v = rb[e];
            const int c = lr + e * (NT / 4);
            Bs[b][4 * lk][c] = v.x;
            Bs[b][4 * lk + 1][c] = v.y;
            Bs[b][4 * lk + 2][c] = v.z;
            Bs[b][4 * lk + 3][c] = v.w;
        }
    };
    const uint32_t nt = (d + kBK - 1) / kBK;
    load(0);
    stage(0);
    __syncthreads();
    for (uint32_t t = 0; t < nt; ++t) {
        const int b = t & 1;
        if (t + 1 < nt) load((t + 1) * kBK);
#pragma unroll
        for (int kk = 0; kk < kBK; ++kk) {
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(&As[b][kk][ty * 8]);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(&As[b][kk][ty * 8 + 4]);
            const float4 bv = *reinterpret_cast<const float4 *>(&Bs[b][kk][tx * 4]);
            const unsigned long long av[4] = {a0.x, a0.y, a1.x, a1.y};
            const unsigned long long bb[4] = {pack2(bv.x, bv.x), pack2(bv.y, bv.y), pack2(bv.z, bv.z),
                                              pack2(bv.w, bv.w)};
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) ffma2(acc[i][j], av[i], bb[j]);
        }
        if (t % kFold == kFold - 1 || t + 1 == nt) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    fadd2(tot[i][j], acc[i][j]);
                    acc[i][j] = 0ull;
                }
        }
        if (t + 1 < nt) stage(b ^ 1);
        __syncthreads();
    }
    // norms of the x rows: four lanes hold a row's squares
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        float v = ss[e];
        v += __shfl_xor_sync(0xffffffffu, v, 1);
        v += __shfl_xor_sync(0xffffffffu, v, 2);
        const uint32_t nz = __ballot_sync(0xffffffffu, any[e]);
        const bool some = ((nz >> (tid & 28)) & 0xFu) != 0u;
        float nrm = norm_up(v, d / 4 + 16);
        if (!norm_in_range(v, some)) {
            // uniform over the row's four lanes, which shuffle among themselves
            double s64 = 0.0;
            for (uint32_t t = lk; t < d; t += 4) s64 += double(xr[e][t]) * double(xr[e][t]);
            const uint32_t mine = 0xFu << (tid & 28);
            s64 += __shfl_xor_sync(mine, s64, 1);
            s64 += __shfl_xor_sync(mine, s64, 2);
            nrm = norm_up64(s64);
        }
        if (lk == 0) xn[lr + e * (BM / 2)] = nrm;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint64_t gr = row0 + ty * 8 + i;
        if (gr >= n) continue;
        const float nx = xn[ty * 8 + i];
        uint32_t cur_l = 0xFFFFFFFFu, bits = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t gc = col0 + tx * 4 + j;
            if (gc >= P) continue;
            float lo, hi;
            unpack2(tot[i / 2][j], lo, hi);
            const float p = (i & 1) ? hi : lo;
            if (proj) proj[gr * P + gc] = p;
            // the norms' product first: a factor of 1e-6 would lose a tiny row's bound to
            // underflow. A sum that overflowed on the way decides nothing (its margin may
            // be finite).
            const float margin = fmaf(c_norm, nx * wnorm[gc], tiny);
            if (fabsf(p) > margin && fabsf(p) <= FLT_MAX) {
                const uint32_t l = gc / K;
                if (l != cur_l) {
                    if (bits) atomicOr(&codes[gr * L + cur_l], bits);
                    cur_l = l;
                    bits = 0u;
                }
                if (p > 0.f) bits |= 1u << (gc % K);
            } else {
                const unsigned long long slot = atomicAdd(rcount, 1ull);
                rlist[slot] = (p > 0.f ? kEntSign : 0ull) | ((unsigned long long)gr << 20) | gc;
            }
        }
        if (bits) atomicOr(&codes[gr * L + cur_l], bits);
    }
}

// A few rows: a warp per projection and kGemvPer rows, which share the
// projection's loads; bound by the latency of W's rows from L2. The GEMM's grid would be a handful of CTAs each walking
// all of d. Lane sums of d / 32 products, then a tree: |p~ - p| <= g(d / 32 + 8)
// sum |w_i x_i|, that sum accumulated beside p~ (gamma2 covers both roundings).
template <bool VEC>
__global__ void __launch_bounds__(256)
k_srp_gemv(const float *__restrict__ X, uint64_t ldx, uint32_t n, const float *__restrict__ Wm, uint32_t P, uint32_t d,
           uint32_t L, uint32_t K, float gamma2, float tiny, uint32_t *__restrict__ codes, float *__restrict__ proj,
           unsigned long long *__restrict__ rlist, unsigned long long *__restrict__ rcount)
{
    const uint32_t lane = threadIdx.x & 31, j = blockIdx.x * 8 + (threadIdx.x >> 5), r0 = blockIdx.y * kGemvPer;
    if (j >= P) return;
    const float *wj = Wm + uint64_t(j) * d;
    float p[kGemvPer], sa[kGemvPer];
#pragma unroll
    for (int r = 0; r < kGemvPer; ++r) p[r] = sa[r] = 0.f;
    for (uint32_t t = lane * 4; t < d; t += 128) {
        const float4 w = load4<VEC>(wj, t, d, true);
#pragma unroll
        for (int r = 0; r < kGemvPer; ++r) {
            const float4 v = load4<VEC>(X + uint64_t(min(r0 + r, n - 1)) * ldx, t, d, r0 + r < n);
            p[r] = fmaf(w.x, v.x, fmaf(w.y, v.y, fmaf(w.z, v.z, fmaf(w.w, v.w, p[r]))));
            sa[r] = fmaf(fabsf(w.x), fabsf(v.x), fmaf(fabsf(w.y), fabsf(v.y),
                         fmaf(fabsf(w.z), fabsf(v.z), fmaf(fabsf(w.w), fabsf(v.w), sa[r]))));
        }
    }
#pragma unroll
    for (int r = 0; r < kGemvPer; ++r) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            p[r] += __shfl_xor_sync(0xffffffffu, p[r], o);
            sa[r] += __shfl_xor_sync(0xffffffffu, sa[r], o);
        }
        if (lane != uint32_t(r) || r0 + r >= n) continue;
        const uint64_t gr = r0 + r;
        if (proj) proj[gr * P + j] = p[r];
        if (fabsf(p[r]) > fmaf(gamma2, sa[r], tiny)) {
            if (p[r] > 0.f) atomicOr(&codes[gr * L + j / K], 1u << (j % K));
        } else {
            rlist[atomicAdd(rcount, 1ull)] = (p[r] > 0.f ? kEntSign : 0ull) | ((unsigned long long)gr << 20) | j;
        }
    }
}

// Upper bounds of the rows' norms, a warp per row.
__global__ void k_row_norms(const float *__restrict__ x, uint64_t ld, uint64_t n, uint32_t d, float *__restrict__ norm)
{
    const int lane = threadIdx.x & 31;
    const uint64_t gw = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t r = gw; r < n; r += nw) {
        double ss = 0.0;
        for (uint32_t t = lane; t < d; t += 32) ss += double(x[r * ld + t]) * double(x[r * ld + t]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        if (lane == 0) norm[r] = norm_up64(ss);
    }
}

// Exact sign of sum_t a_t b_t with fp32 inputs: each product is an fp64
// value m * 2^(e-1075) with a 53-bit integer m; digits of 32 bits starting
// at 2^-384, kept in int64 so that sums over lanes and terms cannot overflow.
constexpr int kLimbs = 24;
constexpr int kLimbBias = 384;

__device__ void limb_add(long long *acc, double v)
{
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int ex = int((bits >> 52) & 0x7FF);
    unsigned long long man = bits & ((1ull << 52) - 1);
    if (ex == 0 && man == 0) return;
    int lsb;
    if (ex == 0) {
        lsb = 1 - 1075;
    } else {
        man |= 1ull << 52;
        lsb = ex - 1075;
    }
    const int pos = lsb + kLimbBias;
    const int q = pos >> 5, r = pos & 31;
    const unsigned long long d0 = (man << r) & 0xffffffffull;
    const unsigned long long d1 = (r == 0 ? (man >> 32) : (man >> (32 - r))) & 0xffffffffull;
    const unsigned long long d2 = (r == 0) ? 0ull : (man >> (64 - r));
    const long long sg = (bits >> 63) ? -1 : 1;
    acc[q] += sg * (long long)d0;
    acc[q + 1] += sg * (long long)d1;
    acc[q + 2] += sg * (long long)d2;
}

__device__ int limb_sign(long long *acc)
{
    for (int i = 0; i < kLimbs - 1; ++i) {
        const long long c = acc[i] >> 32;   // arithmetic shift: floor division
        acc[i] -= c * 4294967296ll;
        acc[i + 1] += c;
    }
    if (acc[kLimbs - 1] != 0) return acc[kLimbs - 1] > 0 ? 1 : -1;
    for (int i = kLimbs - 2; i >= 0; --i)
        if (acc[i] != 0) return 1;
    return 0;
}

// A CTA per listed projection: the FP64 pipe takes tens of cycles per warp
// instruction here, so a warp alone needs 50 us for a row of 4,096 and the few
// entries of a batch were waited for one warp each. fp64 sum first, then the
// exact accumulator.
constexpr int kReThreads = 256;

__global__ void __launch_bounds__(kReThreads)
k_srp_recheck(const float *__restrict__ X, uint64_t ldx, const float *__restrict__ Wm, uint32_t d, uint32_t L,
              uint32_t K, double gamma2, const unsigned long long *__restrict__ rlist,
              const unsigned long long *__restrict__ rcount, uint32_t *__restrict__ codes,
              unsigned long long *__restrict__ stats)
{
    __shared__ double sp[kReThreads / 32], sq[kReThreads / 32];
    __shared__ unsigned long long limb[kLimbs + 2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long nlist = *rcount;
    for (unsigned long long e = blockIdx.x; e < nlist; e += gridDim.x) {
        const unsigned long long ent = rlist[e];
        const uint64_t gr = ent_row(ent);
        const uint32_t gc = ent_col(ent);
        const float *xr = X + gr * ldx;
        const float *wr = Wm + uint64_t(gc) * d;
        double p = 0.0, s = 0.0;
        for (uint32_t t = tid; t < d; t += kReThreads) {
            const double prod = double(xr[t]) * double(wr[t]);
            p += prod;
            s += fabs(prod);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            p += __shfl_xor_sync(0xffffffffu, p, o);
            s += __shfl_xor_sync(0xffffffffu, s, o);
        }
        if (lane == 0) {
            sp[warp] = p;
            sq[warp] = s;
        }
        if (tid < kLimbs + 2) limb[tid] = 0ull;
        __syncthreads();
        p = s = 0.0;
#pragma unroll
        for (int w = 0; w < kReThreads / 32; ++w) {
            p += sp[w];
            s += sq[w];
        }
        int positive = p > 0.0;
        if (!(fabs(p) > gamma2 * s)) {               // uniform: every thread has the same sums
            long long acc[kLimbs + 2];
            for (int i = 0; i < kLimbs + 2; ++i) acc[i] = 0;
            for (uint32_t t = tid; t < d; t += kReThreads) limb_add(acc, double(xr[t]) * double(wr[t]));
            // digits sum exactly in 64-bit integers (two's complement: signs too)
            for (int i = 0; i < kLimbs + 2; ++i) {
                long long v = acc[i];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == 0) atomicAdd(&limb[i], (unsigned long long)v);
            }
            __syncthreads();
            if (tid == 0) {
                for (int i = 0; i < kLimbs + 2; ++i) acc[i] = (long long)limb[i];
                // digits kLimbs, kLimbs+1 stay zero: fold them for safety
                acc[kLimbs - 1] += acc[kLimbs] * 4294967296ll;
                positive = limb_sign(acc) > 0;
                atomicAdd(&stats[1], 1ull);
            }
        }
        if (tid == 0) {
            if (positive) atomicOr(&codes[gr * L + gc / K], 1u << (gc % K));
            atomicAdd(&stats[2], 1ull);
            if (positive != ((ent & kEntSign) != 0)) atomicAdd(&stats[4], 1ull);
        }
        __syncthreads();                             // before the next entry overwrites the sums
    }
}

__global__ void k_add_counter(unsigned long long *dst, const unsigned long long *src)
{
    *dst += *src;
}

// ------------------------------------------------------------------ DOPH

constexpr int kDophWarps = 8;
constexpr int kDophUnroll = 4;     // element loads in flight per lane

// The table of each bin's first densification draws.
__global__ void k_doph_draws(uint32_t nb, uint64_t seed, uint16_t *__restrict__ draw)
{
    const uint32_t t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nb * kDophTable) draw[t] = uint16_t(doph_draw_of(t / kDophTable, t % kDophTable + 1, nb, seed));
}

// 32-bit words of shared memory per set: bin minima, occupancy and, with LIST, the empty bins
__host__ __device__ inline uint32_t doph_words(uint32_t nb, bool list)
{
    return nb + (nb + 31) / 32 + (list ? (nb + 1) / 2 : 0);
}

template <bool LIST>
__global__ void __launch_bounds__(kDophWarps * 32)
k_doph(const uint64_t *__restrict__ off, const uint32_t *__restrict__ elems,
       uint64_t n, uint32_t nb, uint32_t a, uint32_t b, uint64_t seed, uint32_t L,
       uint32_t K, uint32_t W, const uint64_t *__restrict__ ba,
       const uint64_t *__restrict__ bc, const uint16_t *__restrict__ draw,
       uint32_t *__restrict__ buckets, uint32_t *__restrict__ values)
{
    extern __shared__ uint32_t sm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t nbw = (nb + 31) / 32;
    uint32_t *val = sm + warp * doph_words(nb, LIST);
    uint32_t *occ = val + nb;
    uint16_t *empty = reinterpret_cast<uint16_t *>(occ + nbw);     // nb: the empty bins
    const uint64_t gw = uint64_t(blockIdx.x) * kDophWarps + warp;
    const uint64_t stride = uint64_t(gridDim.x) * kDophWarps;
    for (uint64_t i = gw; i < n; i += stride) {
        for (uint32_t k = lane; k < nb; k += 32) val[k] = kEmpty32;
        for (uint32_t k = lane; k < nbw; k += 32) occ[k] = 0u;
        __syncwarp();
        const uint64_t beg = off[i], end = off[i + 1];
        // four element loads in flight per lane, then their bins
        for (uint64_t t0 = beg + lane; t0 < end; t0 += 32 * kDophUnroll) {
            uint32_t e[kDophUnroll];
#pragma unroll
            for (int u = 0; u < kDophUnroll; ++u) {
                const uint64_t t = t0 + 32u * u;
                e[u] = t < end ? elems[t] : 0u;
            }
#pragma unroll
            for (int u = 0; u < kDophUnroll; ++u) {
                if (t0 + 32u * u >= end) break;
                const uint32_t pe = a * e[u] + b;
                const uint32_t bin = __umulhi(pe, nb);
                atomicMin(&val[bin], pe);
                // a bin is occupied iff its minimum is below the empty marker,
                // or an element hashes to the marker's value itself (flagged
                // here; every other occupancy bit is read off val below, with
                // no atomic per element on the few bitmap words)
                if (pe == kEmpty32) atomicOr(&occ[bin >> 5], 1u << (bin & 31));
            }
        }
        __syncwarp();
        uint32_t ne = 0;
        for (uint32_t k0 = 0; k0 < nb; k0 += 32) {                 // a ballot per 32 bins
            const uint32_t k = k0 + lane;
            const uint32_t bits = __ballot_sync(0xffffffffu, k < nb && val[k] != kEmpty32) | occ[k0 >> 5];
            __syncwarp();
            if (lane == 0) occ[k0 >> 5] = bits;
            // the empty bins listed: a third to a seventh of them, so a loop over
            // the list keeps the lanes busy where one over all bins left most
            // idle through the other lanes' draws (with doph_source's table,
            // 100,000 genomic reads, 512 bins: 300 -> 200 us; 10^6 URL sets, 64
            // bins: 801 -> 461 us)
            if constexpr (LIST) {
                const uint32_t none = ~bits & (nb - k0 >= 32 ? 0xffffffffu : (1u << (nb - k0)) - 1u);
                if ((none >> lane) & 1u) empty[ne + __popc(none & ((1u << lane) - 1u))] = uint16_t(k);
                ne += __popc(none);
            }
        }
        __syncwarp();
        if (end > beg) {
            for (uint32_t i = lane; i < (LIST ? ne : nb); i += 32) {
                const uint32_t k = LIST ? empty[i] : i;
                if (LIST || !((occ[k >> 5] >> (k & 31)) & 1u)) val[k] = val[doph_source(k, nb, seed, draw, occ)];
            }
        }
        __syncwarp();
        if (values)
            for (uint32_t k = lane; k < nb; k += 32) values[i * nb + k] = val[k];
        for (uint32_t l = lane; l < L; l += 32) {
            uint64_t h = bc[l];
            for (uint32_t j = 0; j < K; ++j) h += ba[l * K + j] * uint64_t(val[l * K + j]);
            buckets[i * L + l] = uint32_t(h >> (64 - W));
        }
        __syncwarp();
    }
}

}  // namespace

int add_counter(unsigned long long *dst, const unsigned long long *src, cudaStream_t st)
{
    k_add_counter<<<1, 1, 0, st>>>(dst, src);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

int srp_recheck_list(flinng_index *ix, const float *x, uint64_t ld, const unsigned long long *list,
                     const unsigned long long *count, uint32_t *codes)
{
    k_srp_recheck<<<152 * 4, kReThreads, 0, ix->stream>>>(x, ld, ix->srp_w, ix->cfg.dim, ix->cfg.L, ix->cfg.K,
                                                          ix->srp_gamma64, list, count, codes, ix->stats);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

int srp_weight_norms(flinng_index *ix)
{
    k_row_norms<<<152 * 4, 256, 0, ix->stream>>>(ix->srp_w, ix->cfg.dim, ix->P, ix->cfg.dim, ix->w_norm);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

// bytes of the re-check counter and list of one chunk
static size_t list_workspace_bytes(const flinng_index *ix, uint64_t n)
{
    const uint64_t rows = n < uint64_t(kSrpChunkRows) ? n : uint64_t(kSrpChunkRows);
    return carve_bytes<unsigned long long>(2) + carve_bytes<unsigned long long>(rows * ix->P + 1);
}

size_t srp_workspace_bytes(const flinng_index *ix, uint64_t n)
{
    return ix->cfg.precision != FLINNG_PREC_FP32 ? srp_tc_workspace_bytes(ix, n) : list_workspace_bytes(ix, n);
}

// Small batches take the fp32 warp-per-projection kernel: the GEMM's tiles would
// be a few CTAs, each walking all of d. The lines lie where the two cross: 1,024
// projections at d = 4096, 128 rows 145 us against 216 (tiles), 192 rows 208
// against 216; the tensor-core path needs 98 us for any of them (two-term; 108 and
// 158 the single-term forms) against 94 at 72 rows and 118 at 96, and at d = 1024
// 57 (58, 81) against 50 at 96: the line lies between. Less work per row (fewer
// projections) moves the fp32 line out in proportion (384 projections at d = 512:
// equal at 512 rows). In the tensor-core precisions only without projections to
// return: the codes are the same.
bool srp_few_rows(const flinng_index *ix, uint64_t n, const float *proj)
{
    // (a short row leaves most of a warp idle: 2,000 rows x 64 projections of 32
    // dimensions 31 us, 26 in tiles)
    if (ix->cfg.precision == FLINNG_PREC_FP32) return n * ix->P <= (ix->cfg.dim < 128 ? 96 : 192) * 1024;
    return !proj && n <= 96 && n * ix->P <= 96 * 1024;
}

int srp_hash(flinng_index *ix, const float *x, uint64_t ld, uint64_t n,
             uint32_t *buckets, float *proj, void *ws, size_t ws_bytes)
{
    if (ix->h_flag[3]) return set_error(FLINNG_ERR_TIMEOUT, "tensor-core SRP: a pipeline wait timed out");
    const bool few = srp_few_rows(ix, n, proj);
    if (ix->cfg.precision != FLINNG_PREC_FP32 && !few) return srp_hash_tc(ix, x, ld, n, buckets, proj, ws, ws_bytes);
    const cudaStream_t st = ix->stream;
    const uint32_t L = ix->cfg.L, K = ix->cfg.K, d = ix->cfg.dim, P = ix->P;
    Carver c(ws, ~size_t(0));
    unsigned long long *rcount = c.take<unsigned long long>(2);
    unsigned long long *rlist = c.take<unsigned long long>(uint64_t(kSrpChunkRows) * P + 1);
    FL_CUDA(cudaMemsetAsync(ix->stats, 0, kStats * sizeof(unsigned long long), st));
    if (n == 0) return FLINNG_OK;
    FL_CUDA(cudaMemsetAsync(buckets, 0, n * L * sizeof(uint32_t), st));
    const double u = std::ldexp(1.0, -24);
    auto g = [&](double m) { return m * u / (1.0 - m * u); };
    const double kb = kFold * kBK, f = g(kb) + g(std::ceil(d / kb)) * (1 + g(kb));
    const float c_norm = std::nextafter(float(f * 1.0001), INFINITY);
    const float gemv2 = std::nextafter(float(2.0 * g(std::ceil(d / 32.0) + 8)), INFINITY);
    const float tiny = float(d) * ldexpf(1.0f, -146);     // underflow of products and sums
    const bool vec = rows_vec4(x, ld, d);
    if (!ix->sms) FL_CUDA(cudaDeviceGetAttribute(&ix->sms, cudaDevAttrMultiProcessorCount, ix->device));
    for (uint64_t r0 = 0; r0 < n; r0 += kSrpChunkRows) {
        const uint64_t rows = (n - r0) < uint64_t(kSrpChunkRows) ? (n - r0) : uint64_t(kSrpChunkRows);
        const float *xc = x + r0 * ld;
        uint32_t *codes = buckets + r0 * L;
        float *pc = proj ? proj + r0 * P : nullptr;
        FL_CUDA(cudaMemsetAsync(rcount, 0, sizeof(unsigned long long), st));
        if (few) {
            const dim3 grid((P + 7) / 8, unsigned((rows + kGemvPer - 1) / kGemvPer));
            auto fn = vec ? k_srp_gemv<true> : k_srp_gemv<false>;
            fn<<<grid, 256, 0, st>>>(xc, ld, uint32_t(rows), ix->srp_w, P, d, L, K, gemv2, tiny, codes, pc, rlist,
                                     rcount);
        } else {
            // tiles of 128 rows, or of 64 while 128 would leave SMs without a CTA
            const bool wide = ((rows + 127) / 128) * ((P + kBN - 1) / kBN) >= uint64_t(ix->sms);
            const uint64_t bm = wide ? 128 : 64;
            const dim3 grid(unsigned((rows + bm - 1) / bm), (P + kBN - 1) / kBN);
            auto fn = wide ? (vec ? k_srp_fp32<128, true> : k_srp_fp32<128, false>)
                           : (vec ? k_srp_fp32<64, true> : k_srp_fp32<64, false>);
            fn<<<grid, unsigned(2 * bm), 0, st>>>(xc, ld, rows, ix->srp_w, ix->w_norm, P, d, L, K, c_norm, tiny, codes,
                                                  pc, rlist, rcount);
        }
        count_launch();
        FL_CUDA(cudaGetLastError());
        FL_TRY(add_counter(ix->stats, rcount, st));        // undecided after the fp32 pass
        FL_TRY(srp_recheck_list(ix, xc, ld, rlist, rcount, codes));
    }
    return FLINNG_OK;
}

int doph_draws(flinng_index *ix)
{
    const uint32_t nb = ix->P;
    k_doph_draws<<<(nb * kDophTable + 255) / 256, 256, 0, ix->stream>>>(nb, ix->doph_seed, ix->doph_draw);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

int doph_hash(flinng_index *ix, const uint64_t *off, const uint32_t *elems,
              uint64_t n, uint32_t *buckets, uint32_t *values)
{
    if (n == 0) return FLINNG_OK;
    const uint32_t nb = ix->P;
    // the list of empty bins while it costs no resident CTA (100,000 URL sets, 2,048
    // bins: 92 ms with it and two CTAs per SM, 74 without and three)
    auto bytes = [&](bool list) { return size_t(kDophWarps) * doph_words(nb, list) * sizeof(uint32_t); };
    auto ctas = [&](size_t b) { return std::min<size_t>(228 * 1024 / (b + 1024), 2048 / (kDophWarps * 32)); };
    const bool list = ctas(bytes(true)) >= ctas(bytes(false));
    const size_t smem = bytes(list);
    auto fn = list ? k_doph<true> : k_doph<false>;
    FL_TRY(ensure_dyn_smem((const void *)fn, smem));
    uint64_t blocks = (n + kDophWarps - 1) / kDophWarps;
    if (blocks > 152ull * 64) blocks = 152ull * 64;
    fn<<<(unsigned)blocks, kDophWarps * 32, smem, ix->stream>>>(
        off, elems, n, nb, ix->doph_a, ix->doph_b, ix->doph_seed, ix->cfg.L, ix->cfg.K,
        ix->cfg.range_bits, ix->bucket_a, ix->bucket_c, ix->doph_draw, buckets, values);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

}  // namespace flinng
