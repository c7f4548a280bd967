// Sign random projections on the tensor cores (the precision form): the
// dense contraction P = X W^T runs on tcgen05 with BF16 operands and FP32
// accumulation in tensor memory, and the sign bits stay exact.
//
// Exactness. Each fp32 operand is split as x1 = bf16(x), x2 = bf16(x - x1),
// so |x - x1 - x2| <= 2^-16 |x| (bf16 keeps 8 significant bits); likewise w.
// bf16 x bf16 products are exact in fp32. Per 64-wide k-block s the tensor
// cores compute hi_s = sum x1 w1 and lo_s = sum (x1 w2 + x2 w1) into a fresh
// pair of TMEM accumulators; the epilogue adds hi_s + lo_s into an fp32
// register per projection. Short accumulation chains keep the bound tight:
//   |p~ - w.x| <= [g'(64) + 2^-7 g'(128)] (1 + 2^-8)^2 ||x|| ||w||      (blocks)
//              + g(2m) (1 + g'(64)) (1 + 2^-7) (1 + 2^-8)^2 ||x|| ||w||  (sum of m blocks)
//              + 2^-8 (||x|| ||r_w|| + ||r_x|| ||w||)
//              + (1 + 2^-6) ||r_x|| ||r_w||                              (split)
//              + 8 d 2^-126 + sqrt(d) 2^-125 (||x|| + ||w||)           (underflow, flushes)
// where r = x - x1 is what the second term rounds (|x2| <= (1 + 2^-8) |r|, |r -
// x2| <= 2^-8 |r|; the dropped terms are w2.x2, w.(r_x - x2), (r_w - w2).x and
// their cross term): its norm, measured per row, is about a quarter of its
// worst case 2^-8 ||x||, and the worst case alone (3.1 * 2^-16 ||x|| ||w||) was two
// thirds of the margin (8,192 rows of 4,096, BF16: 548 us with it, 523 without;
// a query batch of 10,000 in this form 2,069 -> 2,003). With g(n) = n u / (1 - n u), u = 2^-24, and g' the same with u' = 2^-22:
// four units of fp32 rounding per product accumulated, which also covers a
// tensor-core adder that aligns and truncates. Projections whose |p~| does
// not clear that margin go to a compensated fp32 re-check (two-product,
// two-sum), and the few that stay ambiguous to the fp64 / exact re-check of
// hash.cu.
//
// Single-term forms. FLINNG_PREC_BF16 keeps x1 = bf16(x) only; FLINNG_PREC_FP8
// keeps xq = e4m3(x / s) with a power-of-two scale s per row (s chosen so the
// row's largest |x| / s <= 448; values that would be E4M3 subnormals become
// 0). The quantiser records each row's residual norm ||e_x|| = ||x - s xq||
// (exact fp64 differences, rounded up); with ||x|| and the same for every
// projection row w,
//   |w.x - s_x s_w sum xq wq| <= ||x|| ||e_w|| + ||e_x|| ||w|| + 3 ||e_x|| ||e_w||
// (Cauchy-Schwarz on x = s_x xq + e_x, w = s_w wq + e_w). The tensor cores sum
// the products of one k-block (64 bf16 or 128 e4m3 values) exactly-multiplied
// into fp32 (per-product error u' = 2^-22 of the running magnitude), the
// epilogue adds the blocks in fp32 and scales by s_x s_w (exact), so the
// margin is that residual term plus [g'(kb) + g(m)(1 + g'(kb))] (||x|| +
// ||e_x||) (||w|| + ||e_w||), 2^-23 |p~|, the underflow terms above, and a
// 2^-20 relative slack for evaluating the margin itself in fp32.
//
// Kernel layout (one CTA per 128 points x 128 projections, 576 threads):
//   warp 0     TMA producer: 3-stage ring of {X1, X2, W1, W2} tiles of 128 rows
//              x 64 bf16 (128-byte swizzle), one mbarrier per stage (single-term
//              forms: a 6-stage ring of {X, W} tiles of 128 rows x 128 bytes);
//   warp 1     allocates 512 TMEM columns (two buffers of {hi, lo}); one elected
//              thread issues the MMAs of k-block s into buffer s % 2 - per 16-wide
//              step x1 [w1 w2] (M=128, N=256: hi and the x1 w2 half of lo) and
//              x2 w1 (N=128, into lo) - then commits the stage back to the
//              producer and the buffer to the epilogue (single-term forms: one
//              N=128 MMA per 32-byte step into a 128-column buffer);
//   warps 2-17 epilogue: warp w reads TMEM lanes 32 (w % 4) .. +32 (one point per
//              thread) and 32 of the 128 columns, drains each buffer into fp32
//              registers and hands it back; at the end decides the signs,
//              writes the codes and lists ambiguous projections.
// Every wait on an mbarrier is bounded; on timeout the CTA sets an error flag,
// stops issuing work, waits (bounded) for its copies and MMAs, and frees TMEM.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "internal.cuh"
#include "srp_rows.cuh"

namespace flinng {
namespace {

constexpr int kTM = 128, kTN = 128, kTK = 64;     // tile rows, projections, bf16 K per stage
constexpr int kTileBytes = kTM * 128;             // 16 KB per operand tile (128-byte rows)
// forms of the kernel
constexpr int kFormBf16x2 = 0, kFormBf16 = 1, kFormFp8 = 2;

template <int FORM> struct TcForm;
template <> struct TcForm<kFormBf16x2> {
    static constexpr int kTiles = 4, kStages = 3, kKElems = 64;   // X1, X2, W1, W2
    static constexpr uint32_t kTmemCols = 512;                    // buffer b: hi at 256 b, lo at 256 b + 128
};
template <> struct TcForm<kFormBf16> {
    static constexpr int kTiles = 2, kStages = 6, kKElems = 64;   // X, W
    static constexpr uint32_t kTmemCols = 256;                    // buffer b at 128 b
};
template <> struct TcForm<kFormFp8> {
    static constexpr int kTiles = 2, kStages = 6, kKElems = 128;
    static constexpr uint32_t kTmemCols = 256;
};
template <int FORM>
constexpr size_t tc_smem_bytes() { return size_t(TcForm<FORM>::kStages) * TcForm<FORM>::kTiles * kTileBytes + 1024 + 256; }
constexpr int kEpiWarps = 16;                     // four per TMEM lane quarter, 32 columns each
constexpr int kTcThreads = 64 + 32 * kEpiWarps;
constexpr uint64_t kWaitNs = 1000000000ull;       // bounded mbarrier waits: 1 s
constexpr uint64_t kTcChunkRows = 16384;          // rows split and hashed per launch

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait: false if the phase has not completed within limit_ns
// (0: a single try).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns = kWaitNs)
{
    if (mbar_try_wait(bar, parity)) return true;
    if (limit_ns == 0) return false;
    const uint64_t t0 = global_ns();
    for (;;) {
        for (int i = 0; i < 256; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > limit_ns) return false;
    }
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= uint64_t((addr & 0x3FFFFu) >> 4);
    d |= uint64_t(1) << 16;                 // leading byte offset (unused with 128B swizzle, K-major)
    d |= uint64_t(1024 >> 4) << 32;         // stride byte offset
    d |= uint64_t(1) << 46;                 // version
    d |= uint64_t(2) << 61;                 // 128-byte swizzle
    return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B bf16, both K-major,
// M = 128 rows, N columns.
template <int N>
__host__ __device__ constexpr uint32_t mma_idesc()
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(N >> 3) << 17) | (uint32_t(kTM >> 4) << 24);
}

template <int N>
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(mma_idesc<N>()), "r"(accumulate)
        : "memory");
}

// Instruction descriptor, kind::f8f6f4: D fp32, A and B E4M3 (format 0), both
// K-major, M = 128 rows, N columns.
template <int N>
__host__ __device__ constexpr uint32_t mma_idesc_e4m3()
{
    return (1u << 4) | (uint32_t(N >> 3) << 17) | (uint32_t(kTM >> 4) << 24);
}

template <int N>
__device__ __forceinline__ void mma_e4m3(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(mma_idesc_e4m3<N>()), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(smem_u32(bar)) : "memory");
}

// N consecutive fp32 columns of this warp's 32 TMEM lanes; the caller waits
// (tmem_wait_ld) before reading the registers.
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld()
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

struct TcArgs {
    uint64_t n;            // rows (points) in this launch
    uint32_t P, d, L, K;
    const float *xnorm;    // n: upper bounds of ||x||
    const float *wnorm;    // P: upper bounds of ||w||
    const float *xres;     // n upper bounds of ||x - s_x xq|| (the split: of ||x - x1||)
    const float *wres;     // P upper bounds of ||w - s_w wq|| (||w - w1||)
    const float *xscale;   // FP8: n row scales s_x (powers of two)
    const float *wscale;   // FP8: P row scales s_w
    float c_norm;          // margin factor on ||x|| ||w||
    float c_one;           // MASK = 3: that of the first pass
    float c_sub;           // margin factor on ||x|| + ||w|| (subnormal flushes)
    float tiny;            // absolute margin (underflow)
    uint32_t *codes;       // n x L (zeroed)
    float *proj;           // optional n x P
    unsigned long long *rlist;
    unsigned long long *rcount;
    uint32_t *mask;        // dense second pass: per row ceil(P / 32) words of undecided projections, then as
                           // many of their first-pass signs
    unsigned long long *nund;    // masks written: undecided projections
    unsigned long long *stats;   // masks read: the hash counters
    uint32_t *err;         // set to 1 on a wait timeout
    uint64_t wait_ns;      // limit of the pipeline's waits (the drains after an abort keep kWaitNs)
};

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// MASK: 0 undecided projections are listed; 1 they are marked in a.mask (the
// first pass of the FP8 form whose undecided share is large); 2 only the marked
// ones are decided (its second pass, on the two-term split), the rest listed; 3
// both passes of the BF16 form at once, whose first pass is the split's x1 w1
// half: the sums of that half are kept beside the full ones (64 accumulators a
// thread), so the second pass costs the
// split's two extra MMAs per step and no second reading of the operands.
template <int FORM, int MASK>
__global__ void __launch_bounds__(kTcThreads, 1)
k_srp_tc(const __grid_constant__ CUtensorMap mx1, const __grid_constant__ CUtensorMap mx2,
         const __grid_constant__ CUtensorMap mw1, const __grid_constant__ CUtensorMap mw2, TcArgs a)
{
    using F = TcForm<FORM>;
    constexpr int kStages = F::kStages;
    constexpr int kStageBytes = F::kTiles * kTileBytes;
    constexpr int kW = F::kTiles / 2;                 // tile index of the first W tile in a stage
    constexpr uint32_t kBuf = F::kTmemCols / 2;        // TMEM columns per buffer
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    // 1024-byte aligned tile ring, then barriers and the TMEM address
    unsigned char *ring = tc_smem + ((1024u - (smem_u32(tc_smem) & 1023u)) & 1023u);
    uint64_t *full = reinterpret_cast<uint64_t *>(ring + kStages * kStageBytes);
    uint64_t *empty = full + kStages;        // stage consumed by the MMAs
    uint64_t *tfull = empty + kStages;       // TMEM buffer b holds a finished k-block
    uint64_t *tempty = tfull + 2;            // TMEM buffer b drained by the epilogue
    uint64_t *mdone = tempty + 2;            // every MMA issued has completed
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mdone + 1);
    uint32_t *abort_flag = tmem_slot + 1;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // projection blocks vary fastest: the CTAs that share one X tile run in
    // the same wave, so X is read from DRAM once and W stays in L2
    const uint32_t row0 = blockIdx.y * kTM, col0 = blockIdx.x * kTN;
    const uint32_t nkb = (a.d + F::kKElems - 1) / F::kKElems;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&tfull[b], 1);
            mbar_init(&tempty[b], kEpiWarps);
        }
        mbar_init(mdone, 1);
        *abort_flag = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(F::kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    uint32_t issued = 0;   // producer: k-blocks whose copies were issued
    if (warp == 0) {
        if (lane == 0) {
            for (uint32_t kb = 0; kb < nkb; ++kb) {
                const int s = kb % kStages;
                if (kb >= uint32_t(kStages) && !mbar_wait(&empty[s], ((kb / kStages) - 1) & 1, a.wait_ns)) {
                    atomicExch(abort_flag, 1u);
                    break;
                }
                if (*(volatile uint32_t *)abort_flag) break;
                unsigned char *st = ring + s * kStageBytes;
                mbar_expect_tx(&full[s], kStageBytes);
                const int kx = int(kb * F::kKElems);
                tma_load_2d(st + 0 * kTileBytes, &mx1, &full[s], kx, int(row0));
                if constexpr (F::kTiles == 4) tma_load_2d(st + 1 * kTileBytes, &mx2, &full[s], kx, int(row0));
                tma_load_2d(st + kW * kTileBytes, &mw1, &full[s], kx, int(col0));
                if constexpr (F::kTiles == 4) tma_load_2d(st + 3 * kTileBytes, &mw2, &full[s], kx, int(col0));
                issued = kb + 1;
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            for (uint32_t kb = 0; kb < nkb; ++kb) {
                const int s = kb % kStages;
                const uint32_t b = kb & 1u;
                if (!mbar_wait(&full[s], (kb / kStages) & 1, a.wait_ns) ||
                    (kb >= 2 && !mbar_wait(&tempty[b], ((kb >> 1) - 1) & 1, a.wait_ns))) {
                    atomicExch(abort_flag, 1u);
                    break;
                }
                if (*(volatile uint32_t *)abort_flag) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t st = smem_u32(ring + s * kStageBytes);
                const uint32_t t_hi = tmem + kBuf * b;
                // four 32-byte K steps per 128-byte stage row: 16 bf16 or 32 e4m3
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t off = kk * 32;
                    const uint32_t acc = kk > 0 ? 1u : 0u;     // each k-block starts a fresh accumulator
                    if constexpr (FORM == kFormBf16x2) {
                        // W1 and W2 tiles are adjacent in the stage, so [W1; W2] is one
                        // 256-row B operand: x1 [w1 w2] fills hi and lo in one MMA
                        // (N = 256), then x2 w1 adds into lo (N = 128)
                        const uint64_t x1 = smem_desc(st + 0 * kTileBytes + off);
                        const uint64_t x2 = smem_desc(st + 1 * kTileBytes + off);
                        const uint64_t w12 = smem_desc(st + 2 * kTileBytes + off);
                        mma_bf16<2 * kTN>(t_hi, x1, w12, acc);
                        mma_bf16<kTN>(t_hi + kTN, x2, w12, 1u);
                    } else {
                        const uint64_t xd = smem_desc(st + off);
                        const uint64_t wd = smem_desc(st + kTileBytes + off);
                        if constexpr (FORM == kFormBf16) mma_bf16<kTN>(t_hi, xd, wd, acc);
                        else mma_e4m3<kTN>(t_hi, xd, wd, acc);
                    }
                }
                mma_commit(&empty[s]);
                mma_commit(&tfull[b]);
            }
            mma_commit(mdone);     // arrives once every MMA issued above has completed
        }
    } else {
        // epilogue: TMEM lanes [32 (warp % 4), +32) = one point per thread;
        // columns [32 group, +32) of the tile. Each warp's drain of a k-block is a
        // chain (barrier, TMEM loads, adds): four warps per scheduler overlap theirs
        // and add in pairs. With two (64 columns each) and single adds it took 1.03
        // us a k-block in the two-term form and 1.49 with both passes' sums, against
        // 0.61 for operands and MMAs alone; now 0.68 and 0.70 (0.77 and 0.86 with
        // single adds). 10,000 rows of 4,096: 329 -> 268 us, 8,192 in BF16: 374 -> 228.
        const uint32_t quarter = (warp & 3) * 32;
        const uint32_t group = uint32_t(warp - 2) >> 2;
        const uint32_t tbase = tmem + (quarter << 16) + 32u * group;
        float acc[32];
        float one[MASK == 3 ? 32 : 1];       // the first pass's sums
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = 0.f;
#pragma unroll
        for (int j = 0; j < (MASK == 3 ? 32 : 1); ++j) one[j] = 0.f;
        bool abort = false;
        for (uint32_t kb = 0; kb < nkb; ++kb) {
            const uint32_t b = kb & 1u;
            uint32_t got = 0;
            if (lane == 0) got = mbar_wait(&tfull[b], (kb >> 1) & 1, a.wait_ns) ? 1u : 0u;
            got = __shfl_sync(0xffffffffu, got, 0);
            if (!got) {
                if (lane == 0) atomicExch(abort_flag, 1u);
                abort = true;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // kIn columns in flight: 96 registers a thread (five warps on a scheduler)
            // hold no more beside the accumulators. The buffer goes back to the MMA
            // issuer before its last values are added.
            constexpr int kIn = MASK == 3 ? 8 : FORM == kFormBf16x2 ? 16 : 32;
#pragma unroll
            for (int q = 0; q < 32; q += kIn) {
                uint32_t hv[kIn], lv[kIn];
                tmem_ld(tbase + kBuf * b + q, hv);
                if constexpr (FORM == kFormBf16x2) tmem_ld(tbase + kBuf * b + kTN + q, lv);
                tmem_wait_ld();
                if (q + kIn == 32) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&tempty[b]);
                }
#pragma unroll
                for (int j = 0; j < kIn; j += 2) {
                    float2 h = make_float2(__uint_as_float(hv[j]), __uint_as_float(hv[j + 1])), t = h;
                    if constexpr (FORM == kFormBf16x2)
                        t = __fadd2_rn(h, make_float2(__uint_as_float(lv[j]), __uint_as_float(lv[j + 1])));
                    t = __fadd2_rn(make_float2(acc[q + j], acc[q + j + 1]), t);
                    acc[q + j] = t.x;
                    acc[q + j + 1] = t.y;
                    if constexpr (MASK == 3) {
                        h = __fadd2_rn(make_float2(one[q + j], one[q + j + 1]), h);
                        one[q + j] = h.x;
                        one[q + j + 1] = h.y;
                    }
                }
            }
        }
        uint32_t ab = lane == 0 ? *(volatile uint32_t *)abort_flag : 0u;
        abort = abort || __shfl_sync(0xffffffffu, ab, 0) != 0u;    // warp-uniform
        const uint64_t row = uint64_t(row0) + quarter + lane;
        // bits by column: undecided, first-pass signs
        uint32_t und = 0u, sgn = 0u, decided = 0u, flips = 0u, open = 0u;
        const uint32_t cbase = col0 + 32u * group;
        if (!abort && row < a.n) {
            const float xn = a.xnorm[row], xr = a.xres[row];
            float xs = 1.f;
            if constexpr (FORM == kFormFp8) xs = a.xscale[row];
            uint32_t cur_l = 0xFFFFFFFFu, cur_bits = 0u;
            // this thread's word of the masks
            const uint32_t pw = (a.P + 31) / 32, w0 = cbase / 32;
            uint32_t *mrow = MASK == 1 || MASK == 2 ? a.mask + row * (2 * pw) + w0 : nullptr;
            uint32_t todo = 0xFFFFFFFFu, first = 0u;
            if constexpr (MASK == 2) {
                todo = w0 < pw ? mrow[0] : 0u;
                first = w0 < pw ? mrow[pw] : 0u;
            }
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const uint32_t col = cbase + j;
                if (col >= a.P) break;
                if (MASK == 2 && !((todo >> j) & 1u)) continue;
                float p = acc[j];
                if constexpr (FORM == kFormFp8) p *= xs * __ldg(a.wscale + col);    // powers of two: exact
                const float wn = __ldg(a.wnorm + col), wr = __ldg(a.wres + col);
                if (a.proj) a.proj[row * a.P + col] = MASK == 3 ? one[MASK == 3 ? j : 0] : p;
                // residual term (Cauchy-Schwarz on the quantisation errors) plus
                // accumulation on the quantised operands' norms, then slack
                auto single_margin = [&](float v, float c) {
                    const float resid = fmaf(xn, wr, fmaf(xr, wn, 3.f * xr * wr));
                    const float accum = c * (xn + xr) * (wn + wr);
                    return (resid + accum + fmaf(ldexpf(1.f, -23), fabsf(v), fmaf(a.c_sub, xn + wn, a.tiny))) *
                           (1.f + ldexpf(1.f, -20));
                };
                bool first_pos = p > 0.f, again = MASK == 2;       // again: this is a second look
                float margin;
                if constexpr (FORM == kFormBf16x2) {
                    const float split = fmaf(0x1p-8f, fmaf(xn, wr, xr * wn), (1.f + 0x1p-6f) * xr * wr);
                    margin = fmaf(a.c_norm * xn, wn, fmaf(ldexpf(1.f, -23), fabsf(p), fmaf(a.c_sub, xn + wn, a.tiny)));
                    margin = (margin + split) * (1.f + ldexpf(1.f, -20));
                } else {
                    margin = single_margin(p, a.c_norm);
                }
                if constexpr (MASK == 2) first_pos = ((first >> j) & 1u) != 0u;
                if constexpr (MASK == 3) {
                    const float v = one[j];
                    first_pos = v > 0.f;
                    again = !(fabsf(v) > single_margin(v, a.c_one));
                    if (again) ++open;
                    else p = v, margin = 0.f;                    // decided by the first pass (|v| > 0)
                }
                if (fabsf(p) > margin) {
                    if (MASK >= 2 && again) {
                        ++decided;
                        flips += (p > 0.f) != first_pos ? 1u : 0u;
                    }
                    if (p > 0.f) {
                        const uint32_t l = col / a.K;
                        if (l != cur_l) {
                            if (cur_bits) atomicOr(&a.codes[row * a.L + cur_l], cur_bits);
                            cur_l = l;
                            cur_bits = 0u;
                        }
                        cur_bits |= 1u << (col % a.K);
                    }
                } else {
                    // the tentative sign a later re-check may reverse is the first pass's
                    und |= 1u << j;
                    if (first_pos) sgn |= 1u << j;
                }
            }
            if (cur_bits) atomicOr(&a.codes[row * a.L + cur_l], cur_bits);
            if constexpr (MASK == 1) {
                if (w0 < pw) {
                    mrow[0] = und;
                    mrow[pw] = sgn;
                }
            }
        }
        // lists and counters: one atomic a warp. One per undecided projection
        // and per thread, all on a few words, were 10 us of a wave of tiles in the
        // two-term form and 31 us in the BF16 form's.
        const uint32_t c = __popc(und);
        if constexpr (MASK == 1) {
            const uint32_t all = __reduce_add_sync(0xffffffffu, c);
            if (all && lane == 0) atomicAdd(a.nund, (unsigned long long)all);
        } else if (__any_sync(0xffffffffu, c != 0u)) {
            uint32_t incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, incl, d);
                if (lane >= d) incl += y;
            }
            unsigned long long at = 0;
            if (lane == 31) at = atomicAdd(a.rcount, (unsigned long long)incl);
            at = __shfl_sync(0xffffffffu, at, 31) + (incl - c);
            for (uint32_t m = und; m; m &= m - 1u) {
                const uint32_t j = __ffs(m) - 1;
                a.rlist[at++] = ((sgn >> j) & 1u ? kEntSign : 0ull) | ((unsigned long long)row << 20) | (cbase + j);
            }
        }
        if constexpr (MASK == 3) {
            open = __reduce_add_sync(0xffffffffu, open);
            if (open && lane == 0) atomicAdd(a.nund, (unsigned long long)open);
        }
        if constexpr (MASK >= 2) {
            decided = __reduce_add_sync(0xffffffffu, decided);
            flips = __reduce_add_sync(0xffffffffu, flips);
            if (decided && lane == 0) atomicAdd(&a.stats[3], (unsigned long long)decided);
            if (flips && lane == 0) atomicAdd(&a.stats[4], (unsigned long long)flips);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*(volatile uint32_t *)abort_flag) {
        if (threadIdx.x == 0) atomicExch(a.err, 1u);
        // let the copies this CTA issued land before its shared memory goes away
        if (warp == 0 && lane == 0) {
            for (uint32_t kb = (issued > uint32_t(kStages) ? issued - kStages : 0); kb < issued; ++kb)
                mbar_wait(&full[kb % kStages], (kb / kStages) & 1, kWaitNs);
        }
    }
    if (warp == 1) {
        // every MMA has completed before the columns are freed
        if (lane == 0) mbar_wait(mdone, 0, kWaitNs);
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(F::kTmemCols) : "memory");
    }
    __syncthreads();
}

// Upper bounds of a row's norm and of its residual's norm, by one warp, from
// the lanes' fp32 sums of squares (at most m roundings each). The residuals are
// exact in fp32 (a float minus its rounding to fewer bits); squares lost to
// underflow are covered by the range check for the row and by an absolute term
// for the residual. Out of range (values near 1e18 or 1e-14 alone): fp64.
template <class Residual>
__device__ __forceinline__ void row_bounds(float ss, float rr, bool any, const float *xr, uint32_t d, Residual res_of,
                                           float *norm, float *res)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
        rr += __shfl_xor_sync(0xffffffffu, rr, o);
    }
    any = __any_sync(0xffffffffu, any);
    if (norm_in_range(ss, any)) {
        *norm = norm_up(ss, d / 32 + 16);
        *res = norm_up(__fadd_ru(rr, any ? float(d) * 0x1p-148f : 0.f), d / 32 + 16);
        return;
    }
    double s64 = 0.0, r64 = 0.0;
    for (uint32_t t = lane; t < d; t += 32) {
        const double v = xr[t], e = res_of(xr[t]);
        s64 += v * v;
        r64 += e * e;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s64 += __shfl_xor_sync(0xffffffffu, s64, o);
        r64 += __shfl_xor_sync(0xffffffffu, r64, o);
    }
    *norm = norm_up64(s64);
    *res = norm_up64(r64);
}

__device__ __forceinline__ uint2 pack_bf16x4(__nv_bfloat16 a, __nv_bfloat16 b, __nv_bfloat16 c, __nv_bfloat16 d)
{
    return make_uint2(uint32_t(__bfloat16_as_ushort(a)) | uint32_t(__bfloat16_as_ushort(b)) << 16,
                      uint32_t(__bfloat16_as_ushort(c)) | uint32_t(__bfloat16_as_ushort(d)) << 16);
}

// x -> x1 = bf16(x) and, TWO, x2 = bf16(x - x1); upper bounds of each row's
// norm and of ||x - x1||. A warp per row, four floats per lane and step (d is a
// multiple of 8, so the 8-byte stores are aligned). Bound by the bytes: 10^4
// rows of 4,096 split in 178 us with fp64 sums of squares (the FP64 pipe's
// rate) and 4-byte loads, in 52 us (6.3 TB/s) now.
template <bool VEC, bool TWO>
__global__ void k_split_rows(const float *__restrict__ x, uint64_t ld, uint64_t n, uint32_t d,
                             __nv_bfloat16 *__restrict__ x1, __nv_bfloat16 *__restrict__ x2,
                             float *__restrict__ norm, float *__restrict__ res)
{
    const int lane = threadIdx.x & 31;
    const uint64_t gw = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t r = gw; r < n; r += nw) {
        const float *xr = x + r * ld;
        float ss = 0.f, rr = 0.f;
        bool any = false;
#pragma unroll 4
        for (uint32_t t = lane * 4; t < d; t += 128) {
            const float4 q = load4<VEC>(xr, t, d, true);
            const float v[4] = {q.x, q.y, q.z, q.w};
            __nv_bfloat16 h[4], l[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                h[i] = __float2bfloat16_rn(v[i]);
                const float e = v[i] - __bfloat162float(h[i]);
                l[i] = __float2bfloat16_rn(e);
                ss = fmaf(v[i], v[i], ss);
                rr = fmaf(e, e, rr);
                any |= v[i] != 0.f;
            }
            *reinterpret_cast<uint2 *>(x1 + r * d + t) = pack_bf16x4(h[0], h[1], h[2], h[3]);
            if constexpr (TWO) *reinterpret_cast<uint2 *>(x2 + r * d + t) = pack_bf16x4(l[0], l[1], l[2], l[3]);
        }
        float nrm, rn;
        row_bounds(ss, rr, any, xr, d,
                   [](float v) { return double(v) - double(__bfloat162float(__float2bfloat16_rn(v))); }, &nrm, &rn);
        if (lane == 0) {
            norm[r] = nrm;
            if (res) res[r] = rn;
        }
    }
}

// E4M3 rows: q = e4m3(x / s) with s = 2^e, e the smallest with max |x| / s < 448
// (a value whose quantised magnitude would be below 2^-6, an E4M3 subnormal,
// becomes 0). Per row: upper bounds of ||x|| and of ||x - s q||, and s.
template <bool VEC>
__global__ void k_quant_rows(const float *__restrict__ x, uint64_t ld, uint64_t n, uint32_t d,
                             __nv_fp8_e4m3 *__restrict__ q, float *__restrict__ norm, float *__restrict__ res,
                             float *__restrict__ scale)
{
    const int lane = threadIdx.x & 31;
    const uint64_t gw = (uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const uint64_t nw = (uint64_t(gridDim.x) * blockDim.x) >> 5;
    for (uint64_t r = gw; r < n; r += nw) {
        const float *xr = x + r * ld;
        float mx = 0.f;
#pragma unroll 4
        for (uint32_t t = lane * 4; t < d; t += 128) {
            const float4 v = load4<VEC>(xr, t, d, true);
            mx = fmaxf(mx, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float s = 1.f;
        if (mx > 0.f) {
            int e;
            frexpf(mx / 448.f, &e);      // mx / 448 = f 2^e with f in [0.5, 1): mx / 2^e < 448
            s = ldexpf(1.f, e);
        }
        auto quant = [&](float v) {
            __nv_fp8_e4m3 h(v / s);                       // round to nearest, saturating
            if (fabsf(float(h)) < 0x1p-6f) h = __nv_fp8_e4m3(0.f);
            return h;
        };
        float ss = 0.f, rr = 0.f;
#pragma unroll 2
        for (uint32_t t = lane * 4; t < d; t += 128) {
            const float4 v4 = load4<VEC>(xr, t, d, true);
            const float v[4] = {v4.x, v4.y, v4.z, v4.w};
            uint32_t w = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const __nv_fp8_e4m3 h = quant(v[i]);
                w |= uint32_t(h.__x) << (8 * i);
                const float e = v[i] - float(h) * s;      // exact: s is a power of two
                ss = fmaf(v[i], v[i], ss);
                rr = fmaf(e, e, rr);
            }
            *reinterpret_cast<uint32_t *>(q + r * d + t) = w;
        }
        float nrm, rn;
        row_bounds(ss, rr, mx > 0.f, xr, d, [&](float v) { return double(v) - double(float(quant(v)) * s); }, &nrm, &rn);
        if (lane == 0) {
            norm[r] = nrm;
            res[r] = rn;
            scale[r] = s;
        }
    }
}

// Compensated fp32 re-check of listed projections: two-product and two-sum
// per term (one warp per projection), error at most 2^-23 |p| + 2 g(2d)^2 S
// with S = sum |w x|, in any order of the sums. Decided bits are set; the rest
// go to the next list. xr: the entry's row of x (global or shared memory). The
// rows of W are 16-byte aligned (d % 8 == 0).
template <bool VEC>
__device__ __forceinline__ void recheck2_entry(const float *xr, const float *__restrict__ Wm, uint32_t d,
                                               uint32_t L, uint32_t K, float g2, float tiny, unsigned long long ent,
                                               uint32_t *__restrict__ codes, unsigned long long *__restrict__ out_list,
                                               unsigned long long *__restrict__ out_count,
                                               unsigned long long *__restrict__ stats)
{
    const int lane = threadIdx.x & 31;
    const uint64_t gr = ent_row(ent);
    const uint32_t gc = ent_col(ent);
    const float *wr = Wm + uint64_t(gc) * d;
    // four compensated sums per lane (one per component of a 16-byte load): four
    // independent chains of two-sums
    float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f}, sa = 0.f;
    auto add = [&](float &sum, float &comp, float h, float l) {
        const float sn = sum + h;                   // two-sum
        const float z = sn - sum;
        comp += (sum - (sn - z)) + (h - z) + l;
        sum = sn;
    };
#pragma unroll 2
    for (uint32_t t = lane * 4; t < d; t += 128) {
        float xv[4];                                  // xr may be shared memory: plain loads
        if constexpr (VEC) {
            const float4 x4 = *reinterpret_cast<const float4 *>(xr + t);
            xv[0] = x4.x;
            xv[1] = x4.y;
            xv[2] = x4.z;
            xv[3] = x4.w;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) xv[i] = xr[t + i];
        }
        const float4 w4 = load4<true>(wr, t, d, true);
        const float wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float h = xv[i] * wv[i];
            add(s[i], c[i], h, fmaf(xv[i], wv[i], -h));       // exact product error
            sa = fmaf(fabsf(xv[i]), fabsf(wv[i]), sa);
        }
    }
#pragma unroll
    for (int i = 1; i < 4; ++i) add(s[0], c[0], s[i], c[i]);
    // combine the lanes, halving: each pair by a two-sum
    float ts = s[0], tc = c[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float so = __shfl_down_sync(0xffffffffu, ts, o), co = __shfl_down_sync(0xffffffffu, tc, o);
        add(ts, tc, so, co);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sa += __shfl_xor_sync(0xffffffffu, sa, o);
    sa = __shfl_sync(0xffffffffu, sa, 0);
    const float p = ts + tc;
    const float margin = fmaf(ldexpf(1.f, -23), fabsf(p), fmaf(g2, sa, tiny));
    if (lane == 0) {
        if (fabsf(p) > margin) {
            if (p > 0.f) atomicOr(&codes[gr * L + gc / K], 1u << (gc % K));
            if ((p > 0.f) != ((ent & kEntSign) != 0)) atomicAdd(&stats[4], 1ull);
        } else {
            out_list[atomicAdd(out_count, 1ull)] = ent;
        }
        atomicAdd(&stats[3], 1ull);
    }
}

template <bool VEC>
__global__ void __launch_bounds__(256) k_srp_recheck2(const float *__restrict__ X, uint64_t ldx, const float *__restrict__ Wm, uint32_t d,
                               uint32_t L, uint32_t K, float g2, float tiny,
                               const unsigned long long *__restrict__ rlist,
                               const unsigned long long *__restrict__ rcount, uint32_t *__restrict__ codes,
                               unsigned long long *__restrict__ out_list, unsigned long long *__restrict__ out_count,
                               unsigned long long *__restrict__ stats)
{
    const unsigned long long nlist = *rcount;
    const unsigned long long nwarps = (unsigned long long)gridDim.x * (blockDim.x >> 5);
    for (unsigned long long e = (unsigned long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
         e < nlist; e += nwarps) {
        const unsigned long long ent = rlist[e];
        recheck2_entry<VEC>(X + ent_row(ent) * ldx, Wm, d, L, K, g2, tiny, ent, codes, out_list, out_count, stats);
    }
}

// The listed projections grouped by row (a counting sort on the row), so that
// the re-check stages each row of x once in shared memory for all of its
// entries (the tensor-core epilogue lists a row's projections far apart).
__global__ void k_rows_hist(const unsigned long long *__restrict__ rlist, const unsigned long long *__restrict__ rcount,
                            uint32_t *__restrict__ rowcnt)
{
    const unsigned long long n = *rcount;
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (unsigned long long)gridDim.x * blockDim.x)
        atomicAdd(&rowcnt[ent_row(rlist[e])], 1u);
}

__global__ void k_rows_scatter(const unsigned long long *__restrict__ rlist,
                               const unsigned long long *__restrict__ rcount, const uint32_t *__restrict__ rowoff,
                               uint32_t *__restrict__ fill, unsigned long long *__restrict__ sorted)
{
    const unsigned long long n = *rcount;
    for (unsigned long long e = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
         e += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long ent = rlist[e];
        const uint64_t r = ent_row(ent);
        sorted[rowoff[r] + atomicAdd(&fill[r], 1u)] = ent;
    }
}

// A CTA per row with listed entries: the row of x in shared memory, a warp per
// entry; the same arithmetic, in the same order, as k_srp_recheck2.
__global__ void k_srp_recheck2_rows(const float *__restrict__ X, uint64_t ldx, const float *__restrict__ Wm,
                                    uint32_t d, uint32_t L, uint32_t K, float g2, float tiny, uint32_t rows,
                                    const unsigned long long *__restrict__ sorted, const uint32_t *__restrict__ rowoff,
                                    uint32_t *__restrict__ codes, unsigned long long *__restrict__ out_list,
                                    unsigned long long *__restrict__ out_count, unsigned long long *__restrict__ stats)
{
    extern __shared__ __align__(16) float xs[];
    const uint32_t warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (uint32_t r = blockIdx.x; r < rows; r += gridDim.x) {
        const uint32_t e0 = rowoff[r], e1 = rowoff[r + 1];
        if (e0 == e1) continue;                       // uniform over the CTA
        const float *xg = X + uint64_t(r) * ldx;
        for (uint32_t t = threadIdx.x; t < d; t += blockDim.x) xs[t] = xg[t];
        __syncthreads();
        for (uint32_t e = e0 + warp; e < e1; e += nw)
            recheck2_entry<true>(xs, Wm, d, L, K, g2, tiny, sorted[e], codes, out_list, out_count, stats);
        __syncthreads();                              // before the next row overwrites xs
    }
}

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

int get_encoder(EncodeTiled *fn)
{
    static EncodeTiled cached = nullptr;
    if (!cached) {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        FL_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
        if (!p || q != cudaDriverEntryPointSuccess)
            return set_error(FLINNG_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
        cached = reinterpret_cast<EncodeTiled>(p);
    }
    *fn = cached;
    return FLINNG_OK;
}

// 2-D map over rows x d (d contiguous, row stride d elements) of bf16 or
// 8-bit elements; the box is 128 bytes (64 bf16 or 128 e4m3) x 128 rows.
int make_map(CUtensorMap *m, const void *base, uint64_t rows, uint32_t d, bool bytes)
{
    EncodeTiled enc = nullptr;
    FL_TRY(get_encoder(&enc));
    const uint32_t esz = bytes ? 1u : 2u;
    const cuuint64_t dims[2] = {d, rows};
    const cuuint64_t strides[1] = {uint64_t(d) * esz};
    const cuuint32_t box[2] = {128u / esz, uint32_t(kTM)};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = enc(m, bytes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                           const_cast<void *>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return set_error(FLINNG_ERR_INVALID_ARG, "tensor map: error %d (d=%u)", int(r), d);
    return FLINNG_OK;
}

inline unsigned warp_grid(uint64_t items)
{
    uint64_t b = (items * 32 + 255) / 256;
    if (b > 152ull * 32) b = 152ull * 32;
    return (unsigned)(b ? b : 1);
}

// bytes of one quantised row
inline size_t qrow_bytes(uint32_t precision, uint32_t d)
{
    return precision == FLINNG_PREC_BF16X2 ? size_t(d) * 4 : precision == FLINNG_PREC_BF16 ? size_t(d) * 2 : size_t(d);
}

// A single-term form leaves a share of the projections undecided that grows
// with its residual norms (about a sixth at d = 4096 in BF16, nearly all in
// FP8). Re-checked one by one, each streams its row of W from L2 (2.3 ns per
// projection at d = 4096 with every SM busy, more for a batch of a few rows); a
// dense second pass on the two-term split costs 0.05 ns per projection of a large
// batch, decided or not, and no more than a tile's depth for a small one, so it
// wins from an undecided share of about 2 %: d >= 128 in BF16, any d in FP8.
// 8,192 embeddings in BF16: 4.04 ms re-checked one by one, 0.37 ms with both
// passes in one kernel (MASK = 3); 97 of them 280 against 108 us, in FP8 1,043
// against 158 (128 dimensions, 256 projections: 61 against 45, 77 against 65).
inline bool dense_second_pass(uint32_t precision, uint32_t d)
{
    return precision == FLINNG_PREC_FP8 || (precision == FLINNG_PREC_BF16 && d >= 128);
}

// two: also x2 behind x1 (the BF16 form's second pass)
int quant_rows(uint32_t precision, const float *x, uint64_t ld, uint64_t n, uint32_t d, void *q, float *norm,
               float *res, float *scale, bool two, cudaStream_t st)
{
    const bool vec = rows_vec4(x, ld, d);
    const unsigned grid = warp_grid(n);
    if (precision != FLINNG_PREC_FP8) {
        __nv_bfloat16 *q1 = static_cast<__nv_bfloat16 *>(q);
        auto fn = two ? (vec ? k_split_rows<true, true> : k_split_rows<false, true>)
                      : (vec ? k_split_rows<true, false> : k_split_rows<false, false>);
        fn<<<grid, 256, 0, st>>>(x, ld, n, d, q1, q1 + n * d, norm, res);
    } else {
        auto fn = vec ? k_quant_rows<true> : k_quant_rows<false>;
        fn<<<grid, 256, 0, st>>>(x, ld, n, d, static_cast<__nv_fp8_e4m3 *>(q), norm, res, scale);
    }
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

template <int FORM, int MASK>
int launch_tc(const CUtensorMap &mx1, const CUtensorMap &mx2, const CUtensorMap &mw1, const CUtensorMap &mw2,
              const TcArgs &a, uint64_t rows, cudaStream_t st)
{
    const size_t smem = tc_smem_bytes<FORM>();
    FL_TRY(ensure_dyn_smem((const void *)k_srp_tc<FORM, MASK>, smem));
    dim3 grid((a.P + kTN - 1) / kTN, (unsigned)((rows + kTM - 1) / kTM));
    k_srp_tc<FORM, MASK><<<grid, kTcThreads, smem, st>>>(mx1, mx2, mw1, mw2, a);
    count_launch();
    FL_CUDA(cudaGetLastError());
    return FLINNG_OK;
}

}  // namespace

int srp_tc_prepare_weights(flinng_index *ix)
{
    const uint32_t P = ix->P, d = ix->cfg.dim, prec = ix->cfg.precision;
    if (d % (prec == FLINNG_PREC_FP8 ? 16 : 8) != 0)
        return set_error(FLINNG_ERR_INVALID_ARG, "tensor-core SRP: dim %u is not a multiple of %d", d,
                         prec == FLINNG_PREC_FP8 ? 16 : 8);
    // the single-term forms also keep the two-term split, for the dense second pass
    const size_t split = size_t(P) * d * 4, qb = prec == FLINNG_PREC_FP8 ? split + size_t(P) * d : split;
    FL_CUDA(cudaMalloc(&ix->w_split, qb));
    ix->device_bytes += qb;
    // residual norms of the split, then for FP8 those of its rows and their scales
    const size_t aux = size_t(P) * (prec == FLINNG_PREC_FP8 ? 3 : 1);
    FL_CUDA(cudaMalloc(&ix->w_aux, aux * sizeof(float)));
    ix->device_bytes += aux * sizeof(float);
    FL_TRY(quant_rows(FLINNG_PREC_BF16X2, ix->srp_w, d, P, d, ix->w_split, ix->w_norm, ix->w_aux, nullptr, true,
                      ix->stream));
    if (prec != FLINNG_PREC_FP8) return FLINNG_OK;
    return quant_rows(prec, ix->srp_w, d, P, d, static_cast<char *>(ix->w_split) + split, ix->w_norm, ix->w_aux + P,
                      ix->w_aux + 2 * P, false, ix->stream);
}

// bytes per row of the quantised x: the two-term split where a second pass needs it
static size_t x_bytes(const flinng_index *ix)
{
    return dense_second_pass(ix->cfg.precision, ix->cfg.dim) ? size_t(ix->cfg.dim) * 4
                                                             : qrow_bytes(ix->cfg.precision, ix->cfg.dim);
}

size_t srp_tc_workspace_bytes(const flinng_index *ix, uint64_t n)
{
    const uint64_t rows = n < kTcChunkRows ? n : kTcChunkRows;
    return carve_bytes<char>(rows * x_bytes(ix)) + 3 * carve_bytes<float>(rows) +
           carve_bytes<unsigned long long>(8) + 2 * carve_bytes<unsigned long long>(rows * ix->P + 1) +
           3 * carve_bytes<uint32_t>(rows + 1) + carve_bytes<char>(scan_workspace_bytes(rows + 1)) + 4096;
}

// The same with the rows quantised in the form's own width: what a caller with a
// fixed scratch needs (srp_hash_tc takes as many rows at a time as fit).
size_t srp_tc_least_bytes(const flinng_index *ix, uint64_t n)
{
    const uint64_t rows = n < kTcChunkRows ? n : kTcChunkRows;
    return srp_tc_workspace_bytes(ix, n) - carve_bytes<char>(rows * x_bytes(ix)) +
           carve_bytes<char>(rows * qrow_bytes(ix->cfg.precision, ix->cfg.dim));
}

// Codes of n rows of x (stride ld) on the tensor cores; same contract as srp_hash.
int srp_hash_tc(flinng_index *ix, const float *x, uint64_t ld, uint64_t n, uint32_t *buckets, float *proj,
                void *ws, size_t ws_bytes)
{
    // a wait that timed out in an earlier call (the flag is sticky on the device)
    if (ix->h_flag[3]) return set_error(FLINNG_ERR_TIMEOUT, "tensor-core SRP: a pipeline wait timed out");
    const cudaStream_t st = ix->stream;
    const uint32_t L = ix->cfg.L, K = ix->cfg.K, d = ix->cfg.dim, P = ix->P, prec = ix->cfg.precision;
    const bool bytes = prec == FLINNG_PREC_FP8;
    uint64_t cap = n < kTcChunkRows ? n : kTcChunkRows;     // rows that the workspace holds
    if (srp_tc_workspace_bytes(ix, cap) > ws_bytes) {
        uint64_t lo = 1;
        while (lo < cap) {
            const uint64_t mid = (lo + cap + 1) / 2;
            if (srp_tc_workspace_bytes(ix, mid) <= ws_bytes) lo = mid;
            else cap = mid - 1;
        }
        if (srp_tc_workspace_bytes(ix, cap) > ws_bytes)
            return set_error(FLINNG_ERR_INVALID_ARG, "internal: tensor-core SRP scratch of %zu bytes", ws_bytes);
    }
    const uint64_t chunk = cap;
    Carver c(ws, ~size_t(0));
    char *xq = c.take<char>(cap * x_bytes(ix));
    float *xn = c.take<float>(cap);
    float *xr = c.take<float>(cap);
    float *xsc = c.take<float>(cap);
    unsigned long long *cnt = c.take<unsigned long long>(8);
    unsigned long long *list1 = c.take<unsigned long long>(cap * P + 1);
    unsigned long long *list2 = c.take<unsigned long long>(cap * P + 1);
    uint32_t *rowcnt = c.take<uint32_t>(cap + 1);
    uint32_t *rowoff = c.take<uint32_t>(cap + 1);
    uint32_t *fill = c.take<uint32_t>(cap + 1);
    void *scan_ws = c.take<char>(scan_workspace_bytes(cap + 1));
    FL_CUDA(cudaMemsetAsync(ix->stats, 0, kStats * sizeof(unsigned long long), st));
    if (n == 0) return FLINNG_OK;
    FL_CUDA(cudaMemsetAsync(buckets, 0, n * L * sizeof(uint32_t), st));
    const char *w1p = static_cast<const char *>(ix->w_split), *wqp = bytes ? w1p + size_t(P) * d * 4 : w1p;
    CUtensorMap mw1, mw2, mwq;
    FL_TRY(make_map(&mw1, w1p, P, d, false));
    FL_TRY(make_map(&mw2, w1p + size_t(P) * d * 2, P, d, false));
    if (bytes) FL_TRY(make_map(&mwq, wqp, P, d, true));
    else mwq = mw1;
    // margin factors (see the header comment), in double then rounded up
    const double u = std::ldexp(1.0, -24), up = std::ldexp(1.0, -22);
    auto g = [](double m, double uu) { return m * uu / (1.0 - m * uu); };
    const double q = (1 + std::ldexp(1.0, -8)) * (1 + std::ldexp(1.0, -8));
    const double kb = prec == FLINNG_PREC_FP8 ? 128.0 : double(kTK);     // products per k-block
    const double m_blocks = std::ceil(double(d) / kb);
    const double m64 = std::ceil(double(d) / kTK);
    const double f2 = (g(kTK, up) + std::ldexp(1.0, -7) * g(2 * kTK, up)) * q +
                      g(2 * m64, u) * (1 + g(kTK, up)) * (1 + std::ldexp(1.0, -7)) * q;
    const double f1 = g(kb, up) + g(m_blocks, u) * (1 + g(kb, up));    // times (||x|| + ||e_x||)(||w|| + ||e_w||)
    const float c_two = std::nextafter(float(f2 * 1.0001), INFINITY);
    const float c_norm = prec == FLINNG_PREC_BF16X2 ? c_two : std::nextafter(float(f1 * 1.0001), INFINITY);
    const float c_sub = std::nextafter(float(std::sqrt(double(d)) * std::ldexp(1.0, -125)), INFINITY);
    const float tiny = std::nextafter(float(8.0 * d * std::ldexp(1.0, -126)), INFINITY);
    const double g2d = 2.0 * d * std::ldexp(1.0, -24) / (1.0 - 2.0 * d * std::ldexp(1.0, -24));
    const float g2 = std::nextafter(float(2.0 * g2d * g2d + std::ldexp(1.0, -40)), INFINITY);
    for (uint64_t r0 = 0; r0 < n; r0 += chunk) {
        const uint64_t rows = (n - r0) < chunk ? (n - r0) : chunk;
        const float *xc = x + r0 * ld;
        const bool dense = dense_second_pass(prec, d);
        const bool two = prec == FLINNG_PREC_BF16X2 || (dense && prec == FLINNG_PREC_BF16);
        FL_TRY(quant_rows(prec, xc, ld, rows, d, xq, xn, xr, xsc, two, st));
        CUtensorMap mx1, mx2;
        FL_TRY(make_map(&mx1, xq, rows, d, bytes));
        if (two) FL_TRY(make_map(&mx2, xq + rows * d * 2, rows, d, false));
        else mx2 = mx1;
        FL_CUDA(cudaMemsetAsync(cnt, 0, 8 * sizeof(unsigned long long), st));
        TcArgs a{};
        a.n = rows;
        a.P = P;
        a.d = d;
        a.L = L;
        a.K = K;
        a.xnorm = xn;
        a.wnorm = ix->w_norm;
        a.xres = xr;
        a.wres = bytes ? ix->w_aux + P : ix->w_aux;
        a.xscale = xsc;
        a.wscale = bytes ? ix->w_aux + 2 * P : nullptr;
        a.c_norm = c_norm;
        a.c_sub = c_sub;
        a.tiny = tiny;
        a.codes = buckets + r0 * L;
        a.proj = proj ? proj + r0 * P : nullptr;
        a.rlist = list1;
        a.rcount = cnt;
        a.mask = reinterpret_cast<uint32_t *>(list2);     // free until the list is grouped by row
        a.nund = cnt + 2;
        a.stats = ix->stats;
        a.err = ix->tc_err;
        a.wait_ns = ix->tc_wait_ns ? ix->tc_wait_ns - 1 : kWaitNs;
        if (prec == FLINNG_PREC_BF16X2) FL_TRY((launch_tc<kFormBf16x2, 0>(mx1, mx2, mw1, mw2, a, rows, st)));
        else if (!dense) FL_TRY((launch_tc<kFormBf16, 0>(mx1, mx1, mwq, mwq, a, rows, st)));
        else if (prec == FLINNG_PREC_BF16) {
            a.c_one = c_norm;
            a.c_norm = c_two;
            FL_TRY((launch_tc<kFormBf16x2, 3>(mx1, mx2, mw1, mw2, a, rows, st)));
        } else {
            // FP8: the marked projections again on the two-term split, whose margin
            // leaves a few in a thousand
            FL_TRY((launch_tc<kFormFp8, 1>(mx1, mx1, mwq, mwq, a, rows, st)));
            FL_TRY(quant_rows(FLINNG_PREC_BF16X2, xc, ld, rows, d, xq, xn, xr, nullptr, true, st));
            a.wres = ix->w_aux;
            FL_TRY(make_map(&mx1, xq, rows, d, false));
            FL_TRY(make_map(&mx2, xq + rows * d * 2, rows, d, false));
            a.c_norm = c_two;
            a.proj = nullptr;
            FL_TRY((launch_tc<kFormBf16x2, 2>(mx1, mx2, mw1, mw2, a, rows, st)));
        }
        // stage 2: compensated fp32; stage 3: fp64 / exact. A
        // single-term list (d < 128) is grouped by row, so that each row of x is
        // staged once; the others are short and not worth the passes.
        if (!dense && prec != FLINNG_PREC_BF16X2) {
            // the list grouped by row into list2; stage 2 lists what stays undecided in list1
            FL_CUDA(cudaMemsetAsync(rowcnt, 0, (rows + 1) * sizeof(uint32_t), st));
            FL_CUDA(cudaMemsetAsync(fill, 0, (rows + 1) * sizeof(uint32_t), st));
            k_rows_hist<<<152 * 8, 256, 0, st>>>(list1, cnt, rowcnt);
            count_launch();
            FL_CUDA(cudaGetLastError());
            FL_TRY(scan_exclusive(rowcnt, rowoff, rows, scan_ws, st));
            k_rows_scatter<<<152 * 8, 256, 0, st>>>(list1, cnt, rowoff, fill, list2);
            count_launch();
            FL_CUDA(cudaGetLastError());
            const unsigned grid = unsigned(rows < 152ull * 8 ? rows : 152ull * 8);
            k_srp_recheck2_rows<<<grid, 256, size_t(d) * sizeof(float), st>>>(
                x + r0 * ld, ld, ix->srp_w, d, L, K, g2, tiny, uint32_t(rows), list2, rowoff, buckets + r0 * L, list1,
                cnt + 1, ix->stats);
            count_launch();
            FL_CUDA(cudaGetLastError());
            FL_TRY(srp_recheck_list(ix, x + r0 * ld, ld, list1, cnt + 1, buckets + r0 * L));
        } else {
            auto fn = rows_vec4(xc, ld, d) ? k_srp_recheck2<true> : k_srp_recheck2<false>;
            fn<<<152 * 8, 256, 0, st>>>(x + r0 * ld, ld, ix->srp_w, d, L, K, g2, tiny, list1, cnt,
                                                   buckets + r0 * L, list2, cnt + 1, ix->stats);
            count_launch();
            FL_CUDA(cudaGetLastError());
            FL_TRY(srp_recheck_list(ix, x + r0 * ld, ld, list2, cnt + 1, buckets + r0 * L));
        }
        FL_TRY(add_counter(ix->stats, dense ? cnt + 2 : cnt, st));     // undecided after the first pass
    }
    // no synchronisation here (servers hash on their own streams): the flag
    // lands in pinned memory and the next call on this index reports it
    FL_CUDA(cudaMemcpyAsync(ix->h_flag + 3, ix->tc_err, 4, cudaMemcpyDeviceToHost, st));
    return FLINNG_OK;
}

}  // namespace flinng
