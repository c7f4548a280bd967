// Row loads and norm bounds shared by the SRP kernels (hash.cu, srp_tc.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace flinng {

// Upper bound of a norm from an fp32 sum of squares ss accumulated in chains of
// at most m roundings (sums of non-negative terms: relative error below 2 m u).
// Valid while norm_in_range; callers take fp64 otherwise.
__device__ __forceinline__ float norm_up(float ss, uint32_t m)
{
    return __fmul_ru(__fsqrt_ru(__fmul_ru(ss, __fmaf_ru(2.f * float(m + 4), 0x1p-24f, 1.f))), 1.f + 0x1p-20f);
}

// No overflow, and squares lost to underflow (at most 2^-149 each, d <= 2^16)
// below the relative slack; an all-zero row is its own exact bound.
__device__ __forceinline__ bool norm_in_range(float ss, bool any) { return (ss > 0x1p-90f && ss < 0x1p120f) || !any; }

__device__ __forceinline__ float norm_up64(double ss)
{
    return __double2float_ru(sqrt(ss * (1.0 + 1e-12)) * (1.0 + 1e-7));
}

// Four consecutive floats of a row from t on, zeros past d. VEC: rows are
// 16-byte aligned and d a multiple of four.
template <bool VEC>
__device__ __forceinline__ float4 load4(const float *row, uint32_t t, uint32_t d, bool in)
{
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!in) return v;
    if constexpr (VEC) {
        if (t < d) v = __ldg(reinterpret_cast<const float4 *>(row + t));
    } else {
        if (t < d) v.x = __ldg(row + t);
        if (t + 1 < d) v.y = __ldg(row + t + 1);
        if (t + 2 < d) v.z = __ldg(row + t + 2);
        if (t + 3 < d) v.w = __ldg(row + t + 3);
    }
    return v;
}

// Rows that load4<true> can read: 16-byte aligned, a multiple of four floats.
inline bool rows_vec4(const float *x, uint64_t ld, uint32_t d)
{
    return d % 4 == 0 && ld % 4 == 0 && reinterpret_cast<uintptr_t>(x) % 16 == 0;
}

}  // namespace flinng
