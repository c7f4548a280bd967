// Densification of one-permutation MinHash, shared by the batch kernel (hash.cu)
// and the fused query (query_impl.cuh).
#pragma once
#include "internal.cuh"

namespace flinng {

__device__ __forceinline__ uint64_t splitmix64(uint64_t z)
{
    z += 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Draw att (1, 2, ...) of empty bin k: splitmix64(seed ^ (k << 32 | att)) mod nb.
__device__ __forceinline__ uint32_t doph_draw_of(uint32_t k, uint32_t att, uint32_t nb, uint64_t seed)
{
    const uint64_t z = splitmix64(seed ^ ((uint64_t(k) << 32) | att));
    return (nb & (nb - 1u)) == 0u ? uint32_t(z) & (nb - 1u) : uint32_t(z % nb);
}

// The bin whose value empty bin k takes: its first draw that is occupied (occ: a
// bit per bin, one of them set), within kDophMaxAttempts, else the next occupied
// bin cyclically. The draws depend on the seed and k alone, so the first
// kDophTable come from a table, one 16-byte load: a fifth of the instructions of
// computing them, where that was most of a short set's hashing.
__device__ __forceinline__ uint32_t doph_source(uint32_t k, uint32_t nb, uint64_t seed, const uint16_t *draw,
                                                const uint32_t *occ)
{
    const uint4 d = __ldg(reinterpret_cast<const uint4 *>(draw) + k);
    const uint32_t w[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
    for (uint32_t t = 0; t < kDophTable; ++t) {
        const uint32_t j = (w[t / 2] >> (16 * (t & 1))) & 0xFFFFu;
        if ((occ[j >> 5] >> (j & 31)) & 1u) return j;
    }
    for (uint32_t att = kDophTable + 1; att <= kDophMaxAttempts; ++att) {
        const uint32_t j = doph_draw_of(k, att, nb, seed);
        if ((occ[j >> 5] >> (j & 31)) & 1u) return j;
    }
    for (uint32_t s = 1; s <= nb; ++s) {
        const uint32_t j = (k + s) % nb;
        if ((occ[j >> 5] >> (j & 31)) & 1u) return j;
    }
    return k;
}

}  // namespace flinng
