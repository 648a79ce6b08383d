// variant_keys.cuh -- which matches of a limited rule apply under the variant
// semantics (k_variant.cu, k_memo_impl.cuh).
#pragma once

#include "launch.h"

namespace av {

// The part of draw(key_seed, 13, env, t, p) that depends only on the environment.
__device__ __forceinline__ uint64_t variant_prefix(const VariantParams &vp, int env)
{
    return mix64(mix64(vp.key_seed + 0x9E3779B97F4A7C15ULL * 14) ^ (uint64_t)env);
}

// Key of the match at anchor cell p in rotation g, (p << 2) | g, with random keys
// below (draw(key_seed, 13, env, t, p) >> 48) << 14; keys are below 2^30 and
// distinct within a rule.
__device__ __forceinline__ uint32_t match_key(const VariantParams &vp, uint64_t prefix, int t, uint32_t p, uint32_t g)
{
    uint32_t key = (p << 2) | g;
    if (vp.random_keys)
        key |= (uint32_t)(mix64(prefix ^ (((uint64_t)(uint32_t)t << 32) | p)) >> 48) << 14;
    return key;
}

// Keep only the k matches of m with the largest keys (one warp).
template <int NA>
__device__ __forceinline__ void keep_largest(uint32_t (&m)[NA], int k, const VariantParams &vp, uint64_t prefix, int t)
{
    const int lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    uint32_t kept[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u)
        kept[u] = 0u;
    for (int i = 0; i < k; ++i) {
        uint32_t best = 0;  // this lane's largest key + 1 (0: no candidate left)
        int bu = 0, bb = 0;
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const uint32_t base = (uint32_t)(q + 8 * u) * 32u;
            if (!vp.random_keys) {
                if (m[u]) {  // the highest anchor of the highest word wins
                    const int b = 31 - __clz(m[u]);
                    best = ((base + (uint32_t)b) << 2 | (uint32_t)g) + 1u;
                    bu = u;
                    bb = b;
                }
            } else {
                for (uint32_t x = m[u]; x; x &= x - 1u) {
                    const int b = __ffs(x) - 1;
                    const uint32_t key = match_key(vp, prefix, t, base + (uint32_t)b, (uint32_t)g) + 1u;
                    if (key > best) {
                        best = key;
                        bu = u;
                        bb = b;
                    }
                }
            }
        }
        const uint32_t top = __reduce_max_sync(0xffffffffu, best);
        if (top == 0u)
            break;
        if (best == top) {  // keys are distinct: exactly one lane
#pragma unroll
            for (int u = 0; u < NA; ++u)
                if (u == bu) {
                    kept[u] |= 1u << bb;
                    m[u] &= ~(1u << bb);
                }
        }
    }
#pragma unroll
    for (int u = 0; u < NA; ++u)
        m[u] = kept[u];
}

}  // namespace av
