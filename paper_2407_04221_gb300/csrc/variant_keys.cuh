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

// The random part of the keys of the matches at anchor cell p, draw(key_seed, 13, env,
// t, p) >> 48.
__device__ __forceinline__ uint32_t match_random(uint64_t prefix, int t, uint32_t p)
{
    return (uint32_t)(mix64(prefix ^ (((uint64_t)(uint32_t)t << 32) | p)) >> 48);
}

// Key of the match at anchor cell p in rotation g, (p << 2) | g, with random keys
// below (draw(key_seed, 13, env, t, p) >> 48) << 14; keys are below 2^30 and
// distinct within a rule.
__device__ __forceinline__ uint32_t match_key(const VariantParams &vp, uint64_t prefix, int t, uint32_t p, uint32_t g)
{
    uint32_t key = (p << 2) | g;
    if (vp.random_keys)
        key |= match_random(prefix, t, p) << 14;
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

// keep_largest with random keys from the cells' random parts (shared memory, 32 a word,
// 16-byte aligned), for lanes with many matches: every bit of a word is looked at, in
// straight-line code, where the loop above takes a mix for each match after another.
template <int NA>
__device__ __forceinline__ void keep_largest_cells(uint32_t (&m)[NA], int k, const uint16_t *cells)
{
    const int lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    uint32_t kept[NA];
#pragma unroll
    for (int u = 0; u < NA; ++u)
        kept[u] = 0u;
    for (int i = 0; i < k; ++i) {
        uint32_t best = 0;  // this lane's largest key + 1 (0: no candidate left)
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const uint32_t x = m[u], base = (uint32_t)(q + 8 * u) * 32u;
            if (!__any_sync(0xffffffffu, x != 0u))
                continue;
            uint32_t top = 0;  // of the word: random part << 5 | bit, + 1
            const uint4 *c4 = reinterpret_cast<const uint4 *>(cells + base);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint4 c = c4[j];
                const uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    const int b = 8 * j + h;
                    const uint32_t v = ((w[h >> 1] >> (16 * (h & 1))) & 0xffffu) * 32u + (uint32_t)(b + 1);
                    if ((x >> b) & 1u)
                        top = max(top, v);
                }
            }
            if (top) {
                --top;
                best = max(best, (top >> 5 << 14 | (base + (top & 31u)) << 2 | (uint32_t)g) + 1u);
            }
        }
        const uint32_t top = __reduce_max_sync(0xffffffffu, best);
        if (top == 0u)
            break;
        if (best == top) {  // keys are distinct: exactly one lane
            const uint32_t p = ((best - 1u) >> 2) & 0xfffu, bit = 1u << (p & 31u);
#pragma unroll
            for (int u = 0; u < NA; ++u)
                if ((int)(p >> 5) == q + 8 * u) {
                    kept[u] |= bit;
                    m[u] &= ~bit;
                }
        }
    }
#pragma unroll
    for (int u = 0; u < NA; ++u)
        m[u] = kept[u];
}

}  // namespace av
