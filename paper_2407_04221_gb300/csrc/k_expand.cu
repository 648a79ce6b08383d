// k_expand.cu -- tree-search expansion kernels: one warp per parent for boards
// of at most 16 plane words, one CTA per parent otherwise.
#include <algorithm>

#include "small_step.cuh"

namespace av {
namespace {

// FNV-1a 64 over n bytes (shared memory, 16-byte aligned).
__device__ __forceinline__ uint64_t fnv_bytes(const unsigned char *p, int n)
{
    const uint4 *p4 = reinterpret_cast<const uint4 *>(p);
    uint64_t h = 0xcbf29ce484222325ULL;
    int k = 0;
    for (; k + 16 <= n; k += 16) {
        const uint4 y = p4[k >> 4];
        const uint32_t ws[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int j = 0; j < 16; ++j)
            h = (h ^ ((ws[j >> 2] >> (8 * (j & 3))) & 0xffu)) * 0x100000001b3ULL;
    }
    for (; k < n; ++k)
        h = (h ^ p[k]) * 0x100000001b3ULL;
    return h;
}

// Tree-search expansion: one CTA per parent, the 5 children in turn.  A child's cells
// are made eight at a time by bit transposes and hashed 16 bytes a load (4096 parents of
// 40 x 40: cell by cell, a channel's word each, 471 us with 4 rules and 1733 with 64 that
// fire; 403 and 1623).
template <typename CellT, bool SM>
__global__ void __launch_bounds__(kThreads)
expand_kernel(DevConfig cf, BlockShape bs, const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g,
              const CellT *__restrict__ parents, int F, const int32_t *__restrict__ n_parent,
              CellT *children, int32_t *rewards, uint8_t *done, uint64_t *hashes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const BlockSmem S = block_carve(smem, block_layout(cf, bs, 0, 5), cf, bs);
    const int node = blockIdx.x, env = node / F, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int HW = cf.HW, NW = cf.NW, NWP = cf.NWP, C = cf.C;
    const int stride = block_child_bytes(HW, (int)sizeof(CellT));  // from one child's bytes to the next's
    if (n_parent && node - env * F >= n_parent[env])
        return;  // block-uniform: an empty frontier slot
    const BlockTable tb = block_stage<SM>(cf, bs, S, cf.rules_per_env ? env : 0);
    __syncthreads();
    block_load_planes<CellT>(cf, parents + (size_t)node * HW, S.planes);
    __syncthreads();

    int slot = 0;
    for (int a = 0; a < 5; ++a) {
        if (warp == 0)
            force_plane(cf, S.planes, masks_g, a);
        __syncthreads();
        int warp_rew = 0;
        const bool any = block_match<SM, false>(cf, bs, tb, S, vm_g, NW, 0, slot, warp_rew);
        if (lane == 0)
            S.ctl[warp] = warp_rew;
        int goal = 0;
        for (int i = tid; i < C * NW; i += kThreads) {  // child planes, kept in SET's place
            const int c = i / NW, w = i - c * NW;
            const uint32_t d = S.planes[c * NWP + w].x;
            uint32_t v = d;
            if (any) {
                v = (d & ~S.clrp[i]) | (~d & S.setp[i]);
                S.clrp[i] = 0u;
            }
            S.setp[i] = v;
            if (c == cf.ch_goal && v)
                goal = 1;
        }
        const int goal_left = __syncthreads_or(goal) || cf.ch_goal < 0;
        if (tid == 0) {
            rewards[(size_t)node * 5 + a] = block_reward(S);
            if (done)
                done[(size_t)node * 5 + a] = (uint8_t)!goal_left;
        }
        // its canonical bytes, eight cells a thread, for the hash and the child
        unsigned char *bytes = S.cells + a * stride;
        CellT *dst = children + ((size_t)node * 5 + a) * HW;
        const bool vec = cells8_aligned(dst, HW);
        for (int b = tid; 8 * b < HW; b += kThreads) {
            uint32_t o[4];
            get_bytes8<CellT>(reinterpret_cast<const uint8_t *>(S.setp) + b, NW * 4, C, o);
            if constexpr (sizeof(CellT) == 1) {
                const uint2 x = make_uint2(o[0], o[1]);
                reinterpret_cast<uint2 *>(bytes)[b] = x;
                if (vec)
                    reinterpret_cast<uint2 *>(dst)[b] = x;
            } else {
                const uint4 x = make_uint4(o[0], o[1], o[2], o[3]);
                reinterpret_cast<uint4 *>(bytes)[b] = x;
                if (vec)
                    reinterpret_cast<uint4 *>(dst)[b] = x;
            }
        }
        __syncthreads();  // the bytes; the child's planes are read
        if (!vec)
            for (int p = tid; p < HW; p += kThreads)
                dst[p] = reinterpret_cast<const CellT *>(bytes)[p];
        for (int i = tid; i < C * NW; i += kThreads)
            S.setp[i] = 0u;
    }
    // FNV-1a 64 over the canonical bytes, one thread per child
    if (lane == 0 && warp < 5)
        hashes[(size_t)node * 5 + warp] = fnv_bytes(S.cells + warp * stride, HW * (int)sizeof(CellT));
}

constexpr int kExpWarps = 8;  // parents per CTA at most
constexpr int kExpBatch = 2;  // rules whose first terms are tested together

// Shared memory of expand_warp_kernel: one region per CTA (valid-anchor and column
// masks, the packed table when staged, the boards to hash and their hashes), then
// per warp its planes, a SET / CLEAR region per action, one child's planes, the
// parent's canonical bytes and the writes' scratch.  A child's bytes take its
// SET / CLEAR region's place once the child is made.
struct ExpandLayout {
    int vm, masks, list, hash, tab, warps;                                   // CTA region
    int planes, acc, child, bytes, lead, match, queue, per_warp;             // within a warp's region
    int slot;         // bytes from one action's region to the next's
    int pad, mstride;
};

ExpandLayout expand_layout(const DevConfig &cf)
{
    ExpandLayout L;
    int at = 0;
    auto take = [&](int bytes) {
        const int here = at;
        at = (at + bytes + 15) & ~15;
        return here;
    };
    L.vm = take(kShapes * cf.NW * 4);
    L.masks = take(3 * cf.NW * 4);
    L.list = take((1 + 6 * kExpWarps) * 4);
    L.hash = take(6 * kExpWarps * 8);
    L.tab = take(cf.pk_staged * 4);
    L.warps = at;
    L.pad = small_pad(cf.W);
    L.mstride = 8 * cf.NA + L.pad;
    at = 0;
    const int board = ((cf.HW + 7) / 8 * 8 * cf.cell_bytes + 15) & ~15;
    const int region = (2 * cf.C * cf.NW * 4 + 15) & ~15;
    // 16 bytes apart in their banks, so that threads reading the same place of
    // different boards do not meet
    L.slot = std::max(board, region) + 16;
    L.planes = take((cf.C + 5) * cf.NWP * 8);
    L.acc = take(5 * L.slot);
    L.child = take(cf.C * cf.NW * 4);
    L.bytes = take(board + 16);
    L.lead = take(kExpBatch * 32 * cf.NA * 4);
    L.match = take(4 * L.mstride * 4);
    L.queue = take(kSmallSparse * 4);
    L.per_warp = at;
    return L;
}

// Plane of action a's force in expand_warp_kernel: action 0 has none, which is the
// zero plane C + 1 that padding terms read.
__device__ __forceinline__ int expand_force_plane(int C, int a) { return C + (a == 0 ? 1 : a == 4 ? 0 : a + 1); }

// The force planes of actions 1..4 from the player plane (one warp: quarter g makes
// action g + 1's words).
template <int NA>
__device__ __forceinline__ void expand_forces(const DevConfig &cf, uint2 *P, const uint32_t *masks)
{
    const int lane = threadIdx.x & 31, a = (lane >> 3) + 1, NW = cf.NW;
    const uint2 *pl = P + (cf.ch_player >= 0 ? cf.ch_player : 0) * cf.NWP;
    const int n = (a & 1) ? cf.W : 1, d = n >> 5, r = n & 31;
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        const int w = (lane & 7) + 8 * u;
        if (w >= NW)
            continue;
        uint32_t f = 0;
        if (cf.ch_player >= 0) {
            if (a == 1 || a == 4) {  // toward lower p: bits [32w + n, 32w + n + 32)
                const uint2 e = pl[w + d];
                f = __funnelshift_r(e.x, e.y, r);
            } else if (w > d) {  // toward higher p: bits [32w - n, 32w - n + 32)
                const uint2 e = pl[w - d - 1];
                f = __funnelshift_l(e.x, e.y, r);
            } else if (w == d) {
                f = pl[0].x << r;
            }
            if (a == 2)
                f &= ~masks[w];  // not from the last column onto the first
            else if (a == 4)
                f &= ~masks[NW + w];
            f &= masks[2 * NW + w];
        }
        put_word(P, cf.NWP, expand_force_plane(cf.C, a), w, f);
    }
}

// A batch of terms with its force terms replaced by ones that pass (they read the
// zero plane as absent).
__device__ __forceinline__ uint32_t expand_tile_term(uint32_t p, uint32_t force, uint32_t span)
{
    return (p >> 16) - force < span ? ((force + span) << 16) | 0x8000u : p;
}
__device__ __forceinline__ uint4 expand_tile_terms(const uint4 &p, uint32_t force, uint32_t span)
{
    return make_uint4(expand_tile_term(p.x, force, span), expand_tile_term(p.y, force, span),
                      expand_tile_term(p.z, force, span), expand_tile_term(p.w, force, span));
}

// This lane's cells of a board into its canonical bytes (shared, whole units).
template <typename CellT, int NA>
__device__ __forceinline__ void expand_put(unsigned char *dst, const SmallCells<CellT, NA> &v, int HW)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        const int b = lane + 32 * u;
        if (8 * b >= HW)
            continue;
        if constexpr (sizeof(CellT) == 1)
            reinterpret_cast<uint2 *>(dst)[b] = make_uint2(v.v[u][0], v.v[u][1]);
        else
            reinterpret_cast<uint4 *>(dst)[b] = make_uint4(v.v[u][0], v.v[u][1], v.v[u][2], v.v[u][3]);
    }
}

// Tree-search expansion, one warp per parent, up to eight parents of one environment
// per CTA (they share the staged table).  A parent's five children differ only in
// the force plane, so each rule's terms on tile channels are tested once, and the
// anchors that pass them go through its few force terms once per action.  A child
// no rule wrote is its parent: its cells and its hash are the parent's.  The boards
// that need one are hashed (FNV-1a 64, a serial chain over the bytes) one per
// thread at the end.
//
// What bounds it: instruction issue.  16,384 parents of 16 x 16 with 8 rules: 4,700
// warp-instructions a parent (force terms tested for and skipped in every batch, a
// ballot per channel and word to load the board, all five children rebuilt and hashed,
// hash loads that met in one bank): 98.4 -> 59.8 us.
template <typename CellT, int NA, bool SM>
__global__ void __launch_bounds__(32 * kExpWarps, 4)
expand_warp_kernel(const __grid_constant__ DevConfig cf, const __grid_constant__ ExpandLayout L,
                   const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g,
                   const CellT *__restrict__ parents, int F, const int32_t *__restrict__ n_parent,
                   CellT *children, int32_t *rewards, uint8_t *done, uint64_t *hashes)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const int g = lane >> 3, q = lane & 7;
    const long long first_node = (long long)blockIdx.x * nwarps;  // this CTA's first parent
    const long long node = first_node + warp;
    const long long total_nodes = (long long)cf.B * F;
    const int env = (int)(min(first_node, total_nodes - 1) / F);  // of every parent of the CTA
    const int f0 = (int)(first_node - (long long)env * F), np = n_parent ? min(n_parent[env], F) : F;
    if (f0 >= np)
        return;  // block-uniform: no parent here
    const bool mine = node < total_nodes && f0 + warp < np;  // this warp has a parent to expand
    const int HW = cf.HW, NW = cf.NW, NWP = cf.NWP, C = cf.C;
    const uint32_t force = (uint32_t)(C * NWP * 8), span = (uint32_t)(NWP * 8);

    // ---- the CTA's shared region
    uint32_t *vm = reinterpret_cast<uint32_t *>(smem + L.vm);
    uint32_t *masks = reinterpret_cast<uint32_t *>(smem + L.masks);
    int *list = reinterpret_cast<int *>(smem + L.list);  // [0] entries, then (warp, board) as 6 * warp + board
    uint64_t *hash = reinterpret_cast<uint64_t *>(smem + L.hash);  // [warp][board]
    const uint32_t *pk = cf.pk + cf.pk_off[cf.rules_per_env ? env : 0];
    const uint4 counts = __ldg(reinterpret_cast<const uint4 *>(pk));
    uint32_t *const tab_s = reinterpret_cast<uint32_t *>(smem + L.tab);
    const BlockTable tb = block_table(SM ? tab_s : pk, counts, cf.R);
    for (int i = threadIdx.x; i < kShapes * NW; i += blockDim.x)
        vm[i] = __ldg(vm_g + i);
    for (int i = threadIdx.x; i < 3 * NW; i += blockDim.x)
        masks[i] = __ldg(masks_g + i);
    if (threadIdx.x == 0)
        list[0] = 0;
    if (SM) {
        const int n = (int)(cf.pk_off[(cf.rules_per_env ? env : 0) + 1] - cf.pk_off[cf.rules_per_env ? env : 0]) / 4;
        const int t0 = 1 + 2 * cf.R, t1 = t0 + 4 * (int)counts.x;  // the terms: force terms replaced
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(pk) + i);
            reinterpret_cast<uint4 *>(tab_s)[i] = i >= t0 && i < t1 ? expand_tile_terms(x, force, span) : x;
        }
    }
    // ---- this warp's region
    unsigned char *wr = smem + L.warps + warp * L.per_warp;
    uint2 *planes = reinterpret_cast<uint2 *>(wr + L.planes);
    uint32_t *child = reinterpret_cast<uint32_t *>(wr + L.child);
    uint32_t *lead = reinterpret_cast<uint32_t *>(wr + L.lead);
    SmallOut S;
    S.match = reinterpret_cast<uint32_t *>(wr + L.match);
    S.queue = reinterpret_cast<uint32_t *>(wr + L.queue);
    S.pad = L.pad;
    S.mstride = L.mstride;
    const CellT *par = parents + (size_t)node * HW;
    if (mine) {
        for (int i = lane; i < (C + 5) * NWP / 2; i += 32)  // (NWP is even)
            reinterpret_cast<uint4 *>(planes)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = lane; i < 5 * L.slot / 16; i += 32)
            reinterpret_cast<uint4 *>(wr + L.acc)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (int i = lane; i < 4 * L.mstride; i += 32)
            S.match[i] = 0u;
        __syncwarp();
        const bool vec = cells8_aligned(par, HW);
        for (int b = lane; 8 * b < HW; b += 32)
            put_cells8<CellT>(cf, par, b, vec, planes);
    }
    __syncthreads();  // the shared region

    if (mine) {
        expand_forces<NA>(cf, planes, masks);
        __syncwarp();
        // ---- every rule in its four rotations
        const uint32_t pbase = (uint32_t)__cvta_generic_to_shared(planes) + q * 8;
        int rew = 0;          // lane a: action a's reward
        uint32_t wrote = 0;   // bit a: a rule matched under action a
        for (int r0 = 0; r0 < cf.R; r0 += kExpBatch) {
            uint32_t m[kExpBatch][NA];
            uint32_t alive = 0;
#pragma unroll
            for (int k = 0; k < kExpBatch; ++k) {
                const int r = r0 + k;
                if (k > 0 && r >= cf.R)
                    break;
                const uint32_t *vmr = vm + ((block_ld<SM>(&tb.hdr[2 * r].w) >> (8 * g)) & 0xffu) * NW;
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    m[k][u] = q + 8 * u < NW ? vmr[q + 8 * u] : 0u;
                const uint4 p = block_ld<SM>(tb.terms + 4 * r + g);
                small_terms<NA>(pbase, SM ? p : expand_tile_terms(p, force, span), m[k]);
            }
#pragma unroll
            for (int k = 0; k < kExpBatch; ++k) {
                if (k > 0 && r0 + k >= cf.R)
                    break;
                alive |= __any_sync(0xffffffffu, (m[k][0] | m[k][NA - 1]) != 0u) ? 1u << k : 0u;
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    lead[(k * 32 + lane) * NA + u] = m[k][u];
            }
            for (; alive; alive &= alive - 1) {
                const int k = __ffs(alive) - 1, r = r0 + k;
                const uint4 h0 = block_ld<SM>(tb.hdr + 2 * r), h1 = block_ld<SM>(tb.hdr + 2 * r + 1);
                uint32_t x[NA];
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    x[u] = lead[(k * 32 + lane) * NA + u];
                const uint4 *tp = tb.terms + 4 * h1.x + g;
                bool live = true;
                for (uint32_t b = 1; live && b < h0.x; ++b) {
                    const uint4 p = block_ld<SM>(tp + 4 * (b - 1));
                    small_terms<NA>(pbase, SM ? p : expand_tile_terms(p, force, span), x);
                    live = __any_sync(0xffffffffu, (x[0] | x[NA - 1]) != 0u);
                }
                if (!live)
                    continue;
                // the force terms, action by action
                const uint32_t nf = (h0.y >> 8) & 0xffu;
                const uint32_t *fp = tb.forces + 4 * (h0.y >> 16) + g;
                for (int a = 0; a < 5; ++a) {
                    const uint32_t shift = (uint32_t)(expand_force_plane(C, a) - C) * span;
                    uint32_t y[NA];
#pragma unroll
                    for (int u = 0; u < NA; ++u)
                        y[u] = x[u];
                    for (uint32_t f = 0; f < nf; ++f) {
                        const uint32_t p = block_ld<SM>(fp + 4 * f), neg = block_neg(p);
                        const uint32_t at = pbase + (p >> 16) + shift;
#pragma unroll
                        for (int u = 0; u < NA; ++u) {
                            const uint2 w = lds2(at + 64 * u);
                            y[u] &= __funnelshift_r(w.x, w.y, p) ^ neg;
                        }
                    }
                    if (!__any_sync(0xffffffffu, (y[0] | y[NA - 1]) != 0u))
                        continue;
                    int cnt = 0;
#pragma unroll
                    for (int u = 0; u < NA; ++u)
                        cnt += __popc(y[u]);
                    const int total = __reduce_add_sync(0xffffffffu, cnt);
                    wrote |= 1u << a;
                    if (lane == a)
                        rew += (int)h0.z * total;
                    S.acc = reinterpret_cast<uint32_t *>(wr + L.acc + a * L.slot);
                    small_write<NA, SM>(cf, tb, S, h0, h1, y, total);
                }
            }
        }
        __syncwarp();  // every lane's SET / CLEAR bits
        // ---- the children: the parent's cells, or the written planes'
        const int nbytes = HW * (int)sizeof(CellT);
        const int mode = small_store_mode<CellT, true>(children, nbytes);
        unsigned char *dst = reinterpret_cast<unsigned char *>(children) + (size_t)node * 5 * nbytes;
        SmallCells<CellT, NA> v;
        small_cells<CellT, NA>(cf, planes, v);
        expand_put<CellT, NA>(wr + L.bytes, v, HW);
        const int sh = NW <= 8 ? 3 : 4, w = lane & ((1 << sh) - 1);
        uint32_t goals = 0;    // bit a: a goal tile is left in child a
        uint32_t differs = 0;  // bit a: child a is not its parent
        bool pgoal = cf.ch_goal < 0;
        if (cf.ch_goal >= 0)
            pgoal = __any_sync(0xffffffffu, w < NW && planes[cf.ch_goal * NWP + w].x != 0u);
#pragma unroll 1
        for (int a = 0; a < 5; ++a, dst += nbytes) {
            bool goal = pgoal, diff = false;
            if ((wrote >> a) & 1u) {
                uint32_t *acc = reinterpret_cast<uint32_t *>(wr + L.acc + a * L.slot);
                uint32_t flips = 0, left = 0;
                if (w < NW)
                    for (int c = lane >> sh; c < C; c += 32 >> sh) {
                        const uint32_t d = planes[c * NWP + w].x, st = acc[c * NW + w], cl = acc[(C + c) * NW + w];
                        const uint32_t nd = (d & ~cl) | (~d & st);
                        flips |= nd ^ d;
                        child[c * NW + w] = nd;
                        if (c == cf.ch_goal)
                            left = nd;
                    }
                diff = __any_sync(0xffffffffu, flips != 0u);
                if (diff) {
                    if (cf.ch_goal >= 0)
                        goal = __any_sync(0xffffffffu, left != 0u);
                    __syncwarp();
                    SmallCells<CellT, NA> x;
#pragma unroll
                    for (int u = 0; u < NA; ++u) {
                        uint32_t y[4];
                        // (a unit past the board reads another channel's bytes and is not stored)
                        get_bytes8<CellT>(reinterpret_cast<const uint8_t *>(child) + min(lane + 32 * u, 4 * NW - 1),
                                          NW * 4, C, y);
#pragma unroll
                        for (int i = 0; i < 2 * (int)sizeof(CellT); ++i)
                            x.v[u][i] = y[i];
                    }
                    small_store<CellT, NA, true>(dst, x, nbytes, mode);
                    expand_put<CellT, NA>(reinterpret_cast<unsigned char *>(acc), x, HW);
                    __syncwarp();  // the child's planes may be overwritten
                }
            }
            if (!diff)
                small_store<CellT, NA, true>(dst, v, nbytes, mode);
            goals |= goal ? 1u << a : 0u;
            differs |= diff ? 1u << a : 0u;
        }
        if (lane < 5) {
            rewards[(size_t)node * 5 + lane] = rew;
            if (done)
                done[(size_t)node * 5 + lane] = (uint8_t)!((goals >> lane) & 1u);
        }
        // the boards to hash: the children that differ, and the parent for the others
        const uint32_t need = differs | (differs == 31u ? 0u : 32u);
        int at = 0;
        if (lane == 0) {
            at = atomicAdd(list, __popc(need));
            hash[6 * warp] = differs;  // (read before the hashes are written)
        }
        at = __shfl_sync(0xffffffffu, at, 0);
        if (lane < 6 && ((need >> lane) & 1u))
            list[1 + at + __popc(need & ((1u << lane) - 1u))] = 6 * warp + lane;
    }
    __syncthreads();  // every board's bytes, the list
    const uint32_t differs = mine ? (uint32_t)hash[6 * warp] : 0u;
    __syncthreads();

    // ---- FNV-1a 64 over each listed board's canonical bytes, one thread per board
    const int nbytes = HW * (int)sizeof(CellT);
    for (int i = threadIdx.x; i < list[0]; i += blockDim.x) {
        const int x = list[1 + i], wx = x / 6, board = x - 6 * wx;
        hash[x] = fnv_bytes(smem + L.warps + wx * L.per_warp + (board == 5 ? L.bytes : L.acc + board * L.slot), nbytes);
    }
    __syncthreads();  // the hashes
    if (mine && lane < 5)
        hashes[(size_t)node * 5 + lane] = hash[6 * warp + (((differs >> lane) & 1u) ? lane : 5)];
}

// Parents per CTA on the warp path: 1 while the GPU has room for every warp at
// once (best balance), more for large batches.  The count divides F so that
// a CTA's parents share one environment (and its rule table).
int warps_per_cta(long long units, int F)
{
    int w = units <= 152LL * 32 ? 1 : (units <= 152LL * 64 ? 2 : kExpWarps);
    while (w > 1 && F % w != 0)
        w >>= 1;
    return w;
}

template <typename CellT>
void block_t(const DevConfig &cf, const uint32_t *vm, const uint32_t *masks, const void *parents, int F, const int32_t *n_parent, void *children,
             int32_t *rewards, uint8_t *done, uint64_t *hashes, cudaStream_t st)
{
    const BlockShape bs = block_shape_fit(cf, cf.NW, 0, 5);
    const size_t sm = block_layout(cf, bs, 0, 5).total;
    const unsigned grid = (unsigned)(cf.B * F);
    if (cf.pk_staged)
        expand_kernel<CellT, true><<<grid, kThreads, sm, st>>>(cf, bs, vm, masks,
                                                              (const CellT *)parents, F, n_parent,
                                                              (CellT *)children, rewards, done, hashes);
    else
        expand_kernel<CellT, false><<<grid, kThreads, sm, st>>>(cf, bs, vm, masks,
                                                               (const CellT *)parents, F, n_parent,
                                                               (CellT *)children, rewards, done, hashes);
}

template <typename CellT, int NA>
void warp_t(const DevConfig &cf, const uint32_t *vm, const uint32_t *masks, const void *parents, int F,
            const int32_t *n_parent, void *children, int32_t *rewards, uint8_t *done, uint64_t *hashes,
            cudaStream_t st)
{
    const long long units = (long long)cf.B * F;
    const ExpandLayout L = expand_layout(cf);
    int wpc = warps_per_cta(units, F);
    while (wpc > 1 && L.warps + wpc * L.per_warp > kDynSmemLimit)
        wpc >>= 1;
    const unsigned grid = (unsigned)((units + wpc - 1) / wpc);
    const int sm = L.warps + wpc * L.per_warp;
    if (cf.pk_staged > 0)
        expand_warp_kernel<CellT, NA, true><<<grid, 32 * wpc, sm, st>>>(
            cf, L, vm, masks, (const CellT *)parents, F, n_parent, (CellT *)children, rewards, done, hashes);
    else
        expand_warp_kernel<CellT, NA, false><<<grid, 32 * wpc, sm, st>>>(
            cf, L, vm, masks, (const CellT *)parents, F, n_parent, (CellT *)children, rewards, done, hashes);
}

}  // namespace

cudaError_t configure_expand()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *fn) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    };
    set((const void *)expand_kernel<uint8_t, true>);
    set((const void *)expand_kernel<uint8_t, false>);
    set((const void *)expand_kernel<uint16_t, true>);
    set((const void *)expand_kernel<uint16_t, false>);
#define AV_SETW(CELL, NA)                                            \
    set((const void *)expand_warp_kernel<CELL, NA, true>);           \
    set((const void *)expand_warp_kernel<CELL, NA, false>);
    AV_SETW(uint8_t, 1)
    AV_SETW(uint8_t, 2)
    AV_SETW(uint16_t, 1)
    AV_SETW(uint16_t, 2)
#undef AV_SETW
    return e;
}

void launch_expand(const DevConfig &cf, const uint32_t *vm, const uint32_t *masks, const void *parents, int F,
                   const int32_t *n_parent, void *children,
                   int32_t *rewards, uint8_t *done, uint64_t *hashes, cudaStream_t st)
{
    const bool u8 = cf.cell_bytes == 1;
    if (use_warp_expand(cf)) {
        if (cf.NA == 1) {
            if (u8)
                warp_t<uint8_t, 1>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
            else
                warp_t<uint16_t, 1>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
        } else {
            if (u8)
                warp_t<uint8_t, 2>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
            else
                warp_t<uint16_t, 2>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
        }
        return;
    }
    if (u8)
        block_t<uint8_t>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
    else
        block_t<uint16_t>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
}

}  // namespace av
