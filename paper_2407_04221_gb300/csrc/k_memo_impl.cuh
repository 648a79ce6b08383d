// k_memo_impl.cuh -- fused rollout that remembers, for the board in hand, the
// outcome of each action it has taken on it; included by k_memo_u8.cu and
// k_memo_u16.cu, with the variant step by k_vmemo_u8.cu, k_vmemo_u16.cu,
// k_vmany_u8.cu and k_vmany_u16.cu (boards of at most 16 plane words, any rule count).
//
// A step's result is a function of the board, the action and the step
// counter (Sec. 2.1: the rules are matched on the current board; the action
// enters only as the force tiles next to the player).  While a board stays
// unchanged, the step with action a always pays the same reward, writes the
// same SET / CLEAR bits and leaves the same goal count.  One CTA runs one
// environment and keeps, per action, the outcome of that step on the current
// board once it has been computed: its reward and whether a goal tile is left
// (an action whose step changes the board changes it at once, so the actions
// remembered are the ones that leave it as it is).  A launch walks its steps
// 32 at a time, one step per lane: every lane looks up its step's action, and
// the first step whose action has no outcome yet, or that triggers an
// auto-reset, ends the run of steps that merely repeat the board.  Those steps
// write their rewards, done flags and observations (the board's canonical
// bytes, held in registers) at once, the CTA's warps taking turns.  The step
// that ended the run is evaluated by all warps together (every rule on the
// board with that action's force, as the step-by-step kernels do, the rules
// shared out among the warps); if it leaves the board unchanged its outcome is
// remembered and the walk goes on, else its flips are applied (or the initial
// map restored) and everything remembered is dropped.  No outcome is guessed:
// each is computed once per board and action, so results are exactly those of
// the step-by-step kernels.  Every warp runs the same walk on the same data
// (the action draws, the remembered outcomes and the step counter are the same
// in each), so all of them reach each block barrier together.
#pragma once

#include <algorithm>

#include "small_step.cuh"
#include "variant_keys.cuh"

namespace av {

// The standard step; VariantParams in its place selects the variant step, whose
// outcome is remembered only when no rule has a raw match (it depends on nothing but
// the board and the action then); VariantManyParams the same for rules expected to
// match in many places at once (keep_largest_cells).
struct StandardStep {};

// Keys that a warp's rules would draw one after another (the most matches of a lane,
// rule by rule) from which on a step makes every cell's random key part instead.
constexpr int kMemoMany = 8;

constexpr int kMemoBatch = 2;    // rules per warp whose first terms are tested together (3: 2 % slower)

// Shared memory of one environment (one CTA): per rule each lane's valid-anchor
// words and the first batch of terms; the column masks; tile planes 0..C-1, the force of the action being evaluated (plane
// C) and an all-zero plane C+1 (padding terms read it as absent and pass),
// doubled; SET, then CLEAR planes (every warp ORs the outputs of its rules
// there); for each of two board slots (the current board and the one before it)
// the flip planes of each action's step; three boards' planes (flat: the two
// slots' and the one a step is making); the initial map's planes (flat); per warp
// the anchors of the rules it tests together, one rule's match planes
// [rotation][word] and its queue of matches; reductions (two sets in turn); the packed rule table
// (block_step.cuh) when staged.
struct MemoLayout {
    int vm, first, masks, planes, acc, flip, bplanes, basep, lead, match, queue, red, woff, raw, keys, tab, total;
    int pad, mstride;  // zero words in front of a rotation's match words; words per rotation
};

// Warps per environment (CTA): AV_MEMO_WARPS=1|2|4|8, read by av_create, else 4.
__host__ __device__ inline int memo_warps(const DevConfig &cf)
{
    return cf.memo_warps == 1 || cf.memo_warps == 2 || cf.memo_warps == 8 ? cf.memo_warps : 4;
}

inline MemoLayout memo_layout(const DevConfig &cf, bool staged, bool variant, bool many)
{
    MemoLayout L;
    const int pw = cf.C * cf.NW * 4;  // one plane set, bytes
    const int nw = memo_warps(cf);
    int at = 0;
    auto take = [&](int bytes) {
        const int here = at;
        at = (at + bytes + 15) & ~15;
        return here;
    };
    L.pad = small_pad(cf.W);
    L.mstride = 8 * cf.NA + L.pad;
    L.planes = take((cf.C + 2) * cf.NWP * 8);
    L.vm = take(cf.R * 32 * cf.NA * 4);
    L.first = take(staged ? 0 : cf.R * 4 * 16);
    L.masks = take(3 * cf.NW * 4);
    L.acc = take(2 * pw);
    L.flip = take(10 * pw);
    L.bplanes = take(3 * pw);
    L.basep = take(pw);
    L.lead = take(nw * kMemoBatch * 32 * cf.NA * 4);
    L.match = take(nw * 4 * L.mstride * 4);
    L.queue = take(nw * kSmallSparse * 4);
    L.red = take(8 * 4);
    L.woff = take(cf.C * cf.NW * 2);
    L.raw = take(variant ? cf.R * 32 * cf.NA * 4 : 0);
    L.keys = take(many ? 8 * cf.NA * 32 * 2 : 0);  // (whole words of every lane: all are read)
    L.tab = take(staged ? cf.pk_staged * 4 : 0);
    L.total = at;
    return L;
}

// Whether the packed rule table is copied into shared memory: when the
// environment's region with it still lets six environments share an SM (the
// register budget allows seven); else it is read through the L1 cache.
// AV_MEMO_STAGE=1 (copy) or 0 (do not), read by av_create, forces the choice for
// measurements.
inline bool memo_staged(const DevConfig &cf, bool variant, bool many)
{
    if (cf.pk_staged <= 0 || cf.memo_stage == 2)
        return false;
    const int total = memo_layout(cf, true, variant, many).total;
    if (cf.memo_stage == 1)
        return total <= kDynSmemLimit;
    return total * std::max(1, 24 / memo_warps(cf)) <= 227 * 1024;
}

// Shared memory of one environment, as pointers.
struct MemoSmem {
    uint2 *planes;
    uint32_t *vm;        // [R][NA][32 lanes] valid anchors of the lane's rotation and word
    const uint4 *first;  // [R][rotation] the first batch of terms
    uint32_t *basep, *masks;
    uint32_t *lead;  // this warp's
    SmallOut out;    // the CTA's SET / CLEAR planes, this warp's match planes and queue
    int *red;  // two sets of 4 (alternate evaluations): the step's reward; flags (bit 0: a
               // bit flips, bit 1: a goal tile is left, bit 2: the new board differs from
               // the other slot's, bit 3: no rule has a raw match); the variant step's
               // rules with a raw match
    uint32_t *raw;  // variant step: [R][NA][32 lanes] the rules' raw matches
    uint16_t *keys;  // many matches: the cells' random key parts
    const uint16_t *woff;  // [C * NW] plane entry of flat word i; bit 15: the plane's first
};

// Word x into the doubled planes at entry `at` (as in MemoSmem::woff).
__device__ __forceinline__ void memo_put(uint2 *planes, uint32_t at, uint32_t x)
{
    uint2 *p = planes + (at & 0x7fffu);
    p->x = x;
    if (!(at & 0x8000u))
        p[-1].y = x;
}

// One step of the board in S.planes with action `a`, by all NWARP warps of the
// CTA: the force plane of `a` (each warp writes the same words); every rule in
// its four rotations as in the step-by-step kernels, rule r by warp r mod NWARP:
// the first four terms of up to kMemoBatch rules together, then eight terms per
// vote of those that pass them, and the writes of the matches; then, after a
// barrier, the new board: planes in place, its flips to flip_out and its flat
// planes to bpl_new.  Returns (reward; bit 0: the step changes the board, bit 1: a
// goal tile is left after it, always without a goal channel, bit 2: the new board
// differs from bpl_o, bit 3, variant step: no rule had a raw match), the same in every
// thread, after a second barrier.  The variant step (StepT = VariantParams; key_prefix
// and t make its random keys) has one more barrier, after the raw matches.
template <int NA, bool SM, int NWARP, typename StepT>
static __device__ __forceinline__ int2 memo_step_eval(const DevConfig &cf, const MemoLayout &L, const BlockTable &tb,
                                                       const MemoSmem &S, int a, uint32_t *flip_out,
                                                       uint32_t *bpl_new, const uint32_t *bpl_o, int &parity,
                                                       const StepT &step, uint64_t key_prefix, int t)
{
    constexpr int T = 32 * NWARP;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 3, q = lane & 7;
    const int NW = cf.NW, cnw = cf.C * NW;
    // the reductions alternate between two sets: the set written here was last
    // read two evaluations ago and zeroed in the one in between
    constexpr bool kVariant = std::is_base_of<VariantParams, StepT>::value;
    constexpr bool kMany = std::is_same<StepT, VariantManyParams>::value;
    int *red = S.red + 4 * parity;
    parity ^= 1;
    force_plane(cf, S.planes, S.masks, a);
    __syncwarp();
    const uint32_t pbase = (uint32_t)__cvta_generic_to_shared(S.planes) + q * 8;
    int rew = 0;
    uint64_t raw = 0;  // variant step: this warp's rules with a raw match
    int draws = 0;     // many matches: keys drawn one after another for them
    for (int r0 = warp; r0 < cf.R; r0 += kMemoBatch * NWARP) {
        uint32_t alive = 0;  // bit k: rule r0 + k * NWARP passes its first terms somewhere
        {
            uint32_t m[kMemoBatch][NA];
            uint4 p[kMemoBatch];
#pragma unroll
            for (int k = 0; k < kMemoBatch; ++k) {
                const int r = r0 + k * NWARP;
                if (k > 0 && r >= cf.R)
                    break;
                p[k] = S.first[4 * r + g];
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    m[k][u] = S.vm[(r * NA + u) * 32 + lane];
            }
#pragma unroll
            for (int k = 0; k < kMemoBatch; ++k) {
                if (k > 0 && r0 + k * NWARP >= cf.R)
                    break;
                small_terms<NA>(pbase, p[k], m[k]);  // (a rule without terms has a batch that passes)
                uint32_t any = 0;
#pragma unroll
                for (int u = 0; u < NA; ++u) {
                    any |= m[k][u];
                    S.lead[(k * 32 + lane) * NA + u] = m[k][u];
                }
                alive |= any ? 1u << k : 0u;
            }
            alive = __reduce_or_sync(0xffffffffu, alive);
        }
        for (; alive; alive &= alive - 1) {
            const int k = __ffs(alive) - 1, r = r0 + k * NWARP;
            const uint4 h0 = block_ld<SM>(tb.hdr + 2 * r), h1 = block_ld<SM>(tb.hdr + 2 * r + 1);
            uint32_t m[NA];
#pragma unroll
            for (int u = 0; u < NA; ++u)
                m[u] = S.lead[(k * 32 + lane) * NA + u];
            const uint4 *tp = tb.terms + 4 * h1.x + g;
            bool live = true;
            for (uint32_t b = 1; live && b < h0.x; b += 2) {
                const uint4 p = block_ld<SM>(tp + 4 * (b - 1));
                // (an odd last batch is taken twice)
                const uint4 p2 = block_ld<SM>(tp + 4 * (b + 1 < h0.x ? b : b - 1));
                small_terms<NA>(pbase, p, m);
                small_terms<NA>(pbase, p2, m);
                uint32_t any = 0;
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    any |= m[u];
                live = __any_sync(0xffffffffu, any != 0u);
            }
            if (!live)
                continue;
            int cnt = 0;
#pragma unroll
            for (int u = 0; u < NA; ++u)
                cnt += __popc(m[u]);
            const int total = __reduce_add_sync(0xffffffffu, cnt);
            if constexpr (kVariant) {  // raw matches: which of them apply is decided below
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    S.raw[(r * NA + u) * 32 + lane] = m[u];
                raw |= 1ull << r;
                if (kMany && step.limit[r] > 0)
                    draws += (int)__reduce_max_sync(0xffffffffu, (unsigned)cnt);
                continue;
            }
            rew += (int)h0.z * total;
            small_write<NA, SM>(cf, tb, S.out, h0, h1, m, total);
        }
        __syncwarp();  // the lead anchors may be overwritten
    }
    bool quiet = false;
    if constexpr (kVariant) {
        // every rule with a raw match suppresses the rules of its mask; each rule left
        // applies its matches with the largest keys
        uint32_t *raw_w = reinterpret_cast<uint32_t *>(red) + 2;
        if (lane == 0) {
            if ((uint32_t)raw)
                atomicOr(raw_w, (uint32_t)raw);
            if ((uint32_t)(raw >> 32))
                atomicOr(raw_w + 1, (uint32_t)(raw >> 32));
            if (kMany && draws > kMemoMany)
                atomicOr(red + 1, 16);
        }
        __syncthreads();  // every warp's raw matches
        const uint64_t all = (uint64_t)raw_w[0] | ((uint64_t)raw_w[1] << 32);
        quiet = all == 0;
        bool many = false;
        if constexpr (kMany) {
            many = (red[1] & 16) != 0;
            if (many) {
                for (int p = tid; p < cf.HW; p += T)
                    S.keys[p] = (uint16_t)match_random(key_prefix, t, (uint32_t)p);
                __syncthreads();  // the keys
            }
        }
        uint64_t sup = 0;
        for (uint64_t x = all; x; x &= x - 1u)
            sup |= step.inhibit[__ffsll((long long)x) - 1];
        for (uint64_t x = raw & ~sup; x; x &= x - 1u) {
            const int r = __ffsll((long long)x) - 1, limit = step.limit[r];
            uint32_t m[NA];
            int cnt = 0;
#pragma unroll
            for (int u = 0; u < NA; ++u) {
                m[u] = S.raw[(r * NA + u) * 32 + lane];
                cnt += __popc(m[u]);
            }
            int total = __reduce_add_sync(0xffffffffu, cnt);
            if (limit > 0 && limit < total) {
                if (kMany && many)
                    keep_largest_cells<NA>(m, limit, S.keys);
                else
                    keep_largest<NA>(m, limit, step, key_prefix, t);
                total = limit;
            }
            const uint4 h0 = block_ld<SM>(tb.hdr + 2 * r), h1 = block_ld<SM>(tb.hdr + 2 * r + 1);
            rew += (int)h0.z * total;
            small_write<NA, SM>(cf, tb, S.out, h0, h1, m, total);
        }
    }
    if (rew && lane == 0)
        atomicAdd(red, rew);
    __syncthreads();  // every warp's SET / CLEAR bits and reward
    uint32_t any = 0, goal = 0, diff = 0;
    const int goal0 = cf.ch_goal >= 0 ? cf.ch_goal * NW : cnw;
    for (int i = tid; i < cnw; i += T) {
        const uint32_t at = S.woff[i];
        const uint32_t st = S.out.acc[i], cl = S.out.acc[cnw + i];
        const uint32_t d = S.planes[at & 0x7fffu].x;
        const uint32_t f = (d & cl) | (~d & st), x = d ^ f;  // a bit changes where a match asks for it
        if (st | cl) {
            S.out.acc[i] = 0u;
            S.out.acc[cnw + i] = 0u;
            if (f)
                memo_put(S.planes, at, x);
        }
        flip_out[i] = f;
        bpl_new[i] = x;
        any |= f;
        diff |= bpl_o[i] ^ x;
        if ((uint32_t)(i - goal0) < (uint32_t)NW)
            goal |= x;
    }
    const uint32_t bits = __reduce_or_sync(0xffffffffu, (any ? 1u : 0u) | (goal ? 2u : 0u) | (diff ? 4u : 0u));
    if (bits && lane == 0)
        atomicOr(red + 1, (int)bits);
    if (tid < 4)
        S.red[4 * parity + tid] = 0;  // the set of the next evaluation
    __syncthreads();  // the board after its step, its flips and flags
    const int2 out = *reinterpret_cast<const int2 *>(red);
    return make_int2(out.x, out.y | (cf.ch_goal < 0 ? 2 : 0) | (quiet ? 8 : 0));
}

// The board after a remembered step (planes ^= flip), written also into bpl_new
// (flat), in one pass (all warps); returns whether it differs from bpl_o (every
// thread).
template <int NWARP>
static __device__ __forceinline__ int memo_apply(const MemoSmem &S, int cnw, const uint32_t *flip, uint32_t *bpl_new,
                                                  const uint32_t *bpl_o)
{
    uint32_t diff = 0;
    for (int i = threadIdx.x; i < cnw; i += 32 * NWARP) {
        const uint32_t at = S.woff[i], f = flip[i], x = S.planes[at & 0x7fffu].x ^ f;
        if (f)
            memo_put(S.planes, at, x);
        diff |= bpl_o[i] ^ x;
        bpl_new[i] = x;
    }
    return __syncthreads_or(diff != 0u);
}

// Auto-reset: the initial map's planes into the tile planes and bpl_new (all
// warps).  Returns bit 0: the map differs from bpl_c, the board before the step;
// bit 1: from bpl_o (every thread).
template <int NWARP>
static __device__ __forceinline__ int memo_restore(const MemoSmem &S, int cnw, uint32_t *bpl_new,
                                                    const uint32_t *bpl_c, const uint32_t *bpl_o)
{
    uint32_t dc = 0, dn = 0;
    for (int i = threadIdx.x; i < cnw; i += 32 * NWARP) {
        const uint32_t at = S.woff[i], b = S.basep[i];
        if (S.planes[at & 0x7fffu].x != b)
            memo_put(S.planes, at, b);
        dc |= bpl_c[i] ^ b;
        dn |= bpl_o[i] ^ b;
        bpl_new[i] = b;
    }
    const int changed = __syncthreads_or(dc != 0u);
    return changed ? 1 | (__syncthreads_or(dn != 0u) ? 2 : 0) : 0;
}

template <typename T>
__device__ __forceinline__ void swap_vals(T &a, T &b)
{
    const T t = a;
    a = b;
    b = t;
}

// Fused rollout, one CTA of NWARP warps per environment; see the top of this
// file.  With `actions` non-null the action of every step is actions[env]
// (av_step, n_steps = 1); else step s draws draw(seed, 4, env, 0, s) mod 5.
//
// What bounds it: instruction issue, three quarters of it bookkeeping rather than
// matching, and for few environments the latency of a step on the one that
// changes its board most often.  500 steps of 16,384 16 x 16 boards with
// trajectories: 3.97 ms with seven barriers per evaluation and outputs written
// entry by entry, 3.28 with two, 2.92 with the layout's offsets passed in, one
// lookup per plane word and the step at hand looked up before a whole run (1000
// steps of 1024 boards under a moving player: 2.51, 1.49, 1.30 ms).  Walking on
// warp 0 alone, the others waiting for its commands, takes fewer instructions but
// lengthens each busy environment's chain: 3.57 and 1.34 ms.  Four warps: 72
// registers a thread, seven CTAs per SM (64 spill; six cost 3 %).
template <typename CellT, int NA, bool SM, int NWARP, typename StepT>
__global__ void __launch_bounds__(32 * NWARP, 28 / NWARP)
rollout_memo_kernel(const __grid_constant__ DevConfig cf, const __grid_constant__ MemoLayout L,
                    const __grid_constant__ StepT step, const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g, CellT *cur,
                    const CellT *__restrict__ init, int32_t *tsteps, int n_steps, uint64_t seed,
                    const uint8_t *__restrict__ actions, CellT *obs_traj, int32_t *rew_traj,
                    uint8_t *done_traj, int32_t *rew_sum, uint32_t *status, const int32_t *__restrict__ order,
                    uint32_t *cost)
{
    constexpr int T = 32 * NWARP;
    extern __shared__ __align__(16) unsigned char smem[];
    const long long clock0 = clock64();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int env = order ? order[blockIdx.x] : (int)blockIdx.x;
    const int C = cf.C, NW = cf.NW, NWP = cf.NWP, HW = cf.HW, cnw = C * NW;
    const int nbytes = HW * (int)sizeof(CellT);
    MemoSmem S;
    S.planes = reinterpret_cast<uint2 *>(smem + L.planes);
    S.out.acc = reinterpret_cast<uint32_t *>(smem + L.acc);
    S.basep = reinterpret_cast<uint32_t *>(smem + L.basep);
    S.vm = reinterpret_cast<uint32_t *>(smem + L.vm);
    S.masks = reinterpret_cast<uint32_t *>(smem + L.masks);
    S.lead = reinterpret_cast<uint32_t *>(smem + L.lead) + warp * kMemoBatch * 32 * NA;
    S.out.match = reinterpret_cast<uint32_t *>(smem + L.match) + warp * 4 * L.mstride;
    S.out.queue = reinterpret_cast<uint32_t *>(smem + L.queue) + warp * kSmallSparse;
    S.red = reinterpret_cast<int *>(smem + L.red);
    S.out.pad = L.pad;
    S.out.mstride = L.mstride;
    S.woff = reinterpret_cast<const uint16_t *>(smem + L.woff);
    const int table = cf.rules_per_env ? env : 0;
    const uint32_t *pk = cf.pk + cf.pk_off[table];
    uint32_t *const tab_s = reinterpret_cast<uint32_t *>(smem + L.tab);

    // ---- stage
    const BlockTable tb = block_table(SM ? tab_s : pk, __ldg(reinterpret_cast<const uint4 *>(pk)), cf.R);
    if (SM) {
        const uint32_t n = (cf.pk_off[table + 1] - cf.pk_off[table]) / 4;
        for (uint32_t i = tid; i < n; i += T)
            reinterpret_cast<uint4 *>(tab_s)[i] = __ldg(reinterpret_cast<const uint4 *>(pk) + i);
    }
    {
        // (read from global memory: the staged table is not complete yet)
        const BlockTable tg = block_table(pk, __ldg(reinterpret_cast<const uint4 *>(pk)), cf.R);
        for (int i = tid; i < cf.R * 32 * NA; i += T) {
            const int l = i & 31, r = i / (32 * NA), word = (l & 7) + 8 * ((i >> 5) % NA);
            const uint32_t shape = (__ldg(&tg.hdr[2 * r].w) >> (l & 24)) & 0xffu;  // byte l >> 3
            S.vm[i] = word < NW ? __ldg(vm_g + shape * NW + word) : 0u;
        }
        S.first = SM ? tb.terms : reinterpret_cast<const uint4 *>(smem + L.first);
        if (!SM)  // every rule's first batch heads the terms
            for (int i = tid; i < 4 * cf.R; i += T)
                reinterpret_cast<uint4 *>(smem + L.first)[i] = __ldg(tg.terms + i);
    }
    constexpr bool kVariant = std::is_base_of<VariantParams, StepT>::value;
    uint64_t key_prefix = 0;
    if constexpr (kVariant) {
        S.raw = reinterpret_cast<uint32_t *>(smem + L.raw);
        S.keys = reinterpret_cast<uint16_t *>(smem + L.keys);
        key_prefix = variant_prefix(step, env);
    }
    if (tid < 8)
        S.red[tid] = 0;
    for (int i = tid; i < cnw; i += T) {
        const int c = i / NW, w = i - c * NW;
        reinterpret_cast<uint16_t *>(smem + L.woff)[i] = (uint16_t)((c * NWP + w) | (w ? 0 : 0x8000));
    }
    for (int i = tid; i < 3 * NW; i += T)
        S.masks[i] = __ldg(masks_g + i);
    for (int i = tid; i < (C + 2) * NWP; i += T)
        S.planes[i] = make_uint2(0u, 0u);
    for (int i = tid; i < 2 * cnw; i += T)
        S.out.acc[i] = 0u;
    for (int i = lane; i < 4 * L.mstride; i += 32)
        S.out.match[i] = 0u;
    uint32_t *bpl_c = reinterpret_cast<uint32_t *>(smem + L.bplanes), *bpl_o = bpl_c + cnw, *bpl_n = bpl_o + cnw;
    {
        // the initial map's planes, flat: a byte per channel and eight cells
        uint8_t *fb = reinterpret_cast<uint8_t *>(S.basep);
        for (int i = tid; i < cnw; i += T)
            S.basep[i] = 0u;
        __syncthreads();  // the zeroed planes
        const CellT *src = cur + (size_t)env * HW, *isrc = init + (size_t)env * HW;
        const bool vec = cells8_aligned(src, HW), ivec = cells8_aligned(isrc, HW);
        for (int b = tid; 8 * b < HW; b += T) {
            put_cells8<CellT>(cf, src, b, vec, S.planes);
            uint32_t x[4];
            load_cells8<CellT>(isrc, HW, b, ivec, x[0], x[1], x[2], x[3]);
#pragma unroll
            for (int c = 0; c < 8 * (int)sizeof(CellT); ++c) {
                if (c >= C)
                    break;
                fb[c * NW * 4 + b] = (uint8_t)(x[c >> 2] >> (8 * (c & 3)));
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < cnw; i += T)
        bpl_c[i] = S.planes[S.woff[i] & 0x7fffu].x;

    // Two board slots: the current board and the one before it.  Per slot: the
    // board's planes (flat) and the outcomes remembered for it, in registers the
    // same in every warp: bit a of kq when action a leaves the board unchanged, of
    // kc when it changes it (its flip planes kept in flip_c[a]), of gm when a goal
    // tile is left after it; lane a holds its reward in rw.  The o-names belong to
    // the other slot.  A new board is made in a third set of flat planes, which
    // joins the slots when it becomes the current one.
    uint32_t *flip_c = reinterpret_cast<uint32_t *>(smem + L.flip), *flip_o = flip_c + 5 * cnw;
    uint32_t kq = 0u, kc = 0u, gm = 0u, okq = 0u, okc = 0u, ogm = 0u;
    int rw = 0, orw = 0;
    bool valid_other = false;
    int parity = 0;  // which set of reduction slots the next evaluation uses
    // This lane's cells of the board, made by each warp when it first stores them
    // (a warp of a board that changes every step stores every NWARP-th).
    SmallCells<CellT, NA> v;
    bool have_v = false;
    int t = tsteps[env];
    int sum = 0, warn = 0;
    const int obs_mode = obs_traj ? small_store_mode<CellT, false>(obs_traj, nbytes) : 0;
    const size_t step_stride = (size_t)cf.B * nbytes;  // bytes from one step's boards to the next's
    unsigned char *const obs_env = obs_traj ? reinterpret_cast<unsigned char *>(obs_traj) + (size_t)env * nbytes
                                            : nullptr;
    __syncthreads();  // bpl_c

    for (int b0 = 0; b0 < n_steps; b0 += 32) {
        const int lim = min(32, n_steps - b0);
        const int a_l = lane < lim ? action_at(actions, seed, env, b0 + lane, &warn) : 0;
        int l0 = 0;
        while (l0 < lim) {
            // the step at hand is a plain repeat unless its action has no
            // remembered outcome that leaves the board as it is, or it ends in an
            // auto-reset
            int e = l0;
            const int a0 = __shfl_sync(0xffffffffu, a_l, l0);
            if ((kq >> a0) & 1u) {
                // lane l takes step b0 + l as if every step of this run before it
                // were a plain repeat; the first that is not ends the run
                const bool act = lane >= l0 && lane < lim;
                const bool q_l = (kq >> a_l) & 1u;
                const int r_l = __shfl_sync(0xffffffffu, rw, a_l);
                const bool goal_l = (gm >> a_l) & 1u;
                const int t_l = t + (lane - l0) + 1;
                const bool done_l = !goal_l || (cf.max_steps > 0 && t_l >= cf.max_steps);
                const uint32_t ev = __ballot_sync(0xffffffffu, act && (!q_l || (done_l && cf.auto_reset)));
                e = ev ? __ffs(ev) - 1 : lim;
                if (warp == 0 && act && lane < e) {
                    sum += r_l;
                    if (rew_traj)
                        rew_traj[(size_t)(b0 + lane) * cf.B + env] = r_l;
                    if (done_traj)
                        done_traj[(size_t)(b0 + lane) * cf.B + env] = (uint8_t)done_l;
                }
                if (obs_traj && l0 + warp < e) {  // the warps take turns
                    if (!have_v) {
                        small_cells<CellT, NA>(cf, S.planes, v);
                        have_v = true;
                    }
                    unsigned char *o = obs_env + (size_t)(b0 + l0 + warp) * step_stride;
                    for (int l = l0 + warp; l < e; l += NWARP, o += NWARP * step_stride)
                        small_store<CellT, NA, false>(o, v, nbytes, obs_mode);
                }
                t += e - l0;
                if (e >= lim)
                    break;
            }

            // ---- step b0 + e (every warp)
            const int a = e == l0 ? a0 : __shfl_sync(0xffffffffu, a_l, e);
            const uint32_t bit = 1u << a;
            uint32_t *fl = flip_c + a * cnw;  // flip planes of the current board and action a
            int r;
            bool goal_left, moves;       // moves: the step's own outcome changes the board
            bool made = false, diff_o = false;  // the new board is in the planes and bpl_n; it differs from bpl_o
            if ((kq | kc) & bit) {  // remembered: the board stays (and an auto-reset follows), or changes
                r = __shfl_sync(0xffffffffu, rw, a);
                goal_left = (gm & bit) != 0u;
                moves = (kc & bit) != 0u;
                if (obs_traj)
                    __syncthreads();  // every warp has made the cells of the board it has still to store
            } else {
                const int2 o = memo_step_eval<NA, SM, NWARP, StepT>(cf, L, tb, S, a, fl, bpl_n, bpl_o, parity, step,
                                                                    key_prefix, t);
                r = o.x;
                goal_left = (o.y & 2) != 0;
                moves = (o.y & 1) != 0;
                if (lane == a)
                    rw = r;
                gm = goal_left ? gm | bit : gm & ~bit;
                if (!moves && (!kVariant || (o.y & 8))) {  // the board stays: remember, take the step again
                    kq |= bit;
                    l0 = e;
                    continue;
                }
                if (!kVariant)
                    kc |= bit;
                made = true;
                diff_o = (o.y & 4) != 0;
            }
            t += 1;
            const bool done = !goal_left || (cf.max_steps > 0 && t >= cf.max_steps);
            bool changed;
            if (done && cf.auto_reset) {
                const int d = memo_restore<NWARP>(S, cnw, bpl_n, bpl_c, bpl_o);
                changed = (d & 1) != 0;
                diff_o = (d & 2) != 0;
                t = 0;
            } else {  // (a board-changing outcome: `moves` holds)
                if (!made)
                    diff_o = memo_apply<NWARP>(S, cnw, fl, bpl_n, bpl_o) != 0;
                changed = moves;
            }
            if (warp == 0 && lane == e) {
                sum += r;
                if (rew_traj)
                    rew_traj[(size_t)(b0 + e) * cf.B + env] = r;
                if (done_traj)
                    done_traj[(size_t)(b0 + e) * cf.B + env] = (uint8_t)done;
            }
            if (changed) {
                // the new board becomes the current one and the current the other:
                // if the other slot held the same board, its remembered outcomes
                // hold; else they are dropped
                const bool same = !diff_o && valid_other;
                swap_vals(bpl_c, bpl_o);
                swap_vals(flip_c, flip_o);
                swap_vals(kq, okq);
                swap_vals(kc, okc);
                swap_vals(gm, ogm);
                swap_vals(rw, orw);
                if (!same) {
                    kq = kc = gm = 0u;
                    swap_vals(bpl_c, bpl_n);
                }
                valid_other = true;
                have_v = false;
            }
            if (obs_traj && warp == (e % NWARP)) {
                if (!have_v) {
                    small_cells<CellT, NA>(cf, S.planes, v);
                    have_v = true;
                }
                small_store<CellT, NA, false>(obs_env + (size_t)(b0 + e) * step_stride, v, nbytes, obs_mode);
            }
            l0 = e + 1;
        }
    }
    if (warp == 0) {
        if (!have_v)
            small_cells<CellT, NA>(cf, S.planes, v);
        small_store<CellT, NA, false>(reinterpret_cast<unsigned char *>(cur) + (size_t)env * nbytes, v, nbytes,
                              small_store_mode<CellT, false>(cur, nbytes));
        sum = __reduce_add_sync(0xffffffffu, sum);
        warn = __any_sync(0xffffffffu, warn);
        if (lane == 0) {
            tsteps[env] = t;
            if (rew_sum)
                rew_sum[env] = sum;
            if (warn)
                atomicOr(status + 1, kWarnAction);
            if (cost)  // this launch's time for the environment, in units of 256 cycles
                cost[env] = (uint32_t)min((clock64() - clock0) >> 8, 0xffffffffLL);
        }
    }
}

#ifdef AV_MEMO_ORDER
// Launch order of the next memoising rollout (one CTA): environments by
// decreasing cost in the last launch, in power-of-two buckets (a counting
// sort; the order within a bucket is arbitrary).  Started first, the costly
// environments no longer finish after everything else.
__global__ void __launch_bounds__(1024) memo_order_kernel(const uint32_t *__restrict__ cost, int32_t *order, int B)
{
    __shared__ int hist[33], next[33];
    const int tid = threadIdx.x;
    if (tid < 33)
        hist[tid] = 0;
    __syncthreads();
    for (int i = tid; i < B; i += blockDim.x)
        atomicAdd(&hist[32 - __clz(cost[i])], 1);
    __syncthreads();
    if (tid == 0) {
        int s = 0;
        for (int b = 32; b >= 0; --b) {
            next[b] = s;
            s += hist[b];
        }
    }
    __syncthreads();
    for (int i = tid; i < B; i += blockDim.x)
        order[atomicAdd(&next[32 - __clz(cost[i])], 1)] = i;
}

void launch_memo_order(const uint32_t *cost, int32_t *order, int B, cudaStream_t st)
{
    memo_order_kernel<<<1, 1024, 0, st>>>(cost, order, B);
}
#endif

}  // namespace av

// ---------------------------------------------------------------- launchers
// Compiled once per cell type and step (AV_MEMO_CELL, AV_MEMO_STEP) by k_memo_u8.cu,
// k_memo_u16.cu, k_vmemo_u8.cu, k_vmemo_u16.cu, k_vmany_u8.cu and k_vmany_u16.cu.
#ifdef AV_MEMO_CELL
namespace av {
namespace {

constexpr bool kMemoVariant = std::is_base_of<VariantParams, AV_MEMO_STEP>::value;
constexpr bool kMemoManyStep = std::is_same<AV_MEMO_STEP, VariantManyParams>::value;

template <int NA, bool SM, int NWARP, typename... Args>
void memo_launch(const DevConfig &cf, const AV_MEMO_STEP &step, cudaStream_t st, Args... args)
{
    const MemoLayout L = memo_layout(cf, SM, kMemoVariant, kMemoManyStep);
    rollout_memo_kernel<AV_MEMO_CELL, NA, SM, NWARP, AV_MEMO_STEP><<<cf.B, 32 * NWARP, L.total, st>>>(cf, L, step,
                                                                                                    args...);
}

template <int NA, bool SM, typename... Args>
void memo_warps_launch(const DevConfig &cf, const AV_MEMO_STEP &step, cudaStream_t st, Args... args)
{
    switch (memo_warps(cf)) {
    case 1: return memo_launch<NA, SM, 1>(cf, step, st, args...);
    case 2: return memo_launch<NA, SM, 2>(cf, step, st, args...);
    case 8: return memo_launch<NA, SM, 8>(cf, step, st, args...);
    }
    memo_launch<NA, SM, 4>(cf, step, st, args...);
}

template <typename... Args>
void memo_any_launch(const DevConfig &cf, const AV_MEMO_STEP &step, cudaStream_t st, Args... args)
{
    if (memo_staged(cf, kMemoVariant, kMemoManyStep)) {
        if (cf.NA == 1)
            memo_warps_launch<1, true>(cf, step, st, args...);
        else
            memo_warps_launch<2, true>(cf, step, st, args...);
    } else {
        if (cf.NA == 1)
            memo_warps_launch<1, false>(cf, step, st, args...);
        else
            memo_warps_launch<2, false>(cf, step, st, args...);
    }
}

template <int NWARP>
cudaError_t memo_configure(cudaError_t e)
{
    auto set = [&](auto *fn) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute((const void *)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    };
    set(rollout_memo_kernel<AV_MEMO_CELL, 1, true, NWARP, AV_MEMO_STEP>);
    set(rollout_memo_kernel<AV_MEMO_CELL, 1, false, NWARP, AV_MEMO_STEP>);
    set(rollout_memo_kernel<AV_MEMO_CELL, 2, true, NWARP, AV_MEMO_STEP>);
    set(rollout_memo_kernel<AV_MEMO_CELL, 2, false, NWARP, AV_MEMO_STEP>);
    return e;
}

}  // namespace

cudaError_t AV_MEMO_CONFIGURE()
{
    cudaError_t e = memo_configure<4>(cudaSuccess);
    e = memo_configure<1>(e);
    e = memo_configure<2>(e);
    e = memo_configure<8>(e);
    return e;
}

#ifdef AV_MEMO_VARIANT
// Warps per environment of the variant step.  Four; fewer where the batch fills the GPU
// (about 28 warps an SM) without them and a warp still has few rules, since each CTA's
// setup and barriers take its slots whatever it has to do; eight for the most rules,
// whose keys are drawn rule by rule.  us with the kernels that four warps for every
// board replaced (one warp or one CTA of eight), and with 1 / 2 / 4 / 8 warps:
//   16384 x 5 x 5, 2 rules, one step        47.5:   34.8 /  64.2 /  99.0 /  213
//   16384 x 16 x 16, 3 rules, 100 steps     1974:    961 /  1562 /  2402 / 4913
//   16384 x 16 x 16, 16 rules, 8 steps      1485:    884 /   704 /   810 / 1380
//   4096 x 16 x 16, 8 rules, 100 steps       823:    387 /   334 /   417 /  748
//   1500 x 16 x 16, 3 rules, 100 steps       515:    290 /   291 /   338 /  537
//   2048 x 16 x 16, 4 rules, 100 steps       886:    699 /   614 /   490 /  749
//   700 x 16 x 16, 8 rules, 100 steps        290:    243 /   172 /   162 /  186
//   2048 x 16 x 32, 64 rules, 100 steps     6981:  19918 / 12196 /  8397 / 6910
//   64 x 16 x 16, 64 rules, 100 steps       1549:   3891 /  2294 /  1454 / 1050
// In long rollouts the environments that change their board most decide the end, and
// more warps shorten theirs: the lines lie higher there.
inline int variant_warps(const DevConfig &cf, int n_steps)
{
    constexpr long long kFull = 152 * 28;  // warps on the GPU at a time
    const int work = cf.R * cf.NA;         // rules, and words of a lane
    const bool longer = n_steps >= 32;
    if (work > (longer ? 64 : 96) || (work >= 64 && cf.B * 8LL <= kFull))
        return 8;
    int w = 4;
    for (; w > 1; w /= 2) {
        const int share = work / (w / 2);  // a warp's at half as many
        const int waves = share > 4 ? (longer ? 4 : 2) : longer && share > 1 ? 3 : 1;
        if (share > 8 || cf.B * (long long)w <= waves * kFull)
            break;
    }
    return w;
}

void AV_MEMO_LAUNCH(const DevConfig &cf, const AV_MEMO_STEP &vp, const uint32_t *vm, const uint32_t *masks, void *cur,
                    const void *init, int32_t *t, int n_steps, uint64_t seed, const uint8_t *actions, void *obs_traj,
                    int32_t *rew_traj, uint8_t *done_traj, int32_t *rew_sum, uint32_t *status, cudaStream_t st)
{
    DevConfig c = cf;
    if (cf.memo_warps == 0)
        c.memo_warps = variant_warps(cf, n_steps);
    memo_any_launch(c, vp, st, vm, masks, (AV_MEMO_CELL *)cur, (const AV_MEMO_CELL *)init, t, n_steps, seed, actions,
                    (AV_MEMO_CELL *)obs_traj, rew_traj, done_traj, rew_sum, status, (const int32_t *)nullptr,
                    (uint32_t *)nullptr);
}
#else
void AV_MEMO_LAUNCH(const DevConfig &cf, const uint32_t *vm, const uint32_t *masks, void *cur, const void *init,
                    int32_t *t, int n_steps, uint64_t seed, const uint8_t *actions, void *obs_traj, int32_t *rew_traj,
                    uint8_t *done_traj, int32_t *rew_sum, uint32_t *status, const int32_t *order, uint32_t *cost,
                    cudaStream_t st)
{
    memo_any_launch(cf, StandardStep{}, st, vm, masks, (AV_MEMO_CELL *)cur, (const AV_MEMO_CELL *)init, t, n_steps,
                    seed, actions, (AV_MEMO_CELL *)obs_traj, rew_traj, done_traj, rew_sum, status, order, cost);
}
#endif

}  // namespace av
#endif
