// block_step.cuh -- one step's rule matching and output writes by a CTA of
// kThreads, shared by the block rollout, the band rollout and the CTA-per-parent
// expansion (boards or bands of up to 128 plane words).
//
// Two phases per chunk of rules, with a block barrier between them:
//   match: units of (rule, 32 plane words) dealt to warps; lane = rotation x
//     anchor word (four words a lane), four terms per vote.  A unit's few
//     matches go to a queue; the anchors of a unit with more than kBlkSparse go to the chunk's
//     match planes [rule][rotation][word] in shared memory.
//   write: queued matches dealt to warps, lane = output bit of the rule (one
//     shared atomic each); and units of (rule with match planes, output entry, 32
//     plane words), lane = destination word, which gathers the entry's anchors
//     from the four rotations' match planes (a funnel shift each), ORs them
//     together and then into the SET / CLEAR words of the entry's channels.
// What bounds it: instruction issue and, before, the busiest warp.  With one
// warp per rule that scattered every anchor word by shared atomics (two per
// rotation, channel and word), a rule that matched cost its warp ten times a
// rule that did not, and the other warps waited at the barrier (7.5 stalled
// cycles per issue on 64 x 64 boards with 24 rules that fire).  Dealing both
// phases out in small units levels the warps, and gathering needs one atomic per
// (channel, word) instead of eight.
//
// Packed rule tables (one per table, built by av_create beside the term lists):
// four words (batches, outputs, output bits and force terms in all), per rule eight
// words (batches, outputs | force terms << 8 | first force term << 16, reward,
// shapes; second batch, first output, first output bit,
// output bits | i << 16, where (l * i) >> 11 = l / output bits for l <= 32 when
// there are at most 32 of them), then
//   terms  [batch][rotation][4], every rule's first batch, then rule by rule the
//          others, 32 bits each: plane byte offset << 16 | 0x8000
//          for an absent term | shift; a rule has at least one batch, and its last
//          is filled up with terms that read the zero plane as absent and pass
//   outs   [output][rotation], 32 bits each: word offset << 8 | shift
//   masks  [output]: set channels | clear channels << 16
//   forces [force term][rotation]: the rules' terms on the force plane once more
//   obits  [output bit], 16 bits each: output | (channel, or C + channel for
//          CLEAR) << 8
#pragma once

#include "launch.h"

namespace av {

constexpr int kBlkRules = 8;      // rules per chunk at most
constexpr int kBlkSparse = 16;    // matches of a unit that go to the queue at most

// Sizes of the match planes for boards (or bands) of nw plane words, w cells wide.
struct BlockShape {
    int nw;       // plane words
    int lg;       // log2 of the 32-word groups
    int pad;      // zero words in front of each rotation's match words
    int mstride;  // words per rotation
    int rc;       // rules per chunk
};

__host__ __device__ inline BlockShape block_shape(int nw, int w, int R)
{
    BlockShape b;
    b.nw = nw;
    b.lg = nw <= 32 ? 0 : nw <= 64 ? 1 : 2;
    // the farthest source word of a destination word: a 5 x 5 window's last
    // offset, 4w + 4 cells, and one more for the shifted-in bits
    b.pad = ((4 * w + 4) / 32 + 1 + 7) & ~7;
    b.mstride = (32 << b.lg) + b.pad;
    b.rc = R < kBlkRules ? (R < 1 ? 1 : R) : kBlkRules;
    return b;
}

constexpr int kBlkCtas = 3;  // CTAs of kThreads per SM that the kernels are compiled for (and one more: block_ctas)

// Shared memory of one child's canonical bytes (whole units of eight cells, 16-byte aligned).
__host__ __device__ inline int block_child_bytes(int HW, int cell_bytes) { return (HW * cell_bytes + 15) & ~15; }

struct BlockLayout {
    size_t planes, setp, match, queue, keep, ctl, acts, tab, cells, total;
};

// Control words: 0..7 per-warp rewards, then the names below.
enum {
    kCtlLive = 8,      // three words: bit 4r + k, group k of rule r has match planes (slots taken in turn)
    kCtlQueued = 11,   // three words: matches queued (slots taken in turn)
    kCtlBits = 14,     // two words: bit 0 a cell changed, bit 1 a goal tile is left (slots taken in turn)
    kCtlWarn = 16,     // an action above 4 was seen
    kCtlKnown = 17,    // bit a: the step with action a is remembered to leave the board as it is
    kCtlAct = 18,      // the coming step's action
    kCtlRun = 19,      // length of a run of repeated steps
    kCtlNext = 20,     // the action after a run
    kCtlRew = 21,      // five remembered rewards
    kCtlWords = 28,
};

// planes (C tiles, force, a zero plane that padding terms read) | SET, then
// CLEAR | match planes | queue | the band's anchor mask (bands only) | control |
// actions | packed table when staged | child cells (expansion)
__host__ __device__ inline BlockLayout block_layout(const DevConfig &cf, const BlockShape &bs, int keep_words,
                                                    int n_cell_boards)
{
    BlockLayout L;
    const size_t pw = (size_t)cf.C * bs.nw * 4;
    L.planes = 0;
    L.setp = align16((size_t)(cf.C + 2) * cf.NWP * 8);
    L.match = align16(L.setp + 2 * pw);
    L.queue = align16(L.match + (size_t)bs.rc * 4 * bs.mstride * 4);
    L.keep = align16(L.queue + (size_t)bs.rc * 4 * kBlkSparse * 4);  // (at most 4 units a rule)
    L.ctl = align16(L.keep + (size_t)keep_words * 4);
    L.acts = align16(L.ctl + (size_t)kCtlWords * 4);
    L.tab = align16(L.acts + kActChunk);
    L.cells = align16(L.tab + (size_t)cf.pk_staged * 4);
    L.total = align16(L.cells + (size_t)n_cell_boards * block_child_bytes(cf.HW, cf.cell_bytes));
    return L;
}

// The rules per chunk that let the most CTAs (up to kBlkCtas) share an SM, the
// larger of equals: 64 x 64 boards with 24 rules and 17 KB of packed table fit
// three CTAs with six rules a chunk and two with eight (100 steps of 4096: 20.7 ms
// with three CTAs, 26.6 with two).
inline BlockShape block_shape_fit(const DevConfig &cf, int nw, int keep_words, int n_cell_boards)
{
    BlockShape best = block_shape(nw, cf.W, cf.R);
    const int top = best.rc;
    int most = 0;
    for (int rc = top; rc >= 1 && rc >= top - 4; rc -= 2) {
        BlockShape b = best;
        b.rc = rc;
        const size_t total = block_layout(cf, b, keep_words, n_cell_boards).total + 1024;
        const int ctas = (int)(228 * 1024 / total);
        const int fit = ctas < kBlkCtas ? ctas : kBlkCtas;
        if (fit > most) {
            most = fit;
            best.rc = rc;
        }
    }
    return best;
}

struct BlockSmem {
    uint2 *planes;
    uint32_t *setp, *clrp, *match, *queue, *keep;
    int *ctl;
    uint8_t *acts;
    uint32_t *tab;
    unsigned char *cells;  // expansion: the children's canonical bytes
};

__device__ __forceinline__ BlockSmem block_carve(unsigned char *smem, const BlockLayout &L, const DevConfig &cf,
                                                 const BlockShape &bs)
{
    BlockSmem S;
    S.planes = reinterpret_cast<uint2 *>(smem + L.planes);
    S.setp = reinterpret_cast<uint32_t *>(smem + L.setp);
    S.clrp = S.setp + cf.C * bs.nw;
    S.match = reinterpret_cast<uint32_t *>(smem + L.match);
    S.queue = reinterpret_cast<uint32_t *>(smem + L.queue);
    S.keep = reinterpret_cast<uint32_t *>(smem + L.keep);
    S.ctl = reinterpret_cast<int *>(smem + L.ctl);
    S.acts = smem + L.acts;
    S.tab = reinterpret_cast<uint32_t *>(smem + L.tab);
    S.cells = smem + L.cells;
    return S;
}

// The packed table in use: shared memory when staged, else global memory.
struct BlockTable {
    const uint4 *hdr;      // [R][2]
    const uint4 *terms;    // [batch][rotation]
    const uint4 *outs;     // [output], word g = rotation g
    const uint32_t *masks; // [output]
    const uint32_t *forces; // [force term][rotation]
    const uint16_t *obits; // [output bit]
};

__device__ __forceinline__ BlockTable block_table(const uint32_t *t, const uint4 &counts, int R)
{
    BlockTable b;
    b.hdr = reinterpret_cast<const uint4 *>(t) + 1;
    b.terms = b.hdr + 2 * R;
    b.outs = b.terms + 4 * counts.x;
    b.masks = reinterpret_cast<const uint32_t *>(b.outs + counts.y);
    b.forces = b.masks + counts.y;
    b.obits = reinterpret_cast<const uint16_t *>(b.forces + 4 * counts.w);
    return b;
}

template <bool SM, typename T>
__device__ __forceinline__ T block_ld(const T *p)
{
    return SM ? *p : __ldg(p);
}

// Zero the planes, SET / CLEAR, match planes and control words, and copy the
// packed table of `table` when it is staged.  Returns the table to use.
template <bool SM>
__device__ __forceinline__ BlockTable block_stage(const DevConfig &cf, const BlockShape &bs, const BlockSmem &S,
                                                  int table)
{
    const int tid = threadIdx.x;
    for (int i = tid; i < (cf.C + 2) * cf.NWP; i += kThreads)
        S.planes[i] = make_uint2(0u, 0u);
    for (int i = tid; i < cf.C * bs.nw; i += kThreads) {
        S.setp[i] = 0u;
        S.clrp[i] = 0u;
    }
    for (int i = tid; i < bs.rc * 4 * bs.mstride; i += kThreads)
        S.match[i] = 0u;
    if (tid < kCtlWords)
        S.ctl[tid] = 0;
    const uint32_t *pk = cf.pk + cf.pk_off[table];
    if (SM) {
        const uint32_t n = (cf.pk_off[table + 1] - cf.pk_off[table]) / 4;
        for (uint32_t i = tid; i < n; i += kThreads)
            reinterpret_cast<uint4 *>(S.tab)[i] = __ldg(reinterpret_cast<const uint4 *>(pk) + i);
    }
    return block_table(SM ? S.tab : pk, __ldg(reinterpret_cast<const uint4 *>(pk)), cf.R);
}

// All ones when a term is absent (bit 15: the sign of byte 1), else zero.
__device__ __forceinline__ uint32_t block_neg(uint32_t term)
{
    uint32_t n;
    asm("prmt.b32 %0, %1, 0, 0x9999;" : "=r"(n) : "r"(term));
    return n;
}

// All warps: every rule in its four rotations on the planes in S, the outputs of
// the matches ORed into SET / CLEAR.  The valid-anchor masks are vm_g [shape]
// [vm_nw] from word w0 on, ANDed with S.keep[word] when KEEP (a band's own
// anchors).  `slot` counts the chunks so far (kept by the caller across calls).
// Returns whether any rule matched (block-uniform; then the last thing done was
// a barrier after every SET / CLEAR write) and adds the rewards of this warp's
// units to warp_rew (the same in every lane).
template <bool SM, bool KEEP>
__device__ __forceinline__ bool block_match(const DevConfig &cf, const BlockShape &bs, const BlockTable &tb,
                                            const BlockSmem &S, const uint32_t *__restrict__ vm_g, int vm_nw, int w0,
                                            int &slot, int &warp_rew)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    const int lg = bs.lg, gmask = (1 << lg) - 1, R = cf.R;
    const uint32_t planes = (uint32_t)__cvta_generic_to_shared(S.planes);
    const uint32_t below = (1u << lane) - 1u;
    int rew = 0;
    bool any = false;
    for (int r0 = 0; r0 < R; r0 += bs.rc) {
        const int nr = min(bs.rc, R - r0);
        int *live_w = S.ctl + kCtlLive + slot, *queued_w = S.ctl + kCtlQueued + slot;
        // ---- match
        for (int u = warp; u < nr << lg; u += kWarps) {
            const int rr = u >> lg, k = u & gmask;
            const uint4 h0 = block_ld<SM>(tb.hdr + 2 * (r0 + rr)), h1 = block_ld<SM>(tb.hdr + 2 * (r0 + rr) + 1);
            const int word = 32 * k + q;
            const uint32_t *vmr = vm_g + (size_t)((h0.w >> (8 * g)) & 0xffu) * vm_nw + w0 + word;
            uint32_t m[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                m[v] = word + 8 * v < bs.nw && (!KEEP || w0 + word + 8 * v < vm_nw) ? __ldg(vmr + 8 * v) : 0u;
                if (KEEP)
                    m[v] &= word + 8 * v < bs.nw ? S.keep[word + 8 * v] : 0u;
            }
            const uint4 *tp = tb.terms + g;
            const uint32_t base = planes + 8 * word;
            bool alive = __any_sync(0xffffffffu, (m[0] | m[1] | m[2] | m[3]) != 0u);
            for (uint32_t b = 0; alive && b < h0.x; ++b) {
                const uint4 p = block_ld<SM>(tp + 4 * (b ? h1.x + b - 1 : r0 + rr));
                const uint32_t pj[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t a = base + (pj[j] >> 16), neg = block_neg(pj[j]);
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const uint2 x = lds2(a + 64 * v);
                        m[v] &= __funnelshift_r(x.x, x.y, pj[j]) ^ neg;
                    }
                }
                alive = __any_sync(0xffffffffu, (m[0] | m[1] | m[2] | m[3]) != 0u);
            }
            uint32_t *dst = S.match + (rr * 4 + g) * bs.mstride + bs.pad + word;
            if (!alive) {  // (zeros: the planes hold the previous chunk's)
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    dst[8 * v] = 0u;
                continue;
            }
            const int cnt = __popc(m[0]) + __popc(m[1]) + __popc(m[2]) + __popc(m[3]);
            rew += (int)h0.z * cnt;
            const int total = __reduce_add_sync(0xffffffffu, cnt);
            if (total <= kBlkSparse) {
                int pos = 0;
                if (lane == 0)
                    pos = atomicAdd(queued_w, total);
                pos = __shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    for (;;) {
                        const uint32_t have = __ballot_sync(0xffffffffu, m[v] != 0u);
                        if (!have)
                            break;
                        if (m[v]) {
                            S.queue[pos + __popc(have & below)] =
                                (uint32_t)((rr << 16) | (g << 14) | (32 * (word + 8 * v) + __ffs(m[v]) - 1));
                            m[v] &= m[v] - 1u;
                        }
                        pos += __popc(have);
                    }
                    dst[8 * v] = 0u;
                }
            } else {
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    dst[8 * v] = m[v];
                if (lane == 0)
                    atomicOr(live_w, 1 << (4 * rr + k));
            }
        }
        __syncthreads();  // the chunk's match planes and queue
        const uint32_t live = (uint32_t)*live_w;  // block-uniform, as the queue's length
        const int queued = *queued_w;
        // slots are taken in turn: the next but one was last read before the
        // barrier above, and is next written after another
        slot = slot == 2 ? 0 : slot + 1;
        if (threadIdx.x == 0) {
            const int z = slot == 2 ? 0 : slot + 1;
            S.ctl[kCtlLive + z] = 0;
            S.ctl[kCtlQueued + z] = 0;
        }
        if (!live && !queued)
            continue;
        any = true;
        // ---- write
        for (int i = warp; i < queued; i += kWarps) {
            const uint32_t x = S.queue[i];
            const int r = r0 + (int)(x >> 16), rot = (int)(x >> 14) & 3, anchor = (int)(x & 0x3fffu);
            const uint4 h1 = block_ld<SM>(tb.hdr + 2 * r + 1);
            const uint32_t *outs = reinterpret_cast<const uint32_t *>(tb.outs + h1.y) + rot;
            for (uint32_t b = lane; b < (h1.w & 0xffffu); b += 32) {
                const uint32_t ob = block_ld<SM>(tb.obits + h1.z + b);
                const uint32_t d = block_ld<SM>(outs + 4 * (ob & 0xffu));
                const int cell = anchor + (int)((d >> 8) << 5) + (int)(d & 31u);
                atomicOr(S.setp + (ob >> 8) * bs.nw + (cell >> 5), 1u << (cell & 31));
            }
        }
        int skip = queued;  // units so far, so that the warps stay level
        for (uint32_t x = live; x;) {
            const int rr = (__ffs(x) - 1) >> 2;
            const uint32_t groups = (x >> (4 * rr)) & 15u;  // source groups with match planes
            x &= ~(15u << (4 * rr));
            // an anchor's output lies at most pad - 1 words on
            const uint32_t need = groups | (groups << 1) | (bs.pad > 32 ? groups << 2 : 0u);
            const uint32_t n_out = block_ld<SM>(&tb.hdr[2 * (r0 + rr)].y) & 0xffu;
            const uint32_t first = block_ld<SM>(&tb.hdr[2 * (r0 + rr) + 1].y);
            const uint32_t *mr = S.match + rr * 4 * bs.mstride + bs.pad + lane;
            const int n = (int)n_out << lg;
            for (int i = (warp - skip) & (kWarps - 1); i < n; i += kWarps) {
                if (!((need >> (i & gmask)) & 1u))
                    continue;
                const int o = (int)first + (i >> lg), word = 32 * (i & gmask) + lane;
                const uint4 d = block_ld<SM>(tb.outs + o);
                const uint32_t *b = mr + 32 * (i & gmask);
                const uint32_t *b0 = b - (d.x >> 8), *b1 = b + bs.mstride - (d.y >> 8),
                               *b2 = b + 2 * bs.mstride - (d.z >> 8), *b3 = b + 3 * bs.mstride - (d.w >> 8);
                const uint32_t D = __funnelshift_l(b0[-1], b0[0], d.x) | __funnelshift_l(b1[-1], b1[0], d.y) |
                                   __funnelshift_l(b2[-1], b2[0], d.z) | __funnelshift_l(b3[-1], b3[0], d.w);
                const uint32_t mk = block_ld<SM>(tb.masks + o);
                if (D) {
                    for (uint32_t z = mk & 0xffffu; z; z &= z - 1)
                        atomicOr(S.setp + (__ffs(z) - 1) * bs.nw + word, D);
                    for (uint32_t z = mk >> 16; z; z &= z - 1)
                        atomicOr(S.clrp + (__ffs(z) - 1) * bs.nw + word, D);
                }
            }
            skip += n;
        }
        __syncthreads();  // SET / CLEAR; the match planes may be overwritten
    }
    warp_rew += __reduce_add_sync(0xffffffffu, rew);
    return any;
}

// The step's reward from the warps' shares in S.ctl (written before a barrier).
__device__ __forceinline__ int block_reward(const BlockSmem &S)
{
    int rew = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w)
        rew += S.ctl[w];
    return rew;
}

// Actions of steps [s0, s0 + kActChunk) into the ring S.acts (one per thread).
__device__ __forceinline__ void block_actions(const uint8_t *__restrict__ actions, uint64_t seed, int env, int s0,
                                              int n_steps, const BlockSmem &S)
{
    const int s = s0 + (int)threadIdx.x;
    if (threadIdx.x < kActChunk && s < n_steps)
        S.acts[s & (kActChunk - 1)] = (uint8_t)action_at(actions, seed, env, s, S.ctl + kCtlWarn);
}

// The board after its matches: a bit changes where one asks for it (SET on clear
// cells, CLEAR on set cells; SET / CLEAR left zero).  All threads; `any`: some
// rule matched.  Returns this thread's bits: 1 a cell changed, 2 a goal tile is
// left.
__device__ __forceinline__ int block_combine(const DevConfig &cf, const BlockSmem &S, bool any)
{
    const int NW = cf.NW, NWP = cf.NWP, tid = threadIdx.x;
    int bits = 0;
    if (any) {
        const int dc = kThreads / NW, dw = kThreads % NW;  // (c, w) of i = c * NW + w, stepped without a division
        for (int i = tid, c = tid / NW, w = tid % NW; i < cf.C * NW; i += kThreads, c += dc, w += dw) {
            if (w >= NW) {
                w -= NW;
                ++c;
            }
            uint32_t d = S.planes[c * NWP + w].x;
            const uint32_t st = S.setp[i], cl = S.clrp[i];
            if (st | cl) {
                const uint32_t nd = (d & ~cl) | (~d & st);
                S.setp[i] = 0u;
                S.clrp[i] = 0u;
                if (nd != d) {
                    bits |= 1;
                    put_word(S.planes, NWP, c, w, nd);
                    d = nd;
                }
            }
            if (c == cf.ch_goal && d)
                bits |= 2;
        }
    } else if (cf.ch_goal >= 0) {
        for (int w = tid; w < NW; w += kThreads)
            if (S.planes[cf.ch_goal * NWP + w].x)
                bits |= 2;
    }
    return bits;
}

// Board cells (global) into the doubled tile planes, eight cells a thread.
template <typename CellT>
__device__ __forceinline__ void block_load_planes(const DevConfig &cf, const CellT *__restrict__ src, uint2 *dbl)
{
    if (cells8_aligned(src, cf.HW)) {  // (two loops: the code for ragged units stays out of the first)
        for (int b = threadIdx.x; 8 * b < cf.HW; b += kThreads)
            put_cells8<CellT>(cf, src, b, true, dbl);
    } else {
        for (int b = threadIdx.x; 8 * b < cf.HW; b += kThreads)
            put_cells8<CellT>(cf, src, b, false, dbl);
    }
}

}  // namespace av
