// small_step.cuh -- pieces of one step of a board of at most 16 plane words by one
// warp, shared by the memoising rollout, the single step and the expansion: a
// board's cells from its planes, term tests and the writes of a rule's matches.
// Lane = rotation x anchor word (NA words a lane: q, q + 8); tables are the packed
// ones (block_step.cuh).
#pragma once

#include "block_step.cuh"

namespace av {

constexpr int kSmallSparse = 16;  // matches of a rule written one output bit per lane at most

// Where a warp's matches go: the board's SET, then CLEAR planes ([2][C * NW]; ORed
// with atomics, so warps may share them), and the warp's own match planes
// [rotation][mstride] (`pad` zero words in front) and queue of kSmallSparse matches.
struct SmallOut {
    uint32_t *acc, *match, *queue;
    int pad, mstride;
};

// The farthest word an output moves an anchor on a board w cells wide, and one more.
__host__ __device__ inline int small_pad(int w) { return (4 * w + 4) / 32 + 1; }

// ---- a board's canonical bytes: eight cells a lane (NA of them), 8 bytes (one-
// byte cells) or 16 bytes (two-byte cells) each
template <typename CellT, int NA>
struct SmallCells {
    uint32_t v[NA][2 * sizeof(CellT)];
};

// This lane's units of the board in the doubled tile planes (a byte per channel
// and unit, transposed).
template <typename CellT, int NA>
__device__ __forceinline__ void small_cells(const DevConfig &cf, const uint2 *planes, SmallCells<CellT, NA> &o)
{
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        uint32_t x[4];
        get_cells8<CellT>(cf, planes, (int)(threadIdx.x & 31) + 32 * u, x);
#pragma unroll
        for (int i = 0; i < 2 * (int)sizeof(CellT); ++i)
            o.v[u][i] = x[i];
    }
}

// This lane's units to dst (global): whole 8 or 16 bytes (mode 0), 4-byte stores
// (mode 1), a cell a lane of 32 consecutive ones (mode 2, CELLS; all lanes) or single
// bytes (mode 3); nothing at or past the board's end.
template <typename CellT, int NA, bool CELLS>
__device__ __forceinline__ void small_store(unsigned char *dst, const SmallCells<CellT, NA> &o, int nbytes, int mode)
{
    constexpr int N = 2 * (int)sizeof(CellT);  // words per unit
    const int lane = threadIdx.x & 31;
    if (CELLS && mode == 2) {
        CellT *cells = reinterpret_cast<CellT *>(dst);
        const int n = nbytes / (int)sizeof(CellT);
#pragma unroll
        for (int u = 0; u < NA; ++u)
            for (int at = 256 * u; at < min(n, 256 * (u + 1)); at += 32) {
                // cell at + lane: of the unit of lane (at / 8) % 32 + lane / 8
                const int from = ((at >> 3) & 31) + (lane >> 3), i = lane & 7;
                uint32_t x = 0;
#pragma unroll
                for (int w = 0; w < N; ++w) {
                    const uint32_t y = __shfl_sync(0xffffffffu, o.v[u][w], from);
                    x = i * (int)sizeof(CellT) / 4 == w ? y : x;
                }
                if (at + lane < n)
                    cells[at + lane] = (CellT)(x >> (8 * (i * (int)sizeof(CellT) & 3)));
            }
        return;
    }
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        const int off = 4 * N * (lane + 32 * u);
        if (off >= nbytes)
            continue;
        if (mode == 0) {
            if constexpr (N == 4)
                *reinterpret_cast<uint4 *>(dst + off) = make_uint4(o.v[u][0], o.v[u][1], o.v[u][2], o.v[u][3]);
            else
                *reinterpret_cast<uint2 *>(dst + off) = make_uint2(o.v[u][0], o.v[u][1]);
        } else {
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const int at = off + 4 * i;
                if (mode == 1) {
                    if (at < nbytes)
                        *reinterpret_cast<uint32_t *>(dst + at) = o.v[u][i];
                } else {
                    for (int k = 0; k < 4 && at + k < nbytes; ++k)
                        dst[at + k] = (unsigned char)(o.v[u][i] >> (8 * k));
                }
            }
        }
    }
}

// Boards of an odd number of cells: a cell a lane, whose stores share their sectors, but
// for large boards of one-byte cells, where the shuffles cost more, and where the code
// for it is left out (CELLS): in the memoising rollout's loops it costs boards of whole
// units 3 %.  16,384 steps, bytes and cells: 5 x 5 23.2 / 20.1 us, 21 x 23 of two-byte
// cells 111 / 78, of one-byte cells 77 / 79.
template <typename CellT, bool CELLS>
__host__ __device__ inline int small_store_mode(const void *p, int nbytes)
{
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    constexpr int unit = 8 * (int)sizeof(CellT);
    if (nbytes % unit == 0 && a % unit == 0)
        return 0;
    if (nbytes % 4 == 0 && a % 4 == 0)
        return 1;
    return CELLS && (sizeof(CellT) == 2 || nbytes <= 128) ? 2 : 3;
}

// Four terms (this lane's rotation) at this lane's anchor words.
template <int NA>
__device__ __forceinline__ void small_terms(uint32_t pbase, const uint4 &p, uint32_t (&m)[NA])
{
    const uint32_t pj[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t a = pbase + (pj[j] >> 16), neg = block_neg(pj[j]);
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            const uint2 w = lds2(a + 64 * u);
            m[u] &= __funnelshift_r(w.x, w.y, pj[j]) ^ neg;
        }
    }
}

// The outputs of one rule at its `total` live anchors m (this lane's rotation and
// words) into the CTA's SET / CLEAR planes.  Few anchors: they are listed, and
// each lane takes one output bit of one of them (a shared atomic).  Many: the
// anchors go to the warp's match planes, and each lane takes one output entry
// (four at a time) and destination word, gathers the four rotations' anchors by
// funnel shifts and ORs them into the words of the entry's channels.
template <int NA, bool SM>
__device__ __forceinline__ void small_write(const DevConfig &cf, const BlockTable &tb, const SmallOut &S,
                                           const uint4 &h0, const uint4 &h1, uint32_t (&m)[NA], int total)
{
    const int lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    const int n_bits = (int)(h1.w & 0xffffu);
    if (n_bits == 0)
        return;
    if (total <= kSmallSparse) {
        const uint32_t below = (1u << lane) - 1u;
        int pos = 0;
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            uint32_t have;
            while ((have = __ballot_sync(0xffffffffu, m[u] != 0u)) != 0u) {
                if (m[u]) {
                    S.queue[pos + __popc(have & below)] = (uint32_t)((g << 16) | (32 * (q + 8 * u) + __ffs(m[u]) - 1));
                    m[u] &= m[u] - 1u;
                }
                pos += __popc(have);
            }
        }
        __syncwarp();
        const uint32_t *outs = reinterpret_cast<const uint32_t *>(tb.outs + h1.y);
        const uint16_t *obits = tb.obits + h1.z;
        if (n_bits <= 32) {  // 32 / n_bits anchors at a time
            const int inv = (int)(h1.w >> 16), mine = (lane * inv) >> 11, per = (32 * inv) >> 11;
            const int bit = lane - mine * n_bits;
            const uint32_t ob = block_ld<SM>(obits + bit);
            uint32_t *dst = S.acc + (ob >> 8) * cf.NW;
            const uint32_t *out = outs + 4 * (ob & 0xffu);
            for (int i = mine; mine < per && i < total; i += per) {
                const uint32_t x = S.queue[i];
                const uint32_t d = block_ld<SM>(out + (x >> 16));
                const int cell = (int)(x & 0xffffu) + (int)((d >> 8) << 5) + (int)(d & 31u);
                atomicOr(dst + (cell >> 5), 1u << (cell & 31));
            }
        } else {
            for (int i = 0; i < total; ++i) {
                const uint32_t x = S.queue[i];
                for (int b = lane; b < n_bits; b += 32) {
                    const uint32_t ob = block_ld<SM>(obits + b);
                    const uint32_t d = block_ld<SM>(outs + 4 * (ob & 0xffu) + (x >> 16));
                    const int cell = (int)(x & 0xffffu) + (int)((d >> 8) << 5) + (int)(d & 31u);
                    atomicOr(S.acc + (ob >> 8) * cf.NW + (cell >> 5), 1u << (cell & 31));
                }
            }
        }
    } else {
#pragma unroll
        for (int u = 0; u < NA; ++u)
            S.match[g * S.mstride + S.pad + q + 8 * u] = m[u];
        __syncwarp();
        const int n_out = (int)(h0.y & 0xffu);
        for (int o = g; o < n_out; o += 4) {  // quarter g takes outputs g, g + 4, ...
            const uint4 d = block_ld<SM>(tb.outs + h1.y + o);
            const uint32_t mk = block_ld<SM>(tb.masks + h1.y + o);
#pragma unroll
            for (int u = 0; u < NA; ++u) {
                const uint32_t *b = S.match + S.pad + q + 8 * u;
                const uint32_t *b0 = b - (d.x >> 8), *b1 = b + S.mstride - (d.y >> 8),
                               *b2 = b + 2 * S.mstride - (d.z >> 8), *b3 = b + 3 * S.mstride - (d.w >> 8);
                const uint32_t D = __funnelshift_l(b0[-1], b0[0], d.x) | __funnelshift_l(b1[-1], b1[0], d.y) |
                                   __funnelshift_l(b2[-1], b2[0], d.z) | __funnelshift_l(b3[-1], b3[0], d.w);
                if (D) {
                    for (uint32_t z = mk & 0xffffu; z; z &= z - 1)
                        atomicOr(S.acc + (__ffs(z) - 1) * cf.NW + q + 8 * u, D);
                    for (uint32_t z = mk >> 16; z; z &= z - 1)
                        atomicOr(S.acc + (cf.C + __ffs(z) - 1) * cf.NW + q + 8 * u, D);
                }
            }
        }
    }
    __syncwarp();  // the queue and match planes may be overwritten
}

}  // namespace av
