// k_band.cu -- rollouts of boards larger than one CTA's shared memory (up to
// 256 x 256 cells): the same step (Sec. 2.1; match, write, combine) with the
// board streamed through shared memory in bands of rows.
//
// One cluster of CTAs of kThreads per environment (eight CTAs for few
// environments, one for many).  The board's bit-planes (C tile channels, plain
// 32-bit words) and its SET / CLEAR accumulators live in global memory, where they
// stay in L2 (read past L1, since the cluster's other CTAs write them).  A band is
// `band_rows` rows of anchors plus the rows below it that windows anchored in it
// reach (four for 5 x 5 patterns), `band_nw` plane words in all; CTA r of the
// cluster takes bands r, r + N, ...  It copies the band's planes into shared memory
// in the doubled (word j, word j + 1) layout, the force plane made on the way from
// the player's, masks the whole board's valid anchors to the band's own rows, runs
// the block rollout's matcher (block_match, writes into shared SET / CLEAR), and ORs
// those into the global SET / CLEAR with atomics -- bands overlap in their last
// rows, whose writes merge there.  After a cluster barrier each CTA combines its
// share of the board's words (a bit changes where any match asks for it) and tells
// the others its reward, whether a cell changed and whether a goal tile is left
// (stores into their shared memory); a second cluster barrier ends the step.  Every
// CTA keeps the same counters and remembered steps, so all take the same branches.
//
// What bounds it: the environment whose rules write most, when every environment is
// one CTA (256 environments of 256 x 256 x 16, 24 rules that fire: the busiest SM
// worked 1.8 times the average, at 24 % of its issue rate), then instruction issue.
// 20 steps: 17.1 -> 8.7 ms with eight CTAs per environment.
#include "block_step.cuh"

namespace av {
namespace {

constexpr int kBandCtas = 8;  // CTAs per environment at most

// Force plane word w for `action` from the player plane pl (plain words,
// nw of them): the player at p puts force at p + d (d = -W up, +1 right, +W
// down, -1 left), dropped where it would leave the board.
__device__ __forceinline__ uint32_t force_word(const DevConfig &cf, const uint32_t *pl,
                                               const uint32_t *__restrict__ masks, int nw, int w, int action)
{
    if (cf.ch_player < 0 || action < 1 || action > 4)
        return 0u;
    const int n = (action == 1 || action == 3) ? cf.W : 1;
    const int q = n >> 5, r = n & 31;
    uint32_t f = 0;
    if (action == 1 || action == 4) {  // toward lower p: bits [32w + n, 32w + n + 32)
        const uint32_t lo = w + q < nw ? __ldcg(pl + w + q) : 0u;
        const uint32_t hi = w + q + 1 < nw ? __ldcg(pl + w + q + 1) : 0u;
        f = __funnelshift_r(lo, hi, r);
    } else {  // toward higher p: bits [32w - n, 32w - n + 32)
        const int j = w - q;
        if (j >= 1)
            f = __funnelshift_l(__ldcg(pl + j - 1), __ldcg(pl + j), r);
        else if (j == 0)
            f = __ldcg(pl) << r;
    }
    if (action == 2)
        f &= ~masks[w];  // not from the last column onto the first
    else if (action == 4)
        f &= ~masks[nw + w];
    return f & masks[2 * nw + w];
}

// Barrier of every thread of the cluster, ordering its memory accesses.
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// (x, y) into `slot` (this CTA's shared memory) of CTA `rank` of the cluster.
__device__ __forceinline__ void cluster_put(int2 *slot, int rank, int x, int y)
{
    uint32_t there;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(there)
                 : "r"((uint32_t)__cvta_generic_to_shared(slot)), "r"(rank));
    asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(there), "r"(x), "r"(y) : "memory");
}

// Plane words w of a board (32 cells each): the C channels' words from its cells.
template <typename CellT>
__device__ __forceinline__ void band_load_word(const DevConfig &cf, const CellT *__restrict__ src, bool vec, int w,
                                               uint32_t *planes)
{
    uint32_t x[4][4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        x[b][0] = x[b][1] = x[b][2] = x[b][3] = 0u;
        if (32 * w + 8 * b < cf.HW)
            load_cells8<CellT>(src, cf.HW, 4 * w + b, vec, x[b][0], x[b][1], x[b][2], x[b][3]);
    }
#pragma unroll
    for (int c = 0; c < 8 * (int)sizeof(CellT); ++c) {
        if (c >= cf.C)
            break;
        uint32_t v = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            v |= ((x[b][c >> 2] >> (8 * (c & 3))) & 0xffu) << (8 * b);
        planes[c * cf.NW + w] = v;
    }
}

// Eight cells (unit b) of the board in the planes, stored to n consecutive steps'
// boards dst, dst + stride, ... (stride in cells).
template <typename CellT>
__device__ __forceinline__ void band_store_unit(const DevConfig &cf, const uint32_t *planes, int b, CellT *dst,
                                                size_t stride, int n)
{
    uint32_t x[4] = {0u, 0u, 0u, 0u};
    const unsigned char *p = reinterpret_cast<const unsigned char *>(planes) + b;
#pragma unroll
    for (int c = 0; c < 8 * (int)sizeof(CellT); ++c) {
        if (c >= cf.C)
            break;
        x[c >> 2] |= (uint32_t)__ldcg(p + (size_t)c * cf.NW * 4) << (8 * (c & 3));
    }
    uint32_t o[4];
    cells_of_bytes8<CellT>(x, o);
    const bool vec = cells8_aligned(dst, cf.HW) && (stride & 7) == 0;
    for (int k = 0; k < n; ++k, dst += stride) {
        if (vec) {
            if constexpr (sizeof(CellT) == 1)
                *reinterpret_cast<uint2 *>(dst + 8 * b) = make_uint2(o[0], o[1]);
            else
                *reinterpret_cast<uint4 *>(dst + 8 * b) = make_uint4(o[0], o[1], o[2], o[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (8 * b + i < cf.HW)
                    dst[8 * b + i] = sizeof(CellT) == 1 ? (CellT)(o[i >> 2] >> (8 * (i & 3)))
                                                        : (CellT)(o[i >> 1] >> (16 * (i & 1)));
        }
    }
}

template <typename CellT, bool SM>
__global__ void __launch_bounds__(kThreads, kBlkCtas)
    rollout_band_kernel(const __grid_constant__ DevConfig cf, const __grid_constant__ BlockShape bs, int ctas,
                        int band_rows, const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g,
                        CellT *cur, const CellT *__restrict__ init, int32_t *tsteps, int n_steps, uint64_t seed,
                        const uint8_t *__restrict__ actions, CellT *obs_traj, int32_t *rew_traj,
                        uint8_t *done_traj, int32_t *rew_sum, uint32_t *status, uint32_t *planes_g,
                        uint32_t *set_g, uint32_t *clr_g, uint32_t *base_g)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int2 s_part[2][kBandCtas];  // each CTA's (reward, bits) of a step, two steps in turn
    __shared__ int s_bits;
    const BlockSmem S = block_carve(smem, block_layout(cf, bs, bs.nw, 0), cf, bs);
    int *ctl = S.ctl;
    const int env = blockIdx.x / ctas, rank = blockIdx.x - env * ctas;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int me = rank * kThreads + tid, all = ctas * kThreads;  // this thread among the cluster's
    const int H = cf.H, W = cf.W, HW = cf.HW, NW = cf.NW, NWP = cf.NWP, C = cf.C, NWB = bs.nw;
    uint32_t *P = planes_g + (size_t)env * (C + 1) * NW;
    uint32_t *SETg = set_g + (size_t)env * C * NW;
    uint32_t *CLRg = clr_g + (size_t)env * C * NW;
    uint32_t *BASE = base_g + (size_t)env * C * NW;
    const uint32_t *PL = P + (cf.ch_player >= 0 ? cf.ch_player : 0) * NW;
    auto barrier = [&] {  // of the environment's CTAs
        if (ctas > 1)
            cluster_barrier();
        else
            __syncthreads();
    };

    // ---- stage: shared planes zeroed once (entries past a band's words stay
    // zero), rule table, actions; the board and its initial map as planes
    const BlockTable tb = block_stage<SM>(cf, bs, S, cf.rules_per_env ? env : 0);
    if (tid == 0)
        s_bits = 0;
    __syncthreads();
    block_actions(actions, seed, env, 0, n_steps, S);
    {
        const CellT *src = cur + (size_t)env * HW, *isrc = init + (size_t)env * HW;
        const bool vec = cells8_aligned(src, HW), ivec = cells8_aligned(isrc, HW);
        for (int w = me; w < NW; w += all) {
            band_load_word<CellT>(cf, src, vec, w, P);
            band_load_word<CellT>(cf, isrc, ivec, w, BASE);
        }
        for (int i = me; i < C * NW; i += all) {
            SETg[i] = 0u;
            CLRg[i] = 0u;
        }
    }
    int t = tsteps[env];
    barrier();  // the board; the ring

    int sum = 0, slot = 0, parity = 0;
    bool goal_left = true;  // of the board in hand, once a step has been evaluated on it
    int act = S.acts[0];    // the coming step's action (its ring slot may be refilled)
    uint32_t known = 0;     // bit a: the step with action a is remembered to leave the board as it is
    int known_rew = 0;      // lane a: its reward
    const int n_bands = (H + band_rows - 1) / band_rows;
    const int n_units = (HW + 7) / 8;

    // While the board stays as it is, the step with action a always has the
    // same outcome: an action whose step changed nothing is remembered and its
    // later steps skip the bands until the board changes or resets.
    for (int s = 0; s < n_steps; ++s) {
        const bool refill = ((s + 1) & (kActChunk - 1)) == 0;
        if (refill) {
            __syncthreads();  // the ring's last readers
            block_actions(actions, seed, env, s + 1, n_steps, S);
            __syncthreads();  // the ring's next chunk
        }
        if ((known >> act) & 1u) {
            // A run of repeated steps: from this step on, the steps whose actions
            // are remembered and that end no episode with an auto-reset take their
            // remembered rewards, up to 32 at a time (lane l takes step s + l; every
            // warp walks the same run), never past the ring's chunk.
            const int lim = min(min(32, n_steps - s), ((s + 1) | (kActChunk - 1)) - s);
            const int a_l = lane == 0 ? act : lane < lim ? (int)S.acts[(s + lane) & (kActChunk - 1)] : 0;
            const bool done_l = !goal_left || (cf.max_steps > 0 && t + lane + 1 >= cf.max_steps);
            const bool known_l = (known >> a_l) & 1u;
            const uint32_t stop = __ballot_sync(0xffffffffu, lane < lim && (!known_l || (done_l && cf.auto_reset)));
            const int e = stop ? __ffs(stop) - 1 : lim;  // steps s .. s + e - 1 repeat the board
            const int r_all = __shfl_sync(0xffffffffu, known_rew, a_l), r_l = lane < e ? r_all : 0;
            if (rank == 0 && warp == 0 && lane < e) {
                if (rew_traj)
                    rew_traj[(size_t)(s + lane) * cf.B + env] = r_l;
                if (done_traj)
                    done_traj[(size_t)(s + lane) * cf.B + env] = (uint8_t)done_l;
            }
            if (e > 0) {
                sum += __reduce_add_sync(0xffffffffu, r_l);
                t += e;
                if (obs_traj)
                    for (int b = me; b < n_units; b += all)
                        band_store_unit<CellT>(cf, P, b, obs_traj + ((size_t)s * cf.B + env) * HW, (size_t)cf.B * HW, e);
                if (s + e < n_steps)
                    act = S.acts[(s + e) & (kActChunk - 1)];
                s += e - 1;
                continue;
            }
        }
        int rew;
        const bool was_known = (known >> act) & 1u;
        if (was_known) {
            rew = __shfl_sync(0xffffffffu, known_rew, act);
        } else {
            int warp_rew = 0;
            for (int band = rank; band < n_bands; band += ctas) {
                const int A0 = band * band_rows * W, A1 = min(H, (band + 1) * band_rows) * W;  // anchor cells
                const int w0 = A0 >> 5;
                for (int i = tid; i < (C + 1) * NWB; i += kThreads) {
                    const int c = i / NWB, a = i - c * NWB;
                    const uint32_t v = w0 + a >= NW ? 0u
                                       : c < C      ? __ldcg(P + c * NW + w0 + a)
                                                    : force_word(cf, PL, masks_g, NW, w0 + a, act);
                    put_word(S.planes, NWP, c, a, v);
                }
                for (int a = tid; a < NWB; a += kThreads) {  // the band's own anchors
                    const int g = w0 + a;
                    const int lo = max(A0 - 32 * g, 0), hi = min(A1 - 32 * g, 32);  // those in this word
                    S.keep[a] = lo >= hi ? 0u : ((hi == 32 ? 0xffffffffu : ((1u << hi) - 1u)) & ~((1u << lo) - 1u));
                }
                __syncthreads();
                // (ends with a barrier after the last read of the band's planes)
                if (block_match<SM, true>(cf, bs, tb, S, vm_g, NW, w0, slot, warp_rew)) {
                    for (int i = tid; i < C * NWB; i += kThreads) {
                        const int c = i / NWB, a = i - c * NWB;
                        const uint32_t st = S.setp[i], cl = S.clrp[i];
                        if (st) {
                            atomicOr(&SETg[c * NW + w0 + a], st);
                            S.setp[i] = 0u;
                        }
                        if (cl) {
                            atomicOr(&CLRg[c * NW + w0 + a], cl);
                            S.clrp[i] = 0u;
                        }
                    }
                }
            }
            barrier();  // every band's SET / CLEAR bits
            // ---- this CTA's share of the board: combine, goal test
            int bits = 0;  // 1: a cell changes, 2: a goal tile is left
            for (int i = me; i < C * NW; i += all) {
                uint32_t d = __ldcg(P + i);
                const uint32_t st = __ldcg(SETg + i), cl = __ldcg(CLRg + i);
                if (st | cl) {
                    const uint32_t nd = (d & ~cl) | (~d & st);
                    SETg[i] = 0u;
                    CLRg[i] = 0u;
                    if (nd != d) {
                        bits |= 1;
                        P[i] = nd;
                        d = nd;
                    }
                }
                if (cf.ch_goal >= 0 && d && (uint32_t)(i - cf.ch_goal * NW) < (uint32_t)NW)
                    bits |= 2;
            }
            bits = __reduce_or_sync(0xffffffffu, (unsigned)bits);
            if (lane == 0) {
                ctl[warp] = warp_rew;
                if (bits)
                    atomicOr(&s_bits, bits);
            }
            __syncthreads();  // this CTA's share
            if (warp == 0) {
                const int mine = block_reward(S), b = s_bits;
                if (lane < ctas) {
                    if (ctas > 1)
                        cluster_put(&s_part[parity][rank], lane, mine, b);
                    else
                        s_part[parity][0] = make_int2(mine, b);
                }
            }
            barrier();  // the board after its step, every CTA's part
            rew = 0;
            bits = 0;
            for (int k = 0; k < ctas; ++k) {
                const int2 x = s_part[parity][k];
                rew += x.x;
                bits |= x.y;
            }
            parity ^= 1;
            if (tid == 0)
                s_bits = 0;  // (set again after a barrier)
            goal_left = cf.ch_goal < 0 || (bits & 2);
            if (bits & 1) {
                known = 0;
            } else {  // remember the step: it left the board as it was
                known |= 1u << act;
                if (lane == act)
                    known_rew = rew;
            }
        }
        t += 1;
        const bool done = !goal_left || (cf.max_steps > 0 && t >= cf.max_steps);
        if (done && cf.auto_reset) {
            barrier();  // the board's last readers
            for (int i = me; i < C * NW; i += all)
                P[i] = __ldcg(BASE + i);
            t = 0;
            known = 0;  // the board may have changed
            barrier();
        }
        sum += rew;
        if (rank == 0 && tid == 0) {
            if (rew_traj)
                rew_traj[(size_t)s * cf.B + env] = rew;
            if (done_traj)
                done_traj[(size_t)s * cf.B + env] = (uint8_t)done;
        }
        if (s + 1 < n_steps)
            act = S.acts[(s + 1) & (kActChunk - 1)];
        if (obs_traj)
            for (int b = me; b < n_units; b += all)
                band_store_unit<CellT>(cf, P, b, obs_traj + ((size_t)s * cf.B + env) * HW, 0, 1);
    }
    for (int b = me; b < n_units; b += all)
        band_store_unit<CellT>(cf, P, b, cur + (size_t)env * HW, 0, 1);
    if (rank == 0 && tid == 0) {
        tsteps[env] = t;
        if (rew_sum)
            rew_sum[env] = sum;
        if (ctl[kCtlWarn])
            atomicOr(status + 1, kWarnAction);
    }
    barrier();  // no CTA ends while another may still store into its shared memory
}

}  // namespace

cudaError_t configure_band()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *fn) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    };
    set((const void *)rollout_band_kernel<uint8_t, true>);
    set((const void *)rollout_band_kernel<uint8_t, false>);
    set((const void *)rollout_band_kernel<uint16_t, true>);
    set((const void *)rollout_band_kernel<uint16_t, false>);
    return e;
}

void band_geometry(int H, int W, int *band_rows, int *band_nw, int *na, int *nwp)
{
    // the most rows whose anchors and the four rows below them fit 128 words
    // (with a word of slack on each side), so that the block matcher's lanes
    // (8 x NA words, NA <= 16) cover the band
    int rows = H;
    auto words = [&](int r) { return (31 + r * W + 4 * W + 4 + 31) / 32 + 1; };
    while (rows > 1 && words(rows) > 128)
        --rows;
    *band_rows = rows;
    *band_nw = words(rows);
    int a = 1;
    while (8 * a < *band_nw)
        a *= 2;
    *na = a;
    *nwp = 8 * a + (4 * W + 4) / 32 + 2;  // a lane's words plus the farthest term offset
}

void launch_rollout_band(const DevConfig &cf, int band_rows, int band_nw, const uint32_t *vm, const uint32_t *masks, void *cur,
                         const void *init, int32_t *t, int n_steps, uint64_t seed, const uint8_t *actions,
                         void *obs_traj, int32_t *rew_traj, uint8_t *done_traj, int32_t *rew_sum, uint32_t *status,
                         uint32_t *planes, uint32_t *set, uint32_t *clr, uint32_t *base, cudaStream_t st)
{
    const BlockShape bs = block_shape_fit(cf, band_nw, band_nw, 0);
    const size_t sm = block_layout(cf, bs, bs.nw, 0).total;
    // CTAs per environment: enough that the GPU's SMs (about 300 to 450 CTAs at a
    // time) get several each, so that one busy environment does not decide the
    // launch; no more than bands.
    const int n_bands = (cf.H + band_rows - 1) / band_rows;
    int ctas = kBandCtas;
    while (ctas > 1 && (ctas > n_bands || (long long)cf.B * ctas > 152LL * 32))
        ctas >>= 1;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3((unsigned)(cf.B * ctas));
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = sm;
    lc.stream = st;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)ctas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    lc.attrs = &attr;
    lc.numAttrs = ctas > 1 ? 1 : 0;
#define AV_LAUNCH(CELL, SM)                                                                                       \
    (void)cudaLaunchKernelEx(&lc, rollout_band_kernel<CELL, SM>, cf, bs, ctas, band_rows, vm, masks, (CELL *)cur,   \
                             (const CELL *)init, t, n_steps, seed, actions, (CELL *)obs_traj, rew_traj, done_traj, \
                             rew_sum, status, planes, set, clr, base)
    if (cf.cell_bytes == 1) {
        if (cf.pk_staged)
            AV_LAUNCH(uint8_t, true);
        else
            AV_LAUNCH(uint8_t, false);
    } else {
        if (cf.pk_staged)
            AV_LAUNCH(uint16_t, true);
        else
            AV_LAUNCH(uint16_t, false);
    }
#undef AV_LAUNCH
}

}  // namespace av
