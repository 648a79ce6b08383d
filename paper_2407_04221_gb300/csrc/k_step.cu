// k_step.cu -- one step of every environment given its action (av_step), one
// warp per environment: the launch shape of single-step use, where no outcome
// can be repeated and a CTA's setup is most of the work.
//
// Each warp holds its environment's board as doubled bit-planes (tile
// channels 0..C-1, the force plane C, a zero plane C + 1 that the table's
// padding terms read as absent) and its own SET / CLEAR planes, and copies the
// head of its packed table (rule headers and every rule's first four terms); the
// rest of the table is read where it lies (L1 / L2).  The warp tests every rule in
// its four rotations exactly as the other kernels do (Sec. 2.1, Eq. 2: lane =
// rotation x anchor word, a rule left as soon as no anchor is live), ORs the
// outputs of live matches into SET / CLEAR (the transposed-convolution write,
// Eq. 3), pays reward x matches, combines next = (D & ~CLEAR) | (~D & SET), tests
// the goal, resets on done when asked to and writes the board, its observation, the
// reward, done flag and step counter.  Four environments share a CTA and its
// copy of the valid-anchor and column masks; after staging those no warp waits
// for another.
//
// What bounds it: latency.  On 16,384 boards of 16 x 16 with two-byte cells and 12 rules
// 0.43 of the issue slots are used: eight CTAs of 64 registers a thread keep 32 of 64
// warps on an SM, 3.4 waves, and each warp starts with a chain of dependent loads (table
// offset, header, first terms) and waits on L2 for terms past the fourth and outputs.
// Cells become planes and planes cells eight at a time by bit transposes instead of a
// ballot per channel and word and a rebuilt word per channel, and outputs are written
// per bit or gathered instead of four dependent shuffles an entry: 76.6 -> 45.6 us a
// call, 3,190 -> 1,590 warp-instructions a board.
#include "small_step.cuh"

namespace av {
namespace {

constexpr int kStepWarps = 4;  // environments per CTA
constexpr int kStepBatch = 2;  // rules whose first terms are tested together

struct StepWarpLayout {
    int vm, masks, warps;                         // CTA region
    int planes, acc, head, lead, match, queue, per_warp;  // within a warp's region
    int pad, mstride;
    int total;
};

StepWarpLayout step_warp_layout(const DevConfig &cf)
{
    StepWarpLayout L;
    int at = 0;
    auto take = [&](int bytes) {
        const int here = at;
        at = (at + bytes + 15) & ~15;
        return here;
    };
    L.vm = take(kShapes * cf.NW * 4);
    L.masks = take(3 * cf.NW * 4);
    L.warps = at;
    L.pad = small_pad(cf.W);
    L.mstride = 8 * cf.NA + L.pad;
    at = 0;
    L.planes = take((cf.C + 2) * cf.NWP * 8);
    L.head = take(cf.R * 6 * 16);
    L.lead = take(kStepBatch * 32 * cf.NA * 4);
    L.acc = take(2 * cf.C * cf.NW * 4);
    L.match = take(4 * L.mstride * 4);
    L.queue = take(kSmallSparse * 4);
    L.per_warp = at;
    L.total = L.warps + kStepWarps * L.per_warp;
    return L;
}

// A board's cells (global) into the warp's doubled tile planes (zeroed before).
template <typename CellT>
__device__ __forceinline__ void step_load_planes(const DevConfig &cf, const CellT *__restrict__ src, uint2 *dbl)
{
    const bool vec = cells8_aligned(src, cf.HW);
    for (int b = threadIdx.x & 31; 8 * b < cf.HW; b += 32)
        put_cells8<CellT>(cf, src, b, vec, dbl);
}

// Four warps a CTA, eight CTAs per SM: a CTA's slot waits for its busiest
// environment (16, 8, 4, 2 warps a CTA when measured: 54.5, 49.2, 46.3, 47.1 us on the
// shape above).  Ten, twelve and sixteen CTAs per SM (48, 40, 32 registers) on other
// tables of that shape: 37.5, 38.8, 47.0 us against 35.9.
template <typename CellT, int NA>
__global__ void __launch_bounds__(32 * kStepWarps, 8)
step_warp_kernel(const __grid_constant__ DevConfig cf, const __grid_constant__ StepWarpLayout L,
                 const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g, CellT *cur,
                 const CellT *__restrict__ init, int32_t *tsteps, const uint8_t *__restrict__ actions,
                 CellT *obs, int32_t *rew_out, uint8_t *done_out, int32_t *rew_sum, uint32_t *status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    const int NW = cf.NW, NWP = cf.NWP, C = cf.C, HW = cf.HW;
    uint32_t *vm = reinterpret_cast<uint32_t *>(smem + L.vm);
    uint32_t *masks = reinterpret_cast<uint32_t *>(smem + L.masks);
    for (int i = threadIdx.x; i < kShapes * NW; i += blockDim.x)
        vm[i] = __ldg(vm_g + i);
    for (int i = threadIdx.x; i < 3 * NW; i += blockDim.x)
        masks[i] = __ldg(masks_g + i);
    unsigned char *wr = smem + L.warps + warp * L.per_warp;
    uint2 *planes = reinterpret_cast<uint2 *>(wr + L.planes);
    uint4 *head = reinterpret_cast<uint4 *>(wr + L.head);  // [R][2] headers, then [R][4 rotations] first terms
    uint32_t *lead = reinterpret_cast<uint32_t *>(wr + L.lead);  // the anchors of the rules tested together
    SmallOut S;
    S.acc = reinterpret_cast<uint32_t *>(wr + L.acc);
    S.match = reinterpret_cast<uint32_t *>(wr + L.match);
    S.queue = reinterpret_cast<uint32_t *>(wr + L.queue);
    S.pad = L.pad;
    S.mstride = L.mstride;
    const int env = blockIdx.x * kStepWarps + warp;
    const uint32_t *pk = cf.pk + (env < cf.B ? cf.pk_off[cf.rules_per_env ? env : 0] : 0u);
    int a = 0, t = 0;
    if (env < cf.B) {
        a = (int)actions[env];  // (loaded here so that the barrier below hides it)
        t = tsteps[env] + 1;
        const uint4 *src = reinterpret_cast<const uint4 *>(pk) + 1;
        for (int i = lane; i < 6 * cf.R; i += 32)
            head[i] = __ldg(src + i);
        // (NWP is even) past a plane's words all is zero: the force plane shifts the player's
        for (int i = lane; i < (C + 2) * NWP / 2; i += 32)
            reinterpret_cast<uint4 *>(planes)[i] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        step_load_planes<CellT>(cf, cur + (size_t)env * HW, planes);
        for (int i = lane; i < 2 * C * NW; i += 32)
            S.acc[i] = 0u;
        for (int i = lane; i < 4 * L.mstride; i += 32)
            S.match[i] = 0u;
    }
    __syncthreads();  // the CTA's masks; no block barrier after this
    if (env >= cf.B)
        return;
    const bool warn = a > 4;
    if (warn)
        a = 0;
    const BlockTable tb = block_table(pk, __ldg(reinterpret_cast<const uint4 *>(pk)), cf.R);
    force_plane(cf, planes, masks, a);
    __syncwarp();

    // ---- every rule in its four rotations
    const uint4 *first = head + 2 * cf.R;
    const uint32_t pbase = (uint32_t)__cvta_generic_to_shared(planes) + q * 8;
    int rew = 0;
    for (int r0 = 0; r0 < cf.R; r0 += kStepBatch) {
        uint32_t m[kStepBatch][NA];
        uint32_t alive = 0;  // bit k: rule r0 + k passes its first terms somewhere (warp-uniform)
#pragma unroll
        for (int k = 0; k < kStepBatch; ++k) {
            const int r = r0 + k;
            if (k > 0 && r >= cf.R)
                break;
            const uint32_t *vmr = vm + ((head[2 * r].w >> (8 * g)) & 0xffu) * NW;
#pragma unroll
            for (int u = 0; u < NA; ++u)
                m[k][u] = q + 8 * u < NW ? vmr[q + 8 * u] : 0u;
            small_terms<NA>(pbase, first[4 * r + g], m[k]);
        }
#pragma unroll
        for (int k = 0; k < kStepBatch; ++k) {
            if (k > 0 && r0 + k >= cf.R)
                break;
            alive |= __any_sync(0xffffffffu, (m[k][0] | m[k][NA - 1]) != 0u) ? 1u << k : 0u;
#pragma unroll
            for (int u = 0; u < NA; ++u)
                lead[(k * 32 + lane) * NA + u] = m[k][u];
        }
        // the others' terms, eight per vote, and the writes of their matches
        for (; alive; alive &= alive - 1) {
            const int k = __ffs(alive) - 1, r = r0 + k;
            const uint4 h0 = head[2 * r], h1 = head[2 * r + 1];
            uint32_t x[NA];
#pragma unroll
            for (int u = 0; u < NA; ++u)
                x[u] = lead[(k * 32 + lane) * NA + u];
            const uint4 *tp = tb.terms + 4 * h1.x + g;
            bool live = true;
            for (uint32_t b = 1; live && b < h0.x; b += 2) {
                const uint4 p = __ldg(tp + 4 * (b - 1));
                const uint4 p2 = __ldg(tp + 4 * (b + 1 < h0.x ? b : b - 1));  // (an odd last batch is taken twice)
                small_terms<NA>(pbase, p, x);
                small_terms<NA>(pbase, p2, x);
                live = __any_sync(0xffffffffu, (x[0] | x[NA - 1]) != 0u);
            }
            if (!live)
                continue;
            int cnt = 0;
#pragma unroll
            for (int u = 0; u < NA; ++u)
                cnt += __popc(x[u]);
            const int total = __reduce_add_sync(0xffffffffu, cnt);
            rew += (int)h0.z * total;
            small_write<NA, false>(cf, tb, S, h0, h1, x, total);
        }
    }

    // ---- combine: a bit changes where a match asks for it (SET on clear
    // cells, CLEAR on set cells); then the goal test, done and reset
    __syncwarp();
    int goal = 0;
    const int sh = NW <= 8 ? 3 : 4, w = lane & ((1 << sh) - 1);
    if (w < NW)
        for (int c = lane >> sh; c < C; c += 32 >> sh) {
            const uint32_t d = planes[c * NWP + w].x, st = S.acc[c * NW + w], cl = S.acc[(C + c) * NW + w];
            const uint32_t nd = (d & ~cl) | (~d & st);
            if (nd != d)
                put_word(planes, NWP, c, w, nd);
            if (c == cf.ch_goal && nd)
                goal = 1;
        }
    const int goal_left = cf.ch_goal < 0 || __any_sync(0xffffffffu, goal);
    const int done = !goal_left || (cf.max_steps > 0 && t >= cf.max_steps);
    __syncwarp();
    if (done && cf.auto_reset)
        step_load_planes<CellT>(cf, init + (size_t)env * HW, planes);
    __syncwarp();
    {
        SmallCells<CellT, NA> v;
        small_cells<CellT, NA>(cf, planes, v);
        const int nbytes = HW * (int)sizeof(CellT);
        const size_t at = (size_t)env * nbytes;
        small_store<CellT, NA, true>(reinterpret_cast<unsigned char *>(cur) + at, v, nbytes,
                               small_store_mode<CellT, true>(cur, nbytes));
        if (obs)
            small_store<CellT, NA, true>(reinterpret_cast<unsigned char *>(obs) + at, v, nbytes,
                                   small_store_mode<CellT, true>(obs, nbytes));
    }
    if (lane == 0) {
        tsteps[env] = done && cf.auto_reset ? 0 : t;
        if (rew_out)
            rew_out[env] = rew;
        if (done_out)
            done_out[env] = (uint8_t)done;
        if (rew_sum)
            rew_sum[env] = rew;
        if (warn)
            atomicOr(status + 1, kWarnAction);
    }
}

}  // namespace

cudaError_t configure_step()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *fn) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    };
    set((const void *)step_warp_kernel<uint8_t, 1>);
    set((const void *)step_warp_kernel<uint8_t, 2>);
    set((const void *)step_warp_kernel<uint16_t, 1>);
    set((const void *)step_warp_kernel<uint16_t, 2>);
    return e;
}

bool use_step_warp(const DevConfig &cf)
{
    return cf.path == 0 && cf.NA <= 2 && step_warp_layout(cf).total <= kDynSmemLimit;
}

void launch_step_warp(const DevConfig &cf, const uint32_t *vm, const uint32_t *masks, void *cur, const void *init,
                      int32_t *t, const uint8_t *actions, void *obs, int32_t *rew, uint8_t *done, int32_t *rew_sum,
                      uint32_t *status, cudaStream_t st)
{
    const StepWarpLayout L = step_warp_layout(cf);
    const int grid = (cf.B + kStepWarps - 1) / kStepWarps;
#define AV_STEP_LAUNCH(CELL, NA)                                                                     \
    step_warp_kernel<CELL, NA><<<grid, 32 * kStepWarps, L.total, st>>>(                              \
        cf, L, vm, masks, (CELL *)cur, (const CELL *)init, t, actions, (CELL *)obs, rew, done, rew_sum, status)
    if (cf.cell_bytes == 1) {
        if (cf.NA == 1)
            AV_STEP_LAUNCH(uint8_t, 1);
        else
            AV_STEP_LAUNCH(uint8_t, 2);
    } else {
        if (cf.NA == 1)
            AV_STEP_LAUNCH(uint16_t, 1);
        else
            AV_STEP_LAUNCH(uint16_t, 2);
    }
#undef AV_STEP_LAUNCH
}

}  // namespace av
