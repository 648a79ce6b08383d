// k_variant.cu -- rollouts under the variant rule semantics sketched at the end
// of Sec. 2.1 ("Possible extensions"): a rule applied only once or a fixed
// number of times per step, the tiles to rewrite chosen by the maximum over an
// ordered or random index channel; rules inhibiting others by masking.
//
// A match is (rule r, rotation g, anchor cell p); its key is (p << 2) | g, or
// with random indices ((draw(key_seed, 13, env, t, p) >> 48) << 14) | (p << 2)
// | g, t the env's step counter before the step.  limit[r] = k > 0 keeps the
// k matches of rule r with the largest keys; a rule with any raw match this
// step suppresses the rules of its inhibit mask (decided on raw matches, so
// rule order does not matter).
//
// Boards of at most 16 plane words run the memoising rollout with a variant
// evaluation (k_memo_impl.cuh).  Here: one CTA of kThreads per environment for the
// others, boards staged as bit-planes.  Each step runs two passes over the rules,
// one warp per rule: pass 1 finds which rules have a raw match; after a barrier
// every warp derives the suppressed set; pass 2 takes the rules that matched and are
// not suppressed (a warp's last from registers, the others evaluated again), keeps
// the largest keys by warp max-reductions when the rule is limited, and writes the
// kept matches' outputs.  The combine, goal test and auto-reset are those of the
// standard step.
#include "block_step.cuh"
#include "variant_keys.cuh"

namespace av {
namespace {

// Anchors of rule r in this lane's rotation (lane >> 3) and words
// (lane & 7) + 8u where every term holds.  Returns whether any lane has one
// (warp-uniform); stops early once none is left.
template <int NA, bool SM>
__device__ __forceinline__ bool rule_matches(const DevConfig &cf, const BlockTable &tb, int r, const Smem &S,
                                             uint32_t (&m)[NA])
{
    const int lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    const uint4 h0 = block_ld<SM>(tb.hdr + 2 * r), h1 = block_ld<SM>(tb.hdr + 2 * r + 1);
    const uint32_t *vmr = S.vm + (int)((h0.w >> (8 * g)) & 0xffu) * cf.NW;
#pragma unroll
    for (int u = 0; u < NA; ++u) {
        const int a = q + 8 * u;
        m[u] = a < cf.NW ? vmr[a] : 0u;
    }
    const uint4 *tp = tb.terms + g;
    const unsigned char *pb = reinterpret_cast<const unsigned char *>(S.planes) + q * 8;
    for (uint32_t b = 0; b < h0.x; ++b) {
        const uint4 p = block_ld<SM>(tp + 4 * (b ? h1.x + b - 1 : (uint32_t)r));
        const uint32_t pj[4] = {p.x, p.y, p.z, p.w};
        uint32_t any = 0;
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            uint32_t x = m[u];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint2 w = *reinterpret_cast<const uint2 *>(pb + (pj[j] >> 16) + 64 * u);
                x &= __funnelshift_r(w.x, w.y, pj[j]) ^ block_neg(pj[j]);
            }
            m[u] = x;
            any |= x;
        }
        if (!__any_sync(0xffffffffu, any != 0u))
            return false;
    }
    return true;
}

// Outputs of the kept matches into SET / CLEAR (setp / clrp, NW words per
// channel); returns this lane's reward.
template <int NA, bool SM>
__device__ __forceinline__ int write_matches(const DevConfig &cf, const BlockTable &tb, int r, uint32_t *setp,
                                             uint32_t *clrp, const uint32_t (&m)[NA])
{
    const int lane = threadIdx.x & 31, g = lane >> 3, q = lane & 7;
    uint32_t cnt = 0;
#pragma unroll
    for (int u = 0; u < NA; ++u)
        cnt += __popc(m[u]);
    if (cnt == 0)
        return 0;
    const uint4 h0 = block_ld<SM>(tb.hdr + 2 * r), h1 = block_ld<SM>(tb.hdr + 2 * r + 1);
    for (uint32_t o = h1.y; o < h1.y + (h0.y & 0xffu); ++o) {
        const uint32_t d = block_ld<SM>(reinterpret_cast<const uint32_t *>(tb.outs + o) + g);
        const uint32_t mk = block_ld<SM>(tb.masks + o), sh = d & 31u;
#pragma unroll
        for (int u = 0; u < NA; ++u) {
            if (!m[u])
                continue;
            const int w0 = q + 8 * u + (int)(d >> 8);
            const uint32_t lo = m[u] << sh;
            const uint32_t hi = sh ? (m[u] >> (32u - sh)) : 0u;
            scatter_bits(setp, mk & 0xffffu, cf.NW, w0, lo, hi);
            scatter_bits(clrp, mk >> 16, cf.NW, w0, lo, hi);
        }
    }
    return (int)h0.z * (int)cnt;
}

// CTAs per SM to compile for: the registers of a CTA decide how many share an SM.
// 2156 boards of 56 x 15 take 0.397 ms with four CTAs per SM, 0.348 with five (no
// spills; 0.369 with the unpacked tables before); 445 boards, one wave either way, 1.36
// against 1.47 (1.47).  Larger boards are limited by their planes in shared memory: more
// registers are free there.
constexpr int variant_ctas(int na) { return na <= 4 ? 5 : na == 8 ? 4 : 2; }

template <typename CellT, int NA, bool SM>
__global__ void __launch_bounds__(kThreads, variant_ctas(NA))
    rollout_variant_kernel(DevConfig cf, const __grid_constant__ VariantParams vp,
                           const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g, CellT *cur,
                           const CellT *__restrict__ init, int32_t *tsteps, int n_steps, uint64_t seed,
                           const uint8_t *__restrict__ actions, CellT *obs_traj, int32_t *rew_traj,
                           uint8_t *done_traj, int32_t *rew_sum, uint32_t *status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_raw[2];  // rules with a raw match this step
    __shared__ int s_t;            // the env's step counter
    const Smem S = carve(smem, cf);
    const int env = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int HW = cf.HW, NW = cf.NW, NWP = cf.NWP, C = cf.C;
    const int table = cf.rules_per_env ? env : 0;
    const uint32_t *pk = cf.pk + cf.pk_off[table];
    const BlockTable tb = block_table(SM ? S.rules : pk, __ldg(reinterpret_cast<const uint4 *>(pk)), cf.R);

    stage_common(cf, S, vm_g, masks_g);
    if (SM)
        stage_rules(pk, cf.pk_off[table + 1] - cf.pk_off[table], S.rules);
    if (tid == 0) {
        s_raw[0] = s_raw[1] = 0u;
        s_t = tsteps[env];
    }
    __syncthreads();
    cells_to_planes<CellT>(cf, cur + (size_t)env * HW, S.planes, nullptr);
    cells_to_planes<CellT>(cf, init + (size_t)env * HW, nullptr, S.basep);
    fill_actions(actions, seed, env, 0, n_steps, S);
    __syncthreads();
    if (warp == 0)
        write_force(cf, S, S.acts[0]);
    __syncthreads();

    const uint64_t key_prefix = variant_prefix(vp, env);
    int sum = 0;
    for (int s = 0; s < n_steps; ++s) {
        if (((s + 1) & (kActChunk - 1)) == 0)
            fill_actions(actions, seed, env, s + 1, n_steps, S);
        const int t = s_t;
        // pass 1: which rules have a raw match
        uint32_t last[NA];  // this warp's last matching rule's matches, for pass 2
        int last_r = -1;
        for (int r = warp; r < cf.R; r += kWarps) {
            uint32_t m[NA];
            if (!rule_matches<NA, SM>(cf, tb, r, S, m))
                continue;
            if (lane == 0)
                atomicOr(&s_raw[r >> 5], 1u << (r & 31));
            last_r = r;
#pragma unroll
            for (int u = 0; u < NA; ++u)
                last[u] = m[u];
        }
        __syncthreads();
        const uint64_t raw = (uint64_t)s_raw[0] | ((uint64_t)s_raw[1] << 32);
        uint64_t sup = 0;
        for (uint64_t x = raw; x; x &= x - 1u)
            sup |= vp.inhibit[__ffsll((long long)x) - 1];
        // pass 2: the rules that apply, their kept matches written
        int rew = 0;
        for (int r = warp; r < cf.R; r += kWarps) {
            if (!((raw >> r) & 1u) || ((sup >> r) & 1u))
                continue;
            uint32_t m[NA];
            if (r == last_r) {
#pragma unroll
                for (int u = 0; u < NA; ++u)
                    m[u] = last[u];
            } else {
                rule_matches<NA, SM>(cf, tb, r, S, m);
            }
            if (vp.limit[r] > 0)
                keep_largest<NA>(m, vp.limit[r], vp, key_prefix, t);
            uint32_t kept = 0;
#pragma unroll
            for (int u = 0; u < NA; ++u)
                kept |= m[u];
            if (kept)
                S.flags[0] = 1;  // this lane writes
            rew += write_matches<NA, SM>(cf, tb, r, S.setp, S.clrp, m);
        }
        rew = __reduce_add_sync(0xffffffffu, rew);
        if (lane == 0)
            S.red[warp] = rew;
        __syncthreads();
        if (warp == 0) {
            // combine: a bit changes where any kept match asks for it
            if (S.flags[0]) {
                // one index over every channel's words; (c, w) stepped without a division
                for (int i = lane, c = lane / NW, w = lane - (lane / NW) * NW; i < C * NW; i += 32) {
                    const uint32_t d = S.planes[c * NWP + w].x, st = S.setp[i], cl = S.clrp[i];
                    S.setp[i] = 0u;
                    S.clrp[i] = 0u;
                    put_word(S.planes, NWP, c, w, (d & ~cl) | (~d & st));
                    for (w += 32; w >= NW; w -= NW)
                        ++c;
                }
                __syncwarp();
                if (lane == 0)
                    S.flags[0] = 0;
            }
            int goal = cf.ch_goal < 0;
            if (cf.ch_goal >= 0)
                for (int w = lane; w < NW; w += 32)
                    goal |= S.planes[cf.ch_goal * NWP + w].x != 0u;
            goal = __any_sync(0xffffffffu, goal);
            int tn = t + 1;
            const int done = !goal || (cf.max_steps > 0 && tn >= cf.max_steps);
            if (done && cf.auto_reset) {
                for (int i = lane, c = lane / NW, w = lane - (lane / NW) * NW; i < C * NW; i += 32) {
                    put_word(S.planes, NWP, c, w, S.basep[i]);
                    for (w += 32; w >= NW; w -= NW)
                        ++c;
                }
                tn = 0;
            }
            int total = lane < kWarps ? S.red[lane] : 0;
            total = __reduce_add_sync(0xffffffffu, total);
            sum += total;
            if (lane == 0) {
                if (rew_traj)
                    rew_traj[(size_t)s * cf.B + env] = total;
                if (done_traj)
                    done_traj[(size_t)s * cf.B + env] = (uint8_t)done;
                s_t = tn;
                s_raw[0] = s_raw[1] = 0u;
            }
            __syncwarp();
            if (s + 1 < n_steps)
                write_force(cf, S, S.acts[(s + 1) & (kActChunk - 1)]);
        }
        __syncthreads();
        if (obs_traj)
            store_cells<CellT>(cf, S.planes, obs_traj + ((size_t)s * cf.B + env) * HW, tid, kThreads);
    }
    store_cells<CellT>(cf, S.planes, cur + (size_t)env * HW, tid, kThreads);
    if (tid == 0) {
        tsteps[env] = s_t;
        if (rew_sum)
            rew_sum[env] = sum;
        if (S.flags[1])
            atomicOr(status + 1, kWarnAction);
    }
}

#define AV_FOR_NA(MACRO, CELL) MACRO(CELL, 1) MACRO(CELL, 2) MACRO(CELL, 4) MACRO(CELL, 8) MACRO(CELL, 16)

template <typename CellT, int NA>
void variant_t(const DevConfig &cf, const VariantParams &vp, const uint32_t *vm, const uint32_t *masks, void *cur, const void *init, int32_t *t, int n_steps,
               uint64_t seed, const uint8_t *actions, void *obs_traj, int32_t *rew_traj, uint8_t *done_traj,
               int32_t *rew_sum, uint32_t *status, cudaStream_t st)
{
    const size_t sm = step_smem(cf).total;
    if (cf.pk_staged > 0)
        rollout_variant_kernel<CellT, NA, true><<<cf.B, kThreads, sm, st>>>(
            cf, vp, vm, masks, (CellT *)cur, (const CellT *)init, t, n_steps, seed, actions,
            (CellT *)obs_traj, rew_traj, done_traj, rew_sum, status);
    else
        rollout_variant_kernel<CellT, NA, false><<<cf.B, kThreads, sm, st>>>(
            cf, vp, vm, masks, (CellT *)cur, (const CellT *)init, t, n_steps, seed, actions,
            (CellT *)obs_traj, rew_traj, done_traj, rew_sum, status);
}

}  // namespace

cudaError_t configure_variant()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *fn) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    };
#define AV_SET(CELL, NA)                                        \
    set((const void *)rollout_variant_kernel<CELL, NA, true>);  \
    set((const void *)rollout_variant_kernel<CELL, NA, false>);
    AV_FOR_NA(AV_SET, uint8_t)
    AV_FOR_NA(AV_SET, uint16_t)
#undef AV_SET
    return e;
}

// Boards of at most 16 plane words take the memoising rollout's variant form
// (use_variant_memo), others one CTA of kThreads per environment.
void launch_rollout_variant(const DevConfig &cf, const VariantParams &vp, const uint32_t *vm, const uint32_t *masks, void *cur,
                            const void *init, int32_t *t, int n_steps, uint64_t seed, const uint8_t *actions,
                            void *obs_traj, int32_t *rew_traj, uint8_t *done_traj, int32_t *rew_sum,
                            uint32_t *status, cudaStream_t st)
{
#define AV_CASE(CELL, NA)                                                                                    \
    case NA:                                                                                                \
        variant_t<CELL, NA>(cf, vp, vm, masks, cur, init, t, n_steps, seed, actions, obs_traj, \
                            rew_traj, done_traj, rew_sum, status, st);                                      \
        break;
    if (use_variant_memo(cf)) {
        if (vp.many)
            (cf.cell_bytes == 1 ? launch_rollout_vmany_u8 : launch_rollout_vmany_u16)(
                cf, VariantManyParams{vp}, vm, masks, cur, init, t, n_steps, seed, actions, obs_traj, rew_traj,
                done_traj, rew_sum, status, st);
        else
            (cf.cell_bytes == 1 ? launch_rollout_vmemo_u8 : launch_rollout_vmemo_u16)(
                cf, vp, vm, masks, cur, init, t, n_steps, seed, actions, obs_traj, rew_traj, done_traj, rew_sum, status,
                st);
        return;
    }
    if (cf.cell_bytes == 1) {
        switch (cf.NA) { AV_FOR_NA(AV_CASE, uint8_t) }
    } else {
        switch (cf.NA) { AV_FOR_NA(AV_CASE, uint16_t) }
    }
#undef AV_CASE
}

}  // namespace av
