// k_block.cu -- rollout kernel with one CTA of kThreads per environment, boards
// of up to 128 plane words (used for those of more than 16).
#include "block_step.cuh"

namespace av {
namespace {

// Fused rollout (n_steps >= 1).  With `actions` non-null the action of step
// s is actions[env] (used by av_step, n_steps = 1); else it is drawn.
// SM: the packed rule table is staged in shared memory.  RUNS: runs of
// repeated steps are walked 32 at a time (left out of one-step launches).
//
// A step that has to be evaluated is block_match (two barriers per chunk of
// rules that matched, one per chunk that did not), the combine by all threads
// and the next force plane: a barrier each.  64 x 64 boards, 24 sparse rules
// that fire on most steps, 4096 environments x 100 steps: 64.3 -> 20.8 ms
// (one warp per rule with scattered shared atomics, combine by one warp -> this).
// CTAS: CTAs per SM, see block_ctas.
template <typename CellT, bool SM, bool RUNS, int CTAS>
__global__ void __launch_bounds__(kThreads, CTAS)
rollout_kernel(DevConfig cf, BlockShape bs, const uint32_t *__restrict__ vm_g, const uint32_t *__restrict__ masks_g, CellT *cur,
               const CellT *__restrict__ init, int32_t *tsteps, int n_steps, uint64_t seed,
               const uint8_t *__restrict__ actions, CellT *obs_traj, int32_t *rew_traj,
               uint8_t *done_traj, int32_t *rew_sum, uint32_t *status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const BlockSmem S = block_carve(smem, block_layout(cf, bs, 0, 0), cf, bs);
    int *ctl = S.ctl;
    const int env = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int HW = cf.HW;

    const BlockTable tb = block_stage<SM>(cf, bs, S, cf.rules_per_env ? env : 0);
    __syncthreads();
    block_load_planes<CellT>(cf, cur + (size_t)env * HW, S.planes);
    block_actions(actions, seed, env, 0, n_steps, S);
    int t = tsteps[env];  // the same in every thread
    __syncthreads();
    if (warp == 0) {
        force_plane(cf, S.planes, masks_g, S.acts[0]);
        if (lane == 0)
            ctl[kCtlAct] = S.acts[0];  // the action of the coming step (the ring slot may be refilled)
    }
    __syncthreads();

    int sum = 0;               // of warp 0
    int slot = 0, parity = 0;  // control slots taken in turn
    bool goal_left = true;     // of the board in hand, once a step has been evaluated on it
    bool at_init = false;      // the board in hand is known to be the initial map
    // While the board stays as it is, the step with action a always has the
    // same outcome: an action whose step matched nothing that changes the board
    // is remembered (bit a of ctl[kCtlKnown], its reward in ctl[kCtlRew + a]) and
    // its later steps skip the match; any change of the board forgets them all.
    for (int s = 0; s < n_steps; ++s) {
        const bool refill = ((s + 1) & (kActChunk - 1)) == 0;
        if (refill)
            block_actions(actions, seed, env, s + 1, n_steps, S);
        const int a = ctl[kCtlAct];
        const bool known = (ctl[kCtlKnown] >> a) & 1;  // block-uniform
        // A run of repeated steps: from this step on, the steps whose actions
        // are remembered and that end no episode with an auto-reset take their
        // remembered rewards without a match or a board update, up to 32 at a
        // time (lane l of warp 0 takes step s + l) and never up to the last
        // step of the action ring's chunk (that step refills the ring).  Two
        // block barriers per run instead of two per step: the first publishes
        // the run's length once every warp has read this step's action; after
        // it warp 0 writes the next step's action and force plane, which the
        // second makes visible.
        if (RUNS && known) {
            if (refill)
                __syncthreads();  // the ring's next chunk
            int a_next = 0;
            if (warp == 0) {
                const int lim = min(min(32, n_steps - s), ((s + 1) | (kActChunk - 1)) - s);
                const int a_l = lane == 0 ? a : lane < lim ? (int)S.acts[(s + lane) & (kActChunk - 1)] : 0;
                const bool done_l = !goal_left || (cf.max_steps > 0 && t + lane + 1 >= cf.max_steps);
                const bool known_l = (ctl[kCtlKnown] >> a_l) & 1;
                const uint32_t stop =
                    __ballot_sync(0xffffffffu, lane < lim && (!known_l || (done_l && cf.auto_reset)));
                const int e = stop ? __ffs(stop) - 1 : lim;  // steps s .. s + e - 1 repeat the board
                const int r_l = lane < e ? ctl[kCtlRew + a_l] : 0;
                if (lane < e) {
                    if (rew_traj)
                        rew_traj[(size_t)(s + lane) * cf.B + env] = r_l;
                    if (done_traj)
                        done_traj[(size_t)(s + lane) * cf.B + env] = (uint8_t)done_l;
                }
                sum += __reduce_add_sync(0xffffffffu, r_l);
                a_next = __shfl_sync(0xffffffffu, a_l, e & 31);  // (read from the ring when e = lim)
                if (e == lim && s + e < n_steps)
                    a_next = S.acts[(s + e) & (kActChunk - 1)];
                if (lane == 0)
                    ctl[kCtlRun] = e;
            }
            __syncthreads();
            const int e = ctl[kCtlRun];
            if (e > 0) {
                if (warp == 0 && s + e < n_steps) {
                    force_plane(cf, S.planes, masks_g, a_next);
                    if (lane == 0)
                        ctl[kCtlAct] = a_next;
                }
                if (obs_traj)
                    store_cells_steps<CellT>(cf, S.planes, obs_traj + ((size_t)s * cf.B + env) * HW,
                                             (size_t)cf.B * HW, e, tid, kThreads);
                __syncthreads();
                t += e;
                s += e - 1;
                continue;
            }
        }
        int rew;
        if (known) {
            rew = ctl[kCtlRew + a];
            __syncthreads();  // every warp has read this step's action
        } else {
            int warp_rew = 0;
            const bool any = block_match<SM, false>(cf, bs, tb, S, vm_g, cf.NW, 0, slot, warp_rew);
            int bits = block_combine(cf, S, any);
            bits = __reduce_or_sync(0xffffffffu, (unsigned)bits);
            if (lane == 0) {
                ctl[warp] = warp_rew;
                if (bits)
                    atomicOr(ctl + kCtlBits + parity, bits);
            }
            __syncthreads();  // the board after its step, rewards, bits
            bits = ctl[kCtlBits + parity];
            rew = block_reward(S);
            parity ^= 1;
            const bool changed = bits & 1;
            goal_left = cf.ch_goal < 0 || (bits & 2);
            at_init = at_init && !changed;
            if (tid == 0) {
                ctl[kCtlBits + parity] = 0;  // last read before the previous step's closing barrier
                if (changed) {
                    ctl[kCtlKnown] = 0;
                } else {  // remember the step: it left the board as it was
                    ctl[kCtlKnown] |= 1 << a;
                    ctl[kCtlRew + a] = rew;
                }
            }
        }
        t += 1;
        const bool done = !goal_left || (cf.max_steps > 0 && t >= cf.max_steps);
        if (done && cf.auto_reset) {
            t = 0;
            if (!at_init) {  // (else there is nothing to restore, and what is remembered holds)
                block_load_planes<CellT>(cf, init + (size_t)env * HW, S.planes);
                __syncthreads();
                if (tid == 0)
                    ctl[kCtlKnown] = 0;
                at_init = true;
            }
        }
        if (warp == 0) {
            sum += rew;
            if (lane == 0) {
                if (rew_traj)
                    rew_traj[(size_t)s * cf.B + env] = rew;
                if (done_traj)
                    done_traj[(size_t)s * cf.B + env] = (uint8_t)done;
            }
            if (s + 1 < n_steps) {
                const int a_next = S.acts[(s + 1) & (kActChunk - 1)];
                force_plane(cf, S.planes, masks_g, a_next);
                if (lane == 0)
                    ctl[kCtlAct] = a_next;
            }
        }
        if (obs_traj)
            store_cells<CellT>(cf, S.planes, obs_traj + ((size_t)s * cf.B + env) * HW, tid, kThreads);
        __syncthreads();
    }
    store_cells<CellT>(cf, S.planes, cur + (size_t)env * HW, tid, kThreads);
    if (tid == 0) {
        tsteps[env] = t;
        if (rew_sum)
            rew_sum[env] = sum;
        if (ctl[kCtlWarn])
            atomicOr(status + 1, kWarnAction);
    }
}

// CTAs per SM to run with: three (80 registers a thread), four (64) for batches of more
// than one wave of three whose boards leave the shared memory for it at as many rules
// per chunk.  us with three and four: 2000 boards of 23 x 41 with 2 rules, 20 steps 154 /
// 137, with 16 rules 567 / 524; 2000 of 40 x 40 with 64 rules 2974 / 2759; 300 of 23 x 41
// with 2 rules 40.9 / 42.9; 2000 of 64 x 64 x 16 with 24 rules, which four leave fewer
// per chunk, 2115 / 2135.  Five (48) are slower: 143, 560, 2986.
int block_ctas(const DevConfig &cf)
{
    if (cf.B <= 152 * kBlkCtas)
        return kBlkCtas;
    const BlockShape three = block_shape_fit(cf, cf.NW, 0, 0);
    const bool four = (kBlkCtas + 1) * (block_layout(cf, three, 0, 0).total + 1024) <= 228 * 1024;
    return four ? kBlkCtas + 1 : kBlkCtas;
}

}  // namespace

cudaError_t configure_block()
{
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *fn) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemLimit);
    };
#define AV_SET(CELL, CTAS)                                       \
    set((const void *)rollout_kernel<CELL, true, true, CTAS>);   \
    set((const void *)rollout_kernel<CELL, false, true, CTAS>);  \
    set((const void *)rollout_kernel<CELL, true, false, CTAS>);  \
    set((const void *)rollout_kernel<CELL, false, false, CTAS>);
    AV_SET(uint8_t, kBlkCtas)
    AV_SET(uint8_t, kBlkCtas + 1)
    AV_SET(uint16_t, kBlkCtas)
    AV_SET(uint16_t, kBlkCtas + 1)
#undef AV_SET
    return e;
}

void launch_rollout_block(const DevConfig &cf, const uint32_t *vm, const uint32_t *masks, void *cur, const void *init, int32_t *t,
                          int n_steps, uint64_t seed, const uint8_t *actions, void *obs_traj,
                          int32_t *rew_traj, uint8_t *done_traj, int32_t *rew_sum, uint32_t *status,
                          cudaStream_t st)
{
    const int ctas = block_ctas(cf);
    const BlockShape bs = block_shape_fit(cf, cf.NW, 0, 0);
    const size_t sm = block_layout(cf, bs, 0, 0).total;
#define AV_CTAS(CELL, SM, RUNS, CTAS)                                                       \
    rollout_kernel<CELL, SM, RUNS, CTAS><<<cf.B, kThreads, sm, st>>>(                       \
        cf, bs, vm, masks, (CELL *)cur, (const CELL *)init, t, n_steps, seed, actions,      \
        (CELL *)obs_traj, rew_traj, done_traj, rew_sum, status)
#define AV_LAUNCH(CELL, SM, RUNS)                  \
    if (ctas == kBlkCtas)                          \
        AV_CTAS(CELL, SM, RUNS, kBlkCtas);         \
    else                                           \
        AV_CTAS(CELL, SM, RUNS, kBlkCtas + 1);
#define AV_RUNS(CELL, SM)                  \
    if (n_steps == 1) {                    \
        AV_LAUNCH(CELL, SM, false)         \
    } else {                               \
        AV_LAUNCH(CELL, SM, true)          \
    }
    if (cf.cell_bytes == 1) {
        if (cf.pk_staged) {
            AV_RUNS(uint8_t, true)
        } else {
            AV_RUNS(uint8_t, false)
        }
    } else {
        if (cf.pk_staged) {
            AV_RUNS(uint16_t, true)
        } else {
            AV_RUNS(uint16_t, false)
        }
    }
#undef AV_RUNS
#undef AV_LAUNCH
#undef AV_CTAS
}

}  // namespace av
