// k_expand.cu -- tree-search expansion kernels: one warp per parent for boards
// of at most 16 plane words, one CTA per parent otherwise.
#include "block_step.cuh"

namespace av {
namespace {

// Tree-search expansion: one CTA per parent, the 5 children in turn.
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
        for (int i = tid; i < C * NW; i += kThreads) {  // child planes, kept in SET's place
            const int c = i / NW, w = i - c * NW;
            const uint32_t d = S.planes[c * NWP + w].x;
            uint32_t v = d;
            if (any) {
                v = (d & ~S.clrp[i]) | (~d & S.setp[i]);
                S.clrp[i] = 0u;
            }
            S.setp[i] = v;
        }
        __syncthreads();
        uint16_t *cells = S.cells + (size_t)a * HW;
        CellT *dst = children + ((size_t)node * 5 + a) * HW;
        int goal = 0;
        for (int p = tid; p < HW; p += kThreads) {
            const uint32_t v = gather_cell(cf, nullptr, S.setp, p);
            cells[p] = (uint16_t)v;
            dst[p] = (CellT)v;
            if (cf.ch_goal >= 0)
                goal |= (int)((v >> cf.ch_goal) & 1u);
        }
        const int goal_left = __syncthreads_or(goal) || cf.ch_goal < 0;
        if (tid == 0) {
            rewards[(size_t)node * 5 + a] = block_reward(S);
            if (done)
                done[(size_t)node * 5 + a] = (uint8_t)!goal_left;
        }
        for (int i = tid; i < C * NW; i += kThreads)
            S.setp[i] = 0u;
    }
    __syncthreads();
    // FNV-1a 64 over the canonical bytes, one thread per child
    if ((tid & 31) == 0 && warp < 5) {
        const uint16_t *gc = S.cells + (size_t)warp * HW;
        uint64_t hsh = 0xcbf29ce484222325ULL;
        for (int p = 0; p < HW; ++p) {
            const uint32_t v = gc[p];
            hsh = (hsh ^ (v & 0xffu)) * 0x100000001b3ULL;
            if (sizeof(CellT) == 2)
                hsh = (hsh ^ (v >> 8)) * 0x100000001b3ULL;
        }
        hashes[(size_t)node * 5 + warp] = hsh;
    }
}

// Parents per CTA on the warp path: 1 while the GPU has room for every warp at
// once (best balance), more for large batches.  The count divides F so that
// a CTA's parents share one environment (and its rule table).
int warps_per_cta(long long units, int F)
{
    int w = units <= 152LL * 32 ? 1 : (units <= 152LL * 64 ? 2 : kWarpCtaMax);
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
void warp_t(const DevConfig &cf, const uint32_t *arena, const uint32_t *tab_off, const uint32_t *vm,
            const uint32_t *masks, const void *parents, int F, const int32_t *n_parent, void *children,
            int32_t *rewards, uint8_t *done, uint64_t *hashes, cudaStream_t st)
{
    const long long units = (long long)cf.B * F;
    const int wpc = warps_per_cta(units, F);
    const unsigned grid = (unsigned)((units + wpc - 1) / wpc);
    const ExpandLayout L = expand_layout(cf);
    const size_t sm = L.warps + (size_t)wpc * L.per_warp;
    if (cf.rule_words > 0)
        expand_warp_kernel<CellT, NA, true><<<grid, 32 * wpc, sm, st>>>(
            cf, arena, tab_off, vm, masks, (const CellT *)parents, F, n_parent, (CellT *)children, rewards,
            done, hashes);
    else
        expand_warp_kernel<CellT, NA, false><<<grid, 32 * wpc, sm, st>>>(
            cf, arena, tab_off, vm, masks, (const CellT *)parents, F, n_parent, (CellT *)children, rewards,
            done, hashes);
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

void launch_expand(const DevConfig &cf, const uint32_t *arena, const uint32_t *tab_off, const uint32_t *vm,
                   const uint32_t *masks, const void *parents, int F, const int32_t *n_parent, void *children,
                   int32_t *rewards, uint8_t *done, uint64_t *hashes, cudaStream_t st)
{
    const bool u8 = cf.cell_bytes == 1;
    if (use_warp_expand(cf)) {
        if (cf.NA == 1) {
            if (u8)
                warp_t<uint8_t, 1>(cf, arena, tab_off, vm, masks, parents, F, n_parent, children, rewards, done,
                                      hashes, st);
            else
                warp_t<uint16_t, 1>(cf, arena, tab_off, vm, masks, parents, F, n_parent, children, rewards,
                                       done, hashes, st);
        } else {
            if (u8)
                warp_t<uint8_t, 2>(cf, arena, tab_off, vm, masks, parents, F, n_parent, children, rewards, done,
                                      hashes, st);
            else
                warp_t<uint16_t, 2>(cf, arena, tab_off, vm, masks, parents, F, n_parent, children, rewards,
                                       done, hashes, st);
        }
        return;
    }
    if (u8)
        block_t<uint8_t>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
    else
        block_t<uint16_t>(cf, vm, masks, parents, F, n_parent, children, rewards, done, hashes, st);
}

}  // namespace av
