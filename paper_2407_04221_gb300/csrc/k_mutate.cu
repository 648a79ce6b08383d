// k_mutate.cu -- the mutation operators of the evolution loop (Sec. 3.1.1):
// bits of the initial maps flipped at random, tiles of the mutable rules'
// input and output patterns changed, rule rewards redrawn.  Every decision
// is one counter draw,
//     draw(seed, st, a, b, c) = mix(mix(mix(seed + golden*(st+1)) ^ a) ^ (b<<32 | c)),
// taken when its top 24 bits are below the rate (in units of 2^-24):
//   map bit (cell q, channel c) of env b:      st 9,  a = b, b = q,          c = c
//   input entry (rule r, entry e, channel c):   st 10, a = t, b = 25 r + e,   c = c
//   output entry (rule r, entry e, channel c):  st 11, a = t, b = 25 r + e,   c = c
//   reward of rule r:                           st 12, a = t, b = r, c = 0 (decision), 1 (value)
// A changed ternary entry moves to the next state (cyclically) when bit 39 of
// its draw is 0, to the one after when 1.
//
// One warp per environment (map) or rule table; rule entries are dealt to lanes
// from a dense list of the table's existing (rule, entry) pairs.  What bounds it:
// integer issue, one mix per decision.  The first two mixes depend only on (seed,
// stream, environment).  Of the third, the channels c of one cell or entry differ in
// the low five bits of the state only (z >> 30 does not reach them), so the first
// product for each is another one's plus or minus a multiple of the constant, and
// decisions read bits 39..63 only, so the second needs its upper word alone.  The
// channel count is a template argument: every channel's path is straight-line code.
// 16,384 maps of 16 x 16 x 10 and tables of 12 rules: 114.6 us with a whole mix per
// decision (33 instructions), 72.8 with the products shared, 61.9 unrolled, 54.3 in one launch.
#include <algorithm>
#include <type_traits>

#include "launch.h"

namespace av {
namespace {

constexpr int kMutThreads = 128;

// mix(mix(seed + golden*(st+1)) ^ a): the part of draw() shared by every
// decision of one environment in one stream.
__device__ __forceinline__ uint64_t draw_prefix(uint64_t seed, uint64_t st, uint64_t a)
{
    return mix64(mix64(seed + 0x9E3779B97F4A7C15ULL * (st + 1)) ^ a);
}

__device__ __forceinline__ uint64_t draw_from(uint64_t prefix, uint64_t b, uint64_t c)
{
    return mix64(prefix ^ ((b << 32) | c));
}

constexpr uint64_t kMixOne = 0xbf58476d1ce4e5b9ULL;  // mix64's first factor

// The upper word of a draw from its state after mix64's first product: the last
// xor-shift changes none of the bits that decisions read (and the lowest bit only).
__device__ __forceinline__ uint32_t draw_upper(uint64_t p)
{
    const uint64_t x = p ^ (p >> 27);
    const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32);
    return __umulhi(lo, 0x133111ebu) + lo * 0x94d049bbu + hi * 0x133111ebu;
}

// The decisions of one (prefix, b) for c = 0..N-1: bit c of `hit` when
// draw(.., b, c) >> 40 < p (`last` = (p << 8) - 1, p >= 1), bit c of `far` is bit 39
// of the draw.  The first product for c is the one for c without its lowest set bit
// i plus or minus the constant times 2^i, as bit i of the state's low five bits is
// clear or set.
template <int N>
__device__ __forceinline__ void draw_row(uint64_t prefix, uint32_t b, uint32_t last, uint32_t &hit, uint32_t &far)
{
    const uint64_t z = prefix ^ ((uint64_t)b << 32);
    const uint64_t y = z ^ (z >> 30);
    uint64_t p[N];
    hit = far = 0;
#pragma unroll
    for (int c = 0; c < N; ++c) {
        if (c == 0) {
            p[0] = y * kMixOne;
        } else {
            const int i = (c & 1) ? 0 : (c & 2) ? 1 : (c & 4) ? 2 : (c & 8) ? 3 : 4;
            const uint64_t d = (y >> i) & 1u ? 0ull - (kMixOne << i) : kMixOne << i;
            p[c] = p[c & (c - 1)] + d;
        }
        const uint32_t u = draw_upper(p[c]);
        if (u <= last)
            hit |= 1u << c;
        far |= (c < 7 ? u >> (7 - c) : u << (c - 7)) & (1u << c);
    }
}

// Map b of this warp.  `few`: only the channels that may flip are drawn, one by one
// (see mutate_few).
template <typename CellT, int C>
__device__ __forceinline__ void mutate_map(int b, int HW, uint32_t p_map, uint32_t channels, bool few, uint64_t seed,
                                           CellT *maps)
{
    const int lane = threadIdx.x & 31;
    const uint32_t last = (p_map << 8) - 1u;  // d >> 40 < p_map: upper word at most this (p_map >= 1)
    const uint64_t pre = draw_prefix(seed, 9, (uint64_t)b);
    CellT *m = maps + (size_t)b * HW;
    if (few) {
        for (int q = lane; q < HW; q += 32) {
            const uint64_t z = pre ^ ((uint64_t)q << 32), y = z ^ (z >> 30);
            uint32_t flip = 0;
            for (uint32_t x = channels; x; x &= x - 1u) {
                const uint32_t c = (uint32_t)__ffs(x) - 1u;
                if (draw_upper((y ^ c) * kMixOne) <= last)
                    flip |= 1u << c;
            }
            if (flip)
                m[q] = (CellT)(m[q] ^ flip);
        }
        return;
    }
    for (int q = lane; q < HW; q += 32) {
        uint32_t flip, far;
        draw_row<C>(pre, (uint32_t)q, last, flip, far);
        flip &= channels;
        if (flip)
            m[q] = (CellT)(m[q] ^ flip);
    }
}

// Packed record as 32-bit words: [0] h | w << 8, [1] reward, [2 + e] present,
// [27 + e] absent, [52 + e] set, [77 + e] clear.
constexpr int kRecWords = 102;

// New ternary states of the mask pair (one, two) of one entry from the decisions of
// its channels: those that change (hit), and which way (far, bit 39 of their draws).
__device__ __forceinline__ void mutate_entry(uint32_t &one, uint32_t &two, uint32_t hit, uint32_t far)
{
    const uint32_t o = one, t = two & ~one, z = ~(one | two);  // states 1, 2, 0
    one = (o & ~hit) | (hit & ((z & ~far) | (t & far)));
    two = (two & ~hit) | (hit & ((o & ~far) | (z & far)));
}

// Rule table t of this warp.
template <int C>
__device__ __forceinline__ void mutate_table(int t, int R, uint32_t p_rule, uint32_t p_reward, int32_t reward_min,
                                             uint64_t reward_span, uint64_t mutable_rules, uint64_t seed,
                                             uint32_t *rules)
{
    // Per warp: offsets of each rule's entries in the dense list of the
    // table's mutable (rule, pattern entry) pairs, so that lanes stride over
    // entries that exist (a 1 x 2 pattern has 2 of the 25 slots).
    __shared__ int s_off[kMutThreads / 32][2 * 32 + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int *off = s_off[wid];
    const int halves = R > 32 ? 2 : 1;
    const uint32_t last = (p_rule << 8) - 1u;  // d >> 40 < p_rule: upper word at most this (p_rule >= 1)
    uint32_t *tab = rules + (size_t)t * R * kRecWords;
    if (p_rule > 0) {
        int total = 0;
        for (int half = 0; half < halves; ++half) {  // rules lane and lane + 32
            const int r = lane + 32 * half;
            int n = 0;
            if (r < R && ((mutable_rules >> r) & 1u)) {
                const uint32_t hw = tab[(size_t)r * kRecWords];
                n = min(25, (int)(hw & 0xffu) * (int)((hw >> 8) & 0xffu));  // 25 entries per record
            }
            for (int d = 1; d < 32; d <<= 1) {  // inclusive scan
                const int v = __shfl_up_sync(0xffffffffu, n, d);
                if (lane >= d)
                    n += v;
            }
            off[1 + 32 * half + lane] = total + n;
            total += __shfl_sync(0xffffffffu, n, 31);
        }
        if (lane == 0)
            off[0] = 0;
        __syncwarp();
        const uint64_t pre_in = draw_prefix(seed, 10, (uint64_t)t);
        const uint64_t pre_out = draw_prefix(seed, 11, (uint64_t)t);
        for (int j = lane; j < total; j += 32) {
            int lo = 0, hi = 32 * halves;  // the rule r with off[r] <= j < off[r + 1]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (off[mid] <= j)
                    lo = mid;
                else
                    hi = mid;
            }
            const int r = lo, e = j - off[r];
            const uint32_t k = (uint32_t)(25 * r + e);
            uint32_t *rec = tab + (size_t)r * kRecWords;
            uint32_t pres = rec[2 + e], absn = rec[27 + e], set = rec[52 + e], clr = rec[77 + e];
            uint32_t hit, far;
            draw_row<C + 1>(pre_in, k, last, hit, far);
            mutate_entry(pres, absn, hit, far);
            draw_row<C>(pre_out, k, last, hit, far);
            mutate_entry(set, clr, hit, far);
            rec[2 + e] = pres;
            rec[27 + e] = absn;
            rec[52 + e] = set;
            rec[77 + e] = clr;
        }
    }
    if (p_reward > 0) {
        const uint64_t pre_rw = draw_prefix(seed, 12, (uint64_t)t);
        for (int r = lane; r < R; r += 32) {
            if (!((mutable_rules >> r) & 1u))
                continue;
            if ((uint32_t)(draw_from(pre_rw, (uint64_t)r, 0) >> 40) < p_reward) {
                const uint64_t u = draw_from(pre_rw, (uint64_t)r, 1) >> 32;
                tab[(size_t)r * kRecWords + 1] = (uint32_t)(reward_min + (int64_t)((u * reward_span) >> 32));
            }
        }
    }
}

// One warp per rule table, then one per map: one launch, so that the tables' loads
// and the maps' arithmetic share the SMs and there is one tail (61.4 us in two
// launches of persistent CTAs of 256 threads, 54.3 in one).
template <typename CellT, int C>
__global__ void __launch_bounds__(kMutThreads)
    mutate_kernel(int n_tables, int table_ctas, int R, uint32_t p_rule, uint32_t p_reward, int32_t reward_min,
                  uint64_t reward_span, uint64_t mutable_rules, uint32_t *rules, int n_maps, int HW, uint32_t p_map,
                  uint32_t channels, bool few, CellT *maps, uint64_t seed)
{
    const int wid = threadIdx.x >> 5;
    constexpr int kWarpsPerCta = kMutThreads / 32;
    if ((int)blockIdx.x < table_ctas) {
        const int t = (int)blockIdx.x * kWarpsPerCta + wid;
        if (t < n_tables)
            mutate_table<C>(t, R, p_rule, p_reward, reward_min, reward_span, mutable_rules, seed, rules);
    } else {
        const int b = ((int)blockIdx.x - table_ctas) * kWarpsPerCta + wid;
        if (b < n_maps)
            mutate_map<CellT, C>(b, HW, p_map, channels, few, seed, maps);
    }
}

// Whether a map's flippable channels are drawn one by one, with a first product each,
// instead of all C with shared products and a mask: a decision then takes about 1.6
// times the instructions.  16,384 maps of 16 x 16, us, all C and one by one:
//   C = 4    18.6, with 1 channel 12.0, 2 14.7, 3 18.6
//   C = 8    24.9 to 26.8, with 1 11.0, 4 21.0, 5 24.8, 6 28.7
//   C = 10   28.9 to 31.0, with 1 10.9, 5 24.8, 6 28.8, 8 35.0
//   C = 16   41.1 to 43.2, with 1 10.9, 5 24.8, 10 41.2, 12 47.3
inline bool mutate_few(int C, uint32_t channels) { return 8 * __builtin_popcount(channels) <= 5 * C; }

template <int C>
void mutate_t(int B, int HW, int R, uint32_t p_map, uint32_t channels, uint32_t p_rule, uint32_t p_reward,
              int32_t reward_min, uint64_t reward_span, uint64_t mutable_rules, uint64_t seed, void *maps,
              uint32_t *rules, cudaStream_t st)
{
    using CellT = std::conditional_t<(C <= 8), uint8_t, uint16_t>;
    const uint64_t mask = R >= 64 ? ~0ull : ((1ull << R) - 1ull);
    const int n_maps = maps != nullptr && p_map > 0 && channels != 0 ? B : 0;
    const int n_tables = rules != nullptr && R > 0 && (mutable_rules & mask) != 0 && (p_rule > 0 || p_reward > 0) ? B : 0;
    constexpr int kWarpsPerCta = kMutThreads / 32;
    const int table_ctas = n_tables / kWarpsPerCta + (n_tables % kWarpsPerCta != 0);
    const int map_ctas = n_maps / kWarpsPerCta + (n_maps % kWarpsPerCta != 0);
    if (table_ctas + map_ctas > 0)
        mutate_kernel<CellT, C><<<table_ctas + map_ctas, kMutThreads, 0, st>>>(
            n_tables, table_ctas, R, p_rule, p_reward, reward_min, reward_span, mutable_rules, rules, n_maps, HW, p_map,
            channels, mutate_few(C, channels), (CellT *)maps, seed);
}

}  // namespace

void launch_mutate(int B, int H, int W, int C, int R, uint32_t p_map, uint32_t map_channels, uint32_t p_rule,
                   uint32_t p_reward, int32_t reward_min, int32_t reward_max, uint64_t mutable_rules, uint64_t seed,
                   void *maps, uint32_t *rules, cudaStream_t st)
{
    const uint32_t channels = map_channels & ((1u << C) - 1u);
    const uint64_t span = (uint64_t)((int64_t)reward_max - (int64_t)reward_min + 1);
    switch (C) {  // (checked to be 1..16)
#define AV_CASE(N)                                                                                                  \
    case N:                                                                                                         \
        return mutate_t<N>(B, H * W, R, p_map, channels, p_rule, p_reward, reward_min, span, mutable_rules, seed,    \
                           maps, rules, st);
        AV_CASE(1) AV_CASE(2) AV_CASE(3) AV_CASE(4) AV_CASE(5) AV_CASE(6) AV_CASE(7) AV_CASE(8)
        AV_CASE(9) AV_CASE(10) AV_CASE(11) AV_CASE(12) AV_CASE(13) AV_CASE(14) AV_CASE(15) AV_CASE(16)
#undef AV_CASE
    }
}

}  // namespace av
