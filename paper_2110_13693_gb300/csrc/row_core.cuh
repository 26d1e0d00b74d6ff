// Tours as rows of 32-bit keys in shared memory: sorted in place by 2, 4 or 8
// lanes with 16 keys each, then costed in one pass by one lane.
#pragma once
#include "tour_core.cuh"

namespace wh {
namespace {

constexpr int ROW_MAXN = 128;    // keys of a row (8 lanes of 16)

// Markers of unusable lines (a key's aisle is at most 65,533, so both compare
// above every key); KEY_BAD: location out of range.
constexpr uint32_t KEY_BAD_SKU = 0xFFFFFFFDu;

// Sort the rows of tours list[i0 + lane / G] (those below i1), G = 2, 4 or 8
// lanes a tour with 16 keys each: a merge-exchange network in the lane, then
// bitonic merges across lanes.  One code for every G, its merge stages
// rolled: warps at different stages share the instruction cache (unrolled
// per G, warps of the move kernel waited for instructions more than they
// issued).
__device__ __forceinline__ void sort_rows(const int G, uint32_t* rows, const uint16_t* s_list, const uint16_t* s_base,
                                          const uint8_t* s_n, int i0, int i1, int lane) {
    const int sub = lane & (G - 1), i = i0 + lane / G;
    int n = 0;
    uint32_t* row = rows;
    if (i < i1) {
        const int k = s_list[i];
        n = s_n[k];
        row = rows + s_base[k];
    }
    uint32_t x[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) x[j] = j * G + sub < n ? row[j * G + sub] : KEY_NONE;
    merge_exchange<16>(x);
#pragma unroll 1
    for (int s = 1; s < G; s <<= 1) {
        // blocks of s lanes merged in pairs: every key against its mirror
        const bool low = (lane & s) == 0;
        uint32_t y[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) y[j] = __shfl_xor_sync(0xffffffffu, x[15 - j], 2 * s - 1);
#pragma unroll
        for (int j = 0; j < 16; ++j) x[j] = low ? min(x[j], y[j]) : max(x[j], y[j]);
#pragma unroll 1
        for (int d = s >> 1; d > 0; d >>= 1) {
            const bool l2 = (lane & d) == 0;
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const uint32_t o = __shfl_xor_sync(0xffffffffu, x[j], d);
                x[j] = l2 ? min(x[j], o) : max(x[j], o);
            }
        }
#pragma unroll
        for (int d = 8; d > 0; d >>= 1) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                if ((j ^ d) > j) {
                    const uint32_t p = x[j], r = x[j ^ d];
                    x[j] = min(p, r);
                    x[j ^ d] = max(p, r);
                }
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 16; ++j)
        if (sub * 16 + j < n) row[sub * 16 + j] = x[j];
}

// S-shape and optimal cost of a sorted row of n keys: an aisle ends where the
// next key's aisle is larger, and its DP step runs there.  Markers of unusable
// lines sort last and never end an aisle.
__device__ __forceinline__ void row_costs(const Geo& g, const DPConst& c, const uint32_t* row, int n, bool need_rr,
                                          int& cs, int& cr) {
    DP5 v;
    dp_init(v);
    int pa = 0, m = 0;
    uint32_t key = n > 0 ? row[0] : 0u, lo = key, gi = 0, last = 0;
    for (int p = 0; p < n; p += 4) {
        uint32_t nx[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) nx[j] = p + j + 1 < n ? row[p + j + 1] : KEY_NONE;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (nx[j] > (key | 0xFFFFu)) {
                const int ai = (int)(key >> 16);
                if (need_rr) dp_aisle_rel(v, c, ai - pa, (int)(lo & 0xFFFFu), (int)(key & 0xFFFFu), (int)gi);
                pa = ai;
                ++m;
                last = key;
                lo = nx[j];
                gi = 0;
            } else {
                gi = max(gi, nx[j] - key);
            }
            key = nx[j];
        }
    }
    cs = sshape_cost(g, m, (int)(last >> 16), (int)(last & 0xFFFFu));
    cr = need_rr ? dp_final(v) + c.p2 * pa : 0;
}

}  // namespace
}  // namespace wh
