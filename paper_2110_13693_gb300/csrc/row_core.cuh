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

// ------------------------------------------------- a warp's rows of tours
// A warp takes up to 32 tours, one a lane, possibly changed by a move, as
// many of one plan at a time as its rows of shared memory hold.  Tour by tour
// the lanes take the tour's orders (the next tours' ids and line ranges in
// flight), or every lane takes its own tour's where they are few, and put its
// lines' SKUs, the moved ones already exchanged, into the tour's row; then the
// slot-map gathers of all rows run flat, eight a lane in flight; then the rows
// are sorted (sort_rows).  No dependent gather per line and few registers.
constexpr int ROW_WARPS = 4;                // warps of a CTA
constexpr int ROW_THREADS = ROW_WARPS * 32;
constexpr int ROW_WORDS = 2048;             // keys of a warp's rows: 32 tours of 64 lines
constexpr uint32_t SKU_BAD = 0x7FFFFFFFu;   // in a row before the gathers: unusable SKU
constexpr uint32_t SKU_AT = 0x80000000u;    // a relocated SKU: SKU_AT | its location
constexpr size_t ROW_SMEM = sizeof(uint32_t) * ROW_WORDS * ROW_WARPS;

// per warp, in shared memory
struct RowList {
    uint16_t base[32], list[32];
    uint8_t n[32];
};

// A lane's tour: sequence positions q0 .. q1 - 1 of checked order ids, at most
// ub <= ROW_MAXN lines.  mv: {type, a, b, plan} of the move that changes it
// (type 0 for none), tk: {-, -, order of the move's list or -, order removed
// or list tag or -1}; add: the order added, or -1.
struct RowTour {
    int q0, q1, ub, add;
    int4 tk, mv;
};

__device__ __forceinline__ int order_lines_checked(const EvalArgs& a, int o, int& lb, int& le) {
    if ((unsigned)o >= (unsigned)a.n_orders) return -1;
    lb = a.order_off[o];
    le = a.order_off[o + 1];
    if (lb < 0 || le < lb || le > a.n_lines) return -1;
    return le - lb;
}

// Tours per warp and turn that give every warp of the grid work (32 where
// there is enough: a warp reads its tours one after another).
inline int row_unit(int64_t items, int64_t warps) {
    const int64_t u = (items + warps - 1) / warps;
    return u < 4 ? 4 : u > 32 ? 32 : (int)u;
}

// CTAs per SM of a kernel over rows
template <typename K>
cudaError_t rows_per_sm(K kern, int* per_sm) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ROW_SMEM);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, kern, ROW_THREADS, ROW_SMEM);
    if (e == cudaSuccess && *per_sm < 1) e = cudaErrorInvalidConfiguration;
    return e;
}

// The tour of one lane into its row, order by order (four orders' ids and line
// ranges, then four lines' SKUs, in flight), the move applied.
__device__ __forceinline__ void walk_row_lane(const EvalArgs& a, const RowTour& w, uint32_t* row, int& n, bool& primary) {
    const bool swap = w.mv.x >= 2;
    const int rem = !swap && w.tk.w >= 0 ? w.tk.w : -1, q_end = w.add >= 0 ? w.q1 + 1 : w.q1;
    int hit_min = 0x7fffffff;
    bool own_has_s1 = false;
    uint32_t* at = row;
    for (int q = w.q0; q < q_end; q += 4) {
        int o[4], lb[4], le[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) o[u] = q + u < w.q1 ? a.order_seq[q + u] : q + u < q_end ? w.add : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            lb[u] = le[u] = 0;
            if (o[u] >= 0 && !(q + u < w.q1 && o[u] == rem)) {
                lb[u] = a.order_off[o[u]];
                le[u] = a.order_off[o[u] + 1];
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            for (int l = lb[u]; l < le[u]; l += 4) {
                uint32_t sk[4];
#pragma unroll
                for (int v = 0; v < 4; ++v) sk[v] = l + v < le[u] ? (uint32_t)a.line_sku[l + v] : SKU_BAD;
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    if (l + v >= le[u]) continue;
                    uint32_t k = sk[v] < (uint32_t)a.n_sku ? sk[v] : SKU_BAD;
                    const bool s1 = k == (uint32_t)w.mv.y;
                    if (swap && (s1 || (w.mv.x == 2 && k == (uint32_t)w.mv.z))) {
                        hit_min = min(hit_min, o[u]);
                        own_has_s1 |= s1 && o[u] == w.tk.z;
                        k = w.mv.x == 3 ? SKU_AT | (uint32_t)w.mv.z : (uint32_t)(s1 ? w.mv.z : w.mv.y);
                    }
                    *at++ = k;
                }
            }
        }
    }
    n = (int)(at - row);
    primary = !swap || (hit_min == w.tk.z && (w.tk.w == -2 || !own_has_s1));
}

// Runs the lanes of `todo`.  For every batch done(mine, primary, base, n, bad)
// is called by the whole warp: whether this lane's task is in the batch,
// whether it is the counted one of its tour (only those rows are sorted), its
// row's place and length, and whether some row holds a line without a usable
// location (it sorts to its row's end).
template <typename Done>
__device__ __forceinline__ void run_rows(const EvalArgs& a, uint32_t* rows, RowList& rl, const RowTour& w, unsigned todo,
                                         int lane, Done done) {
    const unsigned lt_mask = (1u << lane) - 1u;
    uint16_t* bases = rl.base;
    uint16_t* list = rl.list;
    uint8_t* ns = rl.n;
    while (todo) {
        // the next tasks of one plan that fit the rows
        const int plan = __shfl_sync(0xffffffffu, w.mv.w, __ffs(todo) - 1);
        const bool cand = ((todo >> lane) & 1u) && w.mv.w == plan;
        const int incl = warp_inclusive_scan(cand ? w.ub : 0);
        const bool mine = cand && incl <= ROW_WORDS;
        const unsigned take = __ballot_sync(0xffffffffu, mine);
        const int total = __shfl_sync(0xffffffffu, incl, 31 - __clz(take));
        todo &= ~take;
        const int base = mine ? incl - w.ub : 0;
        const int32_t* map = a.slot_map + (int64_t)plan * a.slot_stride;
        bool primary = true;
        int n = 0;
        const int orders = mine ? w.q1 - w.q0 + (w.add >= 0 ? 1 : 0) : 0;
        if (3 * (int)__reduce_max_sync(0xffffffffu, (unsigned)orders) <= 2 * __popc(take)) {
            // every lane its own: 131,072 moves on tours of one order 330 us
            // tour by tour, 211 so, and with a very popular SKU 580 and 301
            // (of 16 orders 357 and 333; of 24 it takes as long or longer)
            if (mine) walk_row_lane(a, w, rows + base, n, primary);
        } else {
            // ids two tasks ahead, line ranges one task ahead
            int j = __ffs(take) - 1, j2 = j;
            unsigned left = take & (take - 1);
            auto first_ids = [&](int k) {
                const int b0 = __shfl_sync(0xffffffffu, w.q0, k), b1 = __shfl_sync(0xffffffffu, w.q1, k);
                return b0 + lane < b1 ? a.order_seq[b0 + lane] : -1;
            };
            int o_cur = first_ids(j), o_nxt = -1;
            int lb_cur = 0, le_cur = 0;
            if (o_cur >= 0) {
                lb_cur = a.order_off[o_cur];
                le_cur = a.order_off[o_cur + 1];
            }
            if (left) {
                j2 = __ffs(left) - 1;
                o_nxt = first_ids(j2);
            }
            for (;;) {
                const int b0 = __shfl_sync(0xffffffffu, w.q0, j), b1 = __shfl_sync(0xffffffffu, w.q1, j);
                const int jadd = __shfl_sync(0xffffffffu, w.add, j), jbase = __shfl_sync(0xffffffffu, base, j);
                const int type = __shfl_sync(0xffffffffu, w.mv.x, j);
                const int mb = __shfl_sync(0xffffffffu, w.mv.y, j), mc = __shfl_sync(0xffffffffu, w.mv.z, j);
                const int tz = __shfl_sync(0xffffffffu, w.tk.z, j), tw = __shfl_sync(0xffffffffu, w.tk.w, j);
                const int jj = j;
                const bool more = left != 0;
                int o0 = o_cur, lb0 = lb_cur, le0 = le_cur;   // this lane's order of the first 32
                j = j2;
                o_cur = o_nxt;
                lb_cur = le_cur = 0;
                if (more) {
                    if (o_cur >= 0) {
                        lb_cur = a.order_off[o_cur];
                        le_cur = a.order_off[o_cur + 1];
                    }
                    left &= left - 1;
                    if (left) {
                        j2 = __ffs(left) - 1;
                        o_nxt = first_ids(j2);
                    }
                }
                const bool swap = type >= 2;
                const int rem = !swap && tw >= 0 ? tw : -1;
                const int b_end = jadd >= 0 ? b1 + 1 : b1;
                if (b0 + lane < b1) {
                    if (o0 == rem) lb0 = le0 = 0;
                } else if (b0 + lane < b_end) {   // the added order comes last
                    o0 = jadd;
                    lb0 = a.order_off[o0];
                    le0 = a.order_off[o0 + 1];
                }
                uint32_t* row = rows + jbase;
                // the lines' indices at their places (lanes over orders;
                // ids and line counts were checked with the tour's count)
                int cnt_all = 0;
                for (int qb = b0; qb < b_end; qb += 32) {
                    int lb = lb0, le = le0;
                    if (qb > b0) {
                        const int q = qb + lane;
                        lb = le = 0;
                        if (q < b_end) {
                            const int o = q < b1 ? a.order_seq[q] : jadd;
                            if (!(q < b1 && o == rem)) {
                                lb = a.order_off[o];
                                le = a.order_off[o + 1];
                            }
                        }
                    }
                    const int cnt = le - lb;
                    const int inc = warp_inclusive_scan(cnt);
                    uint32_t* at = row + cnt_all + inc - cnt;
                    for (int l = lb; l < le; ++l) *at++ = (uint32_t)l;
                    cnt_all += __shfl_sync(0xffffffffu, inc, 31);
                }
                __syncwarp();
                // their SKUs, the move applied: an exchanged SKU takes the
                // other's place, a relocated one its new location
                int hit_min = 0x7fffffff;
                bool own_has_s1 = false;
                for (int x0 = 0; x0 < cnt_all; x0 += 64) {
                    int l[2];
                    uint32_t sk[2];
    #pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int x = x0 + 32 * u + lane;
                        l[u] = x < cnt_all ? (int)row[x] : -1;
                        sk[u] = l[u] >= 0 ? (uint32_t)a.line_sku[l[u]] : SKU_BAD;
                    }
    #pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        uint32_t k = sk[u] < (uint32_t)a.n_sku ? sk[u] : SKU_BAD;
                        if (swap) {
                            const bool s1 = k == (uint32_t)mb, hit = s1 || (type == 2 && k == (uint32_t)mc);
                            // a moved SKU's line: the order that holds it
                            // (a SKU move keeps every order of the tour)
                            for (unsigned hits = __ballot_sync(0xffffffffu, hit); hits; hits &= hits - 1) {
                                const int src = __ffs(hits) - 1;
                                const int hl = __shfl_sync(0xffffffffu, l[u], src);
                                const bool h1 = __shfl_sync(0xffffffffu, (int)s1, src) != 0;
                                for (int qb = b0; qb < b1; qb += 32) {
                                    int o = o0, lb = lb0, le = le0;
                                    if (qb > b0) {
                                        lb = le = 0;
                                        if (qb + lane < b1) {
                                            o = a.order_seq[qb + lane];
                                            lb = a.order_off[o];
                                            le = a.order_off[o + 1];
                                        }
                                    }
                                    if (hl >= lb && hl < le) {
                                        hit_min = min(hit_min, o);
                                        own_has_s1 |= h1 && o == tz;
                                    }
                                }
                            }
                            if (hit) k = type == 3 ? SKU_AT | (uint32_t)mc : (uint32_t)(s1 ? mc : mb);
                        }
                        if (l[u] >= 0) row[x0 + 32 * u + lane] = k;
                    }
                }
                if (swap) {
                    hit_min = __reduce_min_sync(0xffffffffu, hit_min);
                    own_has_s1 = __any_sync(0xffffffffu, own_has_s1);
                }
                if (lane == jj) {
                    n = cnt_all;
                    primary = !swap || (hit_min == tz && (tw == -2 || !own_has_s1));
                }
                if (!more) break;
            }
        }
        __syncwarp();
        // keys, all rows at once (what lies between rows is translated
        // too and read by nobody)
        bool bad = false;
        for (int x0 = lane; x0 < total; x0 += 256) {
            uint32_t sk[8];
            int loc[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) sk[u] = x0 + 32 * u < total ? rows[x0 + 32 * u] : SKU_BAD;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                loc[u] = sk[u] < (uint32_t)a.n_sku ? map[sk[u]] : ((sk[u] & SKU_AT) ? (int)(sk[u] & ~SKU_AT) : -1);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (x0 + 32 * u >= total) continue;
                const bool in = (uint32_t)loc[u] < (uint32_t)a.g.n_loc;
                bad |= !in;
                rows[x0 + 32 * u] = in ? loc_key(a.g, loc[u]) : KEY_BAD;
            }
        }
        bad = __any_sync(0xffffffffu, bad);
        // sort: those over 64 lines first
        const bool cost = mine && primary;
        const unsigned big = __ballot_sync(0xffffffffu, cost && n > 64), all = __ballot_sync(0xffffffffu, cost);
        const int n_big = __popc(big), n_all = __popc(all);
        if (mine) {
            bases[lane] = (uint16_t)base;
            ns[lane] = (uint8_t)n;
        }
        if (cost) list[n > 64 ? __popc(big & lt_mask) : n_big + __popc(all & ~big & lt_mask)] = (uint16_t)lane;
        __syncwarp();
        for (int k = 0; k < n_all;) {
            const int G = k < n_big ? 8 : 4, end = k < n_big ? n_big : n_all;
            sort_rows(G, rows, list, bases, ns, k, end, lane);
            k = min(k + 32 / G, end);
        }
        __syncwarp();
        done(mine, primary, base, n, bad);
        __syncwarp();
    }
}

}  // namespace
}  // namespace wh
