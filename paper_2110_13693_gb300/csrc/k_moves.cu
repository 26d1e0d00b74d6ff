// Move-delta kernels for sm_103a: the change of a plan's S-shape and optimal
// costs under a neighbourhood move (Sec. 5: subroutine 4 evaluates a change of
// product position; the picking list decides which orders share a tour).
//
// Only the tours a move changes are re-costed:
//   order swap (o1, o2)     -> the two tours holding them, each with one order
//                              exchanged;
//   relocate (o, tour)      -> the source tour without o, the target with o;
//   SKU-slot swap (s1, s2)  -> every tour holding an order with s1 or s2,
//                              under the plan's slotting with the two
//                              locations exchanged.
// Pipeline: per-tour line counts and the plan's order -> tour map; the SKU ->
// orders index of the order book; per move a check, a status and a task count;
// an exclusive scan of the counts; the task list; a warp per 32 tasks (one for
// each task over ROW_MAXN lines) re-costing the changed tours and adding
// (new - old) into the move's two int64 deltas.  A SKU-swap move lists one task
// per (order with s1 or s2); of the tasks that land in the same tour only the
// one of the smallest such order counts, so no de-duplication pass is needed.
#include "row_core.cuh"
#include "feat_core.cuh"

namespace wh {

namespace {

// plan of global tour t: largest p with plan_tour_off[p] <= t
__device__ __forceinline__ int plan_of_tour(const EvalArgs& a, int t) {
    int lo = 0, hi = a.n_plans - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.plan_tour_off[mid] <= t) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void k_mv_tours(MoveArgs M) {
    const EvalArgs& a = M.a;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < a.n_tours; t += gridDim.x * blockDim.x) {
        const int p = plan_of_tour(a, t);
        const int q0 = a.tour_off[t], q1 = a.tour_off[t + 1];
        int lines = 0;
        if (q0 < 0 || q1 < q0 || (int64_t)q1 > a.n_seq) {
            flag(a.status, WH_STATUS_BAD_OFFSET);
            lines = -1;
        } else {
            for (int q = q0; q < q1; ++q) {
                const int o = a.order_seq[q];
                int lb, le;
                const int c = order_lines_checked(a, o, lb, le);
                if (c < 0) {
                    flag(a.status, WH_STATUS_BAD_ORDER);
                    lines = -1;
                    break;
                }
                lines += c;
                M.order_tour[(int64_t)p * a.n_orders + o] = t;
            }
        }
        M.tour_lines[t] = lines;
    }
}

// The same index built one plan per CTA (grid stride over plans): the
// plan's order -> tour row is filled in shared memory (-1 where the plan does
// not hold the order) and written out in one coalesced pass, so the table
// needs no clearing pass and no tour searches for its plan.  Used when a row
// fits MVT_MAX_ORDERS entries.
constexpr int MVT_THREADS = 256;
constexpr int MVT_MAX_ORDERS = 12288;   // 48 KB of shared memory

__global__ void __launch_bounds__(MVT_THREADS) k_mv_tours_plan(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ int32_t s_row[];
    const EvalArgs& a = M.a;
    for (int p = blockIdx.x; p < a.n_plans; p += gridDim.x) {
        for (int o = threadIdx.x; o < a.n_orders; o += blockDim.x) s_row[o] = -1;
        __syncthreads();
        int t0 = a.plan_tour_off[p], t1 = a.plan_tour_off[p + 1];
        if (t0 < 0 || t1 < t0 || t1 > a.n_tours || (p == 0 && t0 != 0) || (p == a.n_plans - 1 && t1 != a.n_tours)) {
            if (threadIdx.x == 0) flag(a.status, WH_STATUS_BAD_OFFSET);
            t0 = max(t0, 0);
            t1 = min(t1, a.n_tours);
        }
        for (int t = t0 + threadIdx.x; t < t1; t += blockDim.x) {
            const int q0 = a.tour_off[t], q1 = a.tour_off[t + 1];
            int lines = 0;
            if (q0 < 0 || q1 < q0 || (int64_t)q1 > a.n_seq) {
                flag(a.status, WH_STATUS_BAD_OFFSET);
                lines = -1;
            } else {
                // four orders' ids, then their line ranges, in flight
                for (int q = q0; q < q1 && lines >= 0; q += 4) {
                    int o[4], cnt[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) o[u] = q + u < q1 ? a.order_seq[q + u] : 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        int lb, le;
                        cnt[u] = q + u < q1 ? order_lines_checked(a, o[u], lb, le) : 0;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        if (q + u >= q1 || lines < 0) continue;
                        if (cnt[u] < 0) {
                            flag(a.status, WH_STATUS_BAD_ORDER);
                            lines = -1;
                        } else {
                            lines += cnt[u];
                            s_row[o[u]] = t;
                        }
                    }
                }
            }
            M.tour_lines[t] = lines;
        }
        __syncthreads();
        int32_t* row = M.order_tour + (int64_t)p * a.n_orders;
        for (int o = threadIdx.x; o < a.n_orders; o += blockDim.x) row[o] = s_row[o];
        __syncthreads();
    }
}

__global__ void k_mv_sku_count(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    const EvalArgs& a = M.a;
    for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < a.n_lines; l += gridDim.x * blockDim.x) {
        const int s = a.line_sku[l];
        if ((unsigned)s < (unsigned)a.n_sku) atomicAdd(&M.sku_cur[s], 1);
    }
}

// Places in sku_orders for every SKU's orders: a block scan of 1,024 SKUs'
// counts and one atomic a block for its place among the blocks (the lists'
// order does not matter), cursors reset.  One block scanning all of 50,000
// SKUs in turn took 49 us, 21 us with 16 SKUs a thread.
constexpr int SKU_ALLOC_T = 1024;

__global__ void __launch_bounds__(SKU_ALLOC_T) k_mv_sku_alloc(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    __shared__ int warp_tot[32];
    __shared__ int s_base;
    const int n = M.a.n_sku, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int i = blockIdx.x * SKU_ALLOC_T + tid;
    const int v = i < n ? M.sku_cur[i] : 0;
    const int incl = warp_inclusive_scan(v);
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int t = warp_tot[lane], tot = warp_inclusive_scan(t);
        warp_tot[lane] = tot - t;
        if (lane == 31) s_base = tot ? atomicAdd(&M.sku_cur[n], tot) : 0;
    }
    __syncthreads();
    if (i < n) {
        M.sku_off[i] = s_base + warp_tot[w] + incl - v;
        M.sku_cur[i] = 0;
    }
}

// Every order once in the list of each of its SKUs, also where the SKU is on
// several of its lines: a line is skipped when one before it has its SKU.  A
// lane looks back over the lines of its own order up to MVS_SERIAL lines, four
// lines' SKUs and then their places in flight; a longer order is taken by the
// whole warp, 32 lines at a time.
constexpr int MVS_SERIAL = 32;

__global__ void k_mv_sku_fill(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    const EvalArgs& a = M.a;
    const int lane = threadIdx.x & 31;
    auto place = [&](int s) { return M.sku_off[s] + atomicAdd(&M.sku_cur[s], 1); };
    auto put = [&](int s, int o, int k) {
        // (orders with malformed, overlapping line ranges hold more lines
        // than there are)
        if (k < a.n_lines) M.sku_orders[k] = o;
        else atomicSub(&M.sku_cur[s], 1);
    };
    for (int o0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); o0 < a.n_orders; o0 += gridDim.x * blockDim.x) {
        const int o = o0 + lane;
        int lb = 0, le = 0;
        if (o < a.n_orders && order_lines_checked(a, o, lb, le) < 0) lb = le = 0;
        const bool lng = le - lb > MVS_SERIAL;
        for (int l0 = lb; !lng && l0 < le; l0 += 4) {
            int s[4], k[4];
            bool add[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = l0 + u < le ? a.line_sku[l0 + u] : -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                add[u] = (unsigned)s[u] < (unsigned)a.n_sku;
#pragma unroll
                for (int v = 0; v < u; ++v) add[u] &= s[v] != s[u];
            }
            for (int l = lb; l < l0; ++l) {
                const int t = a.line_sku[l];
#pragma unroll
                for (int u = 0; u < 4; ++u) add[u] &= t != s[u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) k[u] = add[u] ? place(s[u]) : 0;
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (add[u]) put(s[u], o, k[u]);
        }
        for (unsigned longs = __ballot_sync(0xffffffffu, lng); longs; longs &= longs - 1) {
            const int src = __ffs(longs) - 1;
            const int b = __shfl_sync(0xffffffffu, lb, src), e = __shfl_sync(0xffffffffu, le, src);
            for (int l0 = b; l0 < e; l0 += 32) {
                const int s = l0 + lane < e ? a.line_sku[l0 + lane] : -1;
                // of equal SKUs among the 32 the first lane's line counts
                const unsigned same = __match_any_sync(0xffffffffu, s);
                bool add = (unsigned)s < (unsigned)a.n_sku && (same & ((1u << lane) - 1u)) == 0;
#pragma unroll 8
                for (int l = b; l < l0; ++l) add &= a.line_sku[l] != s;
                if (add) put(s, o0 + src, place(s));
            }
        }
    }
}

// status and task count of every move; deltas zeroed
__global__ void k_mv_count(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    const EvalArgs& a = M.a;
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M.n_moves; m += gridDim.x * blockDim.x) {
        const int4 mv = M.moves[m];
        M.delta[2 * m] = 0;
        M.delta[2 * m + 1] = 0;
        int st = 3, cnt = 0;
        const int p = mv.w;
        if (p >= 0 && p < a.n_plans) {
            const int64_t row = (int64_t)p * a.n_orders;
            if (mv.x == 0 || mv.x == 1) {
                int lb, le;
                const int la = order_lines_checked(a, mv.y, lb, le);
                const int ta = la >= 0 ? M.order_tour[row + mv.y] : -1;
                if (ta >= 0 && M.tour_lines[ta] >= 0) {
                    if (mv.x == 0) {
                        const int lbb = order_lines_checked(a, mv.z, lb, le);
                        const int tb = lbb >= 0 ? M.order_tour[row + mv.z] : -1;
                        if (tb >= 0 && M.tour_lines[tb] >= 0) {
                            if (ta == tb) st = 2;
                            else if (M.max_lines > 0 && (M.tour_lines[ta] - la + lbb > M.max_lines ||
                                                         M.tour_lines[tb] - lbb + la > M.max_lines)) st = 1;
                            else { st = 0; cnt = 2; }
                        }
                    } else {
                        const int n_t = a.plan_tour_off[p + 1] - a.plan_tour_off[p];
                        if (mv.z >= 0 && mv.z < n_t) {
                            const int tb = a.plan_tour_off[p] + mv.z;
                            if (tb == ta) st = 2;
                            else if (M.tour_lines[tb] < 0) st = 3;
                            else if ((M.max_orders > 0 && a.tour_off[tb + 1] - a.tour_off[tb] + 1 > M.max_orders) ||
                                     (M.max_lines > 0 && M.tour_lines[tb] + la > M.max_lines)) st = 1;
                            else { st = 0; cnt = 2; }
                        }
                    }
                }
            } else if (mv.x == 2) {
                if (a.slot_stride > 0 && (unsigned)mv.y < (unsigned)a.n_sku && (unsigned)mv.z < (unsigned)a.n_sku) {
                    if (mv.y == mv.z) st = 2;
                    else {
                        st = 0;
                        cnt = M.sku_cur[mv.y] + M.sku_cur[mv.z];
                    }
                }
            } else if (mv.x == 3) {
                // relocation of SKU mv.y to location mv.z, which must be empty
                if (a.slot_stride > 0 && a.loc_used && (unsigned)mv.y < (unsigned)a.n_sku &&
                    (unsigned)mv.z < (unsigned)a.g.n_loc) {
                    const int words = (a.g.n_loc + 31) >> 5;
                    const uint32_t used = a.loc_used[(int64_t)p * words + (mv.z >> 5)] >> (mv.z & 31) & 1u;
                    if (a.slot_map[(int64_t)p * a.slot_stride + mv.y] == mv.z) st = 2;
                    else if (!used) {
                        st = 0;
                        cnt = M.sku_cur[mv.y];
                    }
                }
            }
        }
        M.mstatus[m] = st;
        M.task_off[m] = cnt;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        M.task_off[M.n_moves] = 0;
        *M.long_count = 0;
        if (M.stats) M.stats[0] = M.stats[1] = 0;
    }
}

// ---- exclusive scan of int64 counts in place (n+1 entries): block scans,
// a scan of the block totals, then the carries added
constexpr int SCAN_T = 1024;

__device__ __forceinline__ long long block_excl_scan(long long v, long long* warp_tot, long long& total) {
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += u;
    }
    if (lane == 31) warp_tot[w] = x;
    __syncthreads();
    if (w == 0) {
        long long y = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, y, o);
            if (lane >= o) y += u;
        }
        warp_tot[lane] = y;
    }
    __syncthreads();
    total = warp_tot[(blockDim.x >> 5) - 1];
    const long long r = (w ? warp_tot[w - 1] : 0) + x - v;
    __syncthreads();
    return r;
}

__global__ void k_scan_blocks(int64_t* v, int64_t n, int64_t* block_tot) {
    pdl_trigger();
    pdl_wait();
    __shared__ long long wt[32];
    const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x;
    const long long x = i < n ? v[i] : 0;
    long long tot;
    const long long e = block_excl_scan(x, wt, tot);
    if (i < n) v[i] = e;
    if (threadIdx.x == 0) block_tot[blockIdx.x] = tot;
}

__global__ void k_scan_top(int64_t* block_tot, int nb) {
    pdl_trigger();
    pdl_wait();
    __shared__ long long wt[32];
    __shared__ long long carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int base = 0; base < nb; base += SCAN_T) {
        const int i = base + threadIdx.x;
        const long long x = i < nb ? block_tot[i] : 0;
        long long tot;
        const long long e = block_excl_scan(x, wt, tot);
        const long long c = carry;
        if (i < nb) block_tot[i] = c + e;
        __syncthreads();
        if (threadIdx.x == 0) carry = c + tot;
        __syncthreads();
    }
}

__global__ void k_scan_add(int64_t* v, int64_t n, const int64_t* block_tot) {
    pdl_trigger();
    pdl_wait();
    const int64_t i = (int64_t)blockIdx.x * SCAN_T + threadIdx.x;
    if (i < n) v[i] += block_tot[blockIdx.x];
}

// task = {move, tour, order, tag}: tag >= 0 or -1: order moves (tag = order
// removed, order = order added, -1 = none); tag -2 / -3: SKU swap, `order` is
// the order of s1's / s2's list the task came from.  One move per lane, on
// `unit` lanes of a warp (few where there are few moves); a SKU list longer
// than MVF_SERIAL orders (a popular SKU can sit in hundreds) is written by the
// whole warp, 32 tasks a step, at the same places.
constexpr int MVF_SERIAL = 8;

__global__ void k_mv_fill(MoveArgs M, int unit) {
    pdl_trigger();
    pdl_wait();
    const EvalArgs& a = M.a;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t base = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * unit; base < M.n_moves;
         base += warps * unit) {
        const int m = (int)(base + lane);
        int lb[2] = {0, 0}, ln[2] = {0, 0}, lk[2] = {0, 0};   // a long list per side: begin, length, first task
        int64_t row = 0, t0 = 0;
        if (lane < unit && m < M.n_moves && M.mstatus[m] == 0) {
            const int4 mv = M.moves[m];
            row = (int64_t)mv.w * a.n_orders;
            t0 = M.task_off[m];
            int4* out = M.tasks + t0;
            if (mv.x == 0) {
                const int ta = M.order_tour[row + mv.y], tb = M.order_tour[row + mv.z];
                out[0] = make_int4(m, ta, mv.z, mv.y);
                out[1] = make_int4(m, tb, mv.y, mv.z);
            } else if (mv.x == 1) {
                const int ta = M.order_tour[row + mv.y], tb = a.plan_tour_off[mv.w] + mv.z;
                out[0] = make_int4(m, ta, -1, mv.y);
                out[1] = make_int4(m, tb, mv.y, -1);
            } else {
                int k = 0;
                for (int side = 0; side < (mv.x == 2 ? 2 : 1); ++side) {
                    const int sk = side ? mv.z : mv.y;
                    const int b = M.sku_off[sk], e = b + M.sku_cur[sk];
                    if (e - b > MVF_SERIAL) {
                        lb[side] = b;
                        ln[side] = e - b;
                        lk[side] = k;
                        k += e - b;
                        continue;
                    }
                    for (int i = b; i < e; ++i) {
                        const int o = M.sku_orders[i];
                        out[k++] = make_int4(m, M.order_tour[row + o], o, side ? -3 : -2);
                    }
                }
            }
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            unsigned longs = __ballot_sync(0xffffffffu, ln[side] > 0);
            while (longs) {
                const int src = __ffs(longs) - 1;
                longs &= longs - 1;
                const int b = __shfl_sync(0xffffffffu, lb[side], src), n = __shfl_sync(0xffffffffu, ln[side], src);
                const int k0 = __shfl_sync(0xffffffffu, lk[side], src), mm = __shfl_sync(0xffffffffu, m, src);
                const int64_t r = __shfl_sync(0xffffffffu, row, src);
                int4* out = M.tasks + __shfl_sync(0xffffffffu, t0, src) + k0;
                for (int i0 = lane; i0 < n; i0 += 128) {   // four entries a lane in flight
                    int o[4], t[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) o[u] = i0 + 32 * u < n ? M.sku_orders[b + i0 + 32 * u] : 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u) t[u] = i0 + 32 * u < n ? M.order_tour[r + o[u]] : 0;
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (i0 + 32 * u < n) out[i0 + 32 * u] = make_int4(mm, t[u], o[u], side ? -3 : -2);
                }
            }
        }
    }
}

// Location of SKU s under the move's slotting: the swapped pair for a SKU
// swap, the target location for the relocated SKU.
__device__ __forceinline__ int task_loc(const int32_t* map, int s, const int4 mv) {
    if (mv.x == 2) s = s == mv.y ? mv.z : (s == mv.z ? mv.y : s);
    else if (mv.x == 3 && s == mv.y) return mv.z;
    return map[s];
}

// the line's SKU is one the SKU move changes
__device__ __forceinline__ bool sku_hit(int s, const int4 mv) { return s == mv.y || (mv.x == 2 && s == mv.z); }

// The changed tour of a lane's task: its sequence range, the order added and a
// bound on its lines; ok is cleared when its orders are malformed.
__device__ __forceinline__ void task_tour(const MoveArgs& M, bool has, RowTour& w, bool& ok) {
    const EvalArgs& a = M.a;
    w.q0 = w.q1 = w.ub = 0;
    w.add = has && w.mv.x < 2 && w.tk.z >= 0 ? w.tk.z : -1;
    if (!has) return;
    w.q0 = a.tour_off[w.tk.y];
    w.q1 = a.tour_off[w.tk.y + 1];
    int lb, le;
    const int cur = M.tour_lines[w.tk.y], more = w.add >= 0 ? order_lines_checked(a, w.add, lb, le) : 0;
    ok = cur >= 0 && more >= 0;
    w.ub = ok ? cur + more : 0;
}

// Tasks of at most ROW_MAXN lines: up to 32 a warp, one a lane, read, sorted
// (run_rows) and costed together.
__global__ void __launch_bounds__(ROW_THREADS, 5) k_mv_eval(MoveArgs M, int unit) {
    extern __shared__ __align__(16) uint32_t mv_rows[];
    __shared__ RowList s_rl[ROW_WARPS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t* rows = mv_rows + wid * ROW_WORDS;
    const EvalArgs& a = M.a;
    const DPConst c = dp_const(a.g);
    const int64_t stride = (int64_t)gridDim.x * ROW_WARPS * unit;
    for (int64_t u0 = ((int64_t)blockIdx.x * ROW_WARPS + wid) * unit; u0 < M.n_tasks; u0 += stride) {
        const int64_t i = u0 + lane;
        const bool active = lane < unit && i < M.n_tasks;
        int4 tk = make_int4(-1, -1, -1, -1), mv = make_int4(0, 0, 0, 0);
        if (active) {
            tk = M.tasks[i];
            mv = M.moves[tk.x];
        }
        // an order of the SKU lists outside the plan: nothing to cost
        const bool has = active && tk.y >= 0 && tk.y < a.n_tours;
        bool ok = active;
        RowTour w;
        w.tk = tk;
        w.mv = mv;
        task_tour(M, has, w, ok);
        const bool lng = has && ok && w.ub > ROW_MAXN;
        if (lng) {
            const int slot = atomicAdd(M.long_count, 1);
            if (slot < M.long_cap) M.long_list[slot] = (int32_t)i;
            else { flag(a.status, WH_STATUS_LONG_OVERFLOW); M.mstatus[tk.x] = 3; }
        }
        bool run = false;   // the task's cost counts: cs, cr
        int n = 0, cs = 0, cr = 0;
        run_rows(a, rows, s_rl[wid], w, __ballot_sync(0xffffffffu, has && ok && !lng), lane,
                 [&](bool mine, bool primary, int base, int rn, bool bad) {
                     if (!mine) return;
                     const uint32_t* row = rows + base;
                     n = rn;
                     if (primary) row_costs(a.g, c, row, n, true, cs, cr);
                     if (bad)
                         for (int p = 0; p < n; ++p) ok &= row[p] < KEY_BAD_SKU;
                     run = primary && ok;
                 });
        if (active && !ok) {
            flag(a.status, WH_STATUS_BAD_ORDER);
            M.mstatus[tk.x] = 3;
        }
        if (M.stats) {   // changed tours walked and their lines (the moves' roofline); k_mv_long adds its own
            const bool w = active && ok && !lng;
            const unsigned walked = __reduce_add_sync(0xffffffffu, w ? 1u : 0u);
            const unsigned lines = __reduce_add_sync(0xffffffffu, w ? (unsigned)n : 0u);
            if (lane == 0 && walked) {
                atomicAdd(M.stats, (unsigned long long)walked);
                atomicAdd(M.stats + 1, (unsigned long long)lines);
            }
        }
        long long ds = 0, dr = 0;
        if (run) {
            ds = (long long)cs - M.tour_s_old[tk.y];
            dr = (long long)cr - M.tour_rr_old[tk.y];
        }
        if (active && !lng)   // k_mv_long writes the long ones
            M.task_cost[i] = run ? make_int2(cs, cr) : make_int2(-1, -1);
        const int key = active ? tk.x : -1;
        const long long ss = segmented_sum(ds, key, lane);
        const long long sr = segmented_sum(dr, key, lane);
        const int prev_key = __shfl_up_sync(0xffffffffu, key, 1);
        if (active && (lane == 0 || prev_key != key) && (ss || sr)) {
            atomicAdd(reinterpret_cast<unsigned long long*>(&M.delta[2 * tk.x]), (unsigned long long)ss);
            atomicAdd(reinterpret_cast<unsigned long long*>(&M.delta[2 * tk.x + 1]), (unsigned long long)sr);
        }
    }
}

// The changed tour of task `tk` by one warp: lane j takes the changed tour's orders
// j, j + 32, ... (the added order last), stores their line indices at
// positions given by a warp prefix sum of the order line counts and, for a SKU
// move, looks for the moved SKUs on them; then, if the task is the counted one
// of its tour, the lanes turn positions x, x + 32, ... into keys.  (A popular SKU is
// on many of a tour's orders, and all but one of its tasks there end here.  With a
// lane looking through the tour's orders for every line found, 16,384 moves on tours
// of 200 lines took 1,057 us a call; now 400.)
// Only the first `cap` positions are stored.  Returns ok and sets n and
// primary (all warp-uniform).
__device__ __forceinline__ bool walk_task_warp(const MoveArgs& M, const int4 tk, const int4 mv, uint32_t* kb,
                                               int cap, int lane, int& n_out, bool& primary) {
    const EvalArgs& a = M.a;
    const bool swap = mv.x >= 2;   // SKU moves: swap or relocation
    const int32_t* map = a.slot_map + (int64_t)mv.w * a.slot_stride;
    const int q0 = a.tour_off[tk.y], q1 = a.tour_off[tk.y + 1];
    const int add = (!swap && tk.z >= 0) ? tk.z : -1;
    const int rem = (!swap && tk.w >= 0) ? tk.w : -1;
    bool bad = !(q0 >= 0 && q1 >= q0 && (int64_t)q1 <= a.n_seq);
    const int q_end = bad ? q0 : (add >= 0 ? q1 + 1 : q1);
    int hit_min = 0x7fffffff, n = 0;
    bool own_has_s1 = false;
    // the lines' indices at their positions in the changed tour (lanes over
    // orders)
    for (int qb = q0; qb < q_end; qb += 32) {
        const int q = qb + lane;
        int o = -1, lb = 0, le = 0;
        if (!bad && q < q_end) {
            o = q < q1 ? a.order_seq[q] : add;
            if (q < q1 && o == rem) o = -1;
            else if (order_lines_checked(a, o, lb, le) < 0) { bad = true; lb = le = 0; }
        }
        const int cnt = le - lb;
        const int incl = warp_inclusive_scan(cnt);
        int pos = n + incl - cnt;
        if (swap) {
            for (int l0 = lb; l0 < le; l0 += 4) {
                int sk[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) sk[u] = l0 + u < le ? a.line_sku[l0 + u] : -1;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (sk[u] < 0 || !sku_hit(sk[u], mv)) continue;
                    hit_min = min(hit_min, o);
                    own_has_s1 |= o == tk.z && sk[u] == mv.y;
                }
            }
        }
        for (int l = lb; l < le; ++l, ++pos)
            if (pos < cap) kb[pos] = (uint32_t)l;
        n += __shfl_sync(0xffffffffu, incl, 31);
    }
    bad = __any_sync(0xffffffffu, bad);
    hit_min = __reduce_min_sync(0xffffffffu, hit_min);
    own_has_s1 = __any_sync(0xffffffffu, own_has_s1);
    primary = !swap || (hit_min == tk.z && (tk.w == -2 || !own_has_s1));
    n_out = n;
    if (bad || !primary) return !bad;
    __syncwarp();
    // keys: lanes over positions, four a lane with their SKU and slot loads in
    // flight together
    const int nn = min(n, cap);
    for (int x0 = 0; x0 < nn; x0 += 128) {
        int l[4], sk[4], loc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int x = x0 + 32 * u + lane;
            l[u] = x < nn ? (int)kb[x] : -1;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) sk[u] = l[u] >= 0 ? a.line_sku[l[u]] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            loc[u] = (l[u] >= 0 && (unsigned)sk[u] < (unsigned)a.n_sku) ? task_loc(map, sk[u], mv) : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (l[u] < 0) continue;
            if ((unsigned)sk[u] >= (unsigned)a.n_sku || (unsigned)loc[u] >= (unsigned)a.g.n_loc) {
                bad = true;
                continue;
            }
            kb[x0 + 32 * u + lane] = loc_key(a.g, loc[u]);
        }
    }
    return !__any_sync(0xffffffffu, bad);
}

// Tasks of more than ROW_MAXN lines: one warp per task walks the changed tour
// (walk_task_warp), sorts its keys in shared memory and extracts the per-aisle
// records in parallel (a ballot numbers the aisle runs) into a column of the
// warp's own matrix in global memory; once the matrix's long_cols columns are
// full, or no task is left, every lane runs the DP of one of them.  A task
// with more than MVL_RMAX records runs its scan and DP on one lane right away.
// With one matrix for the first 65,536 tasks and the others' DPs on one lane of
// their warp, 262,144 moves on tours of 200 lines in 40 aisles took 5.9 ms; now
// 4.26 (in 500 aisles, where few tours' records fit, 65,536 moves 1.40 and 1.52 ms).
__device__ __forceinline__ void mv_long_commit(const MoveArgs& M, int64_t i, int cs, int cr) {
    const int4 tk = M.tasks[i];
    M.task_cost[i] = make_int2(cs, cr);
    const long long ds = (long long)cs - M.tour_s_old[tk.y];
    const long long dr = (long long)cr - M.tour_rr_old[tk.y];
    atomicAdd(reinterpret_cast<unsigned long long*>(&M.delta[2 * tk.x]), (unsigned long long)ds);
    atomicAdd(reinterpret_cast<unsigned long long*>(&M.delta[2 * tk.x + 1]), (unsigned long long)dr);
}

__global__ void __launch_bounds__(LONG_WARPS * 32, 6) k_mv_long(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    __shared__ uint32_t buf[LONG_WARPS][LONG_MAXL];
    // the matrix's columns: task, records, largest key
    __shared__ int s_task[LONG_WARPS][32], s_m[LONG_WARPS][32];
    __shared__ uint32_t s_last[LONG_WARPS][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int count = min(*M.long_count, M.long_cap);
    uint32_t* kb = buf[warp];
    const EvalArgs& a = M.a;
    const int gw = blockIdx.x * LONG_WARPS + warp, cols = M.long_cols;
    uint2* rec = M.long_rec + (int64_t)gw * MVL_RMAX * cols;   // record r of column j at [r * cols + j]
    int have = 0;   // columns in use
    auto run_dps = [&] {
        __syncwarp();
        if (lane < have) {
            const uint32_t kl = s_last[warp][lane];
            const int m = s_m[warp][lane];
            mv_long_commit(M, s_task[warp][lane], sshape_cost(a.g, m, (int)(kl >> 16), (int)(kl & 0xFFFFu)),
                           rr_records32_mem(a.g, rec + lane, cols, m));
        }
        have = 0;
        __syncwarp();
    };
    for (int w = gw; w < count; w += gridDim.x * LONG_WARPS) {
        const int i = M.long_list[w];
        const int4 tk = M.tasks[i];
        const int4 mv = M.moves[tk.x];
        int n = 0;
        bool primary = false;
        const bool ok = walk_task_warp(M, tk, mv, kb, LONG_MAXL, lane, n, primary);
        __syncwarp();
        if (lane == 0 && ok && M.stats) {
            atomicAdd(M.stats, 1ull);
            atomicAdd(M.stats + 1, (unsigned long long)n);
        }
        if (!ok || n > LONG_MAXL || !primary) {
            if (lane == 0) {
                if (!ok || n > LONG_MAXL) {
                    flag(a.status, n > LONG_MAXL ? WH_STATUS_TOUR_TOO_LONG : WH_STATUS_BAD_ORDER);
                    M.mstatus[tk.x] = 3;
                }
                M.task_cost[i] = make_int2(-1, -1);
            }
            __syncwarp();
            continue;
        }
        warp_sort_buffer(kb, n, lane);
        // per-aisle records: run r of the sorted keys -> row r of the column
        int m = 0;
        for (int x0 = 0; x0 < n; x0 += 32) {
            const int x = x0 + lane;
            const bool in = x < n;
            const uint32_t key = in ? kb[x] : 0u;
            const int ai = (int)(key >> 16);
            const bool first = in && (x == 0 || (int)(kb[x - 1] >> 16) != ai);
            const bool last = in && (x == n - 1 || (int)(kb[x + 1] >> 16) != ai);
            const unsigned fm = __ballot_sync(0xffffffffu, first);
            const int r = m + __popc(fm & ((2u << lane) - 1u)) - 1;
            if (last && r < MVL_RMAX) {
                const int hi = (int)(key & 0xFFFFu);
                int lo = hi, gi = 0;
                for (int y = x; y > 0 && (int)(kb[y - 1] >> 16) == ai; --y) {
                    const int kp = (int)(kb[y - 1] & 0xFFFFu);
                    gi = max(gi, lo - kp);
                    lo = kp;
                }
                rec[r * cols + have] =
                    make_uint2(((uint32_t)ai << 16) | (uint32_t)lo, ((uint32_t)hi << 16) | (uint32_t)gi);
            }
            m += __popc(fm);
        }
        if (lane == 0) {
            const uint32_t kl = n > 0 ? kb[n - 1] : 0u;   // rightmost aisle, its deepest slot
            if (m <= MVL_RMAX) {
                s_task[warp][have] = i;
                s_m[warp][have] = m;
                s_last[warp][have] = kl;
            } else {
                // more aisles than the matrix keeps: scan and DP here
                DP5 v;
                dp_init(v);
                int pa = 0, lo = 0, prev = 0, gi = 0;
                for (int x = 0; x < n; ++x) {
                    const uint32_t key = kb[x];
                    const int ai = (int)(key >> 16), k = (int)(key & 0xFFFFu);
                    const bool first = (x == 0) || ((int)(kb[x - 1] >> 16) != ai);
                    const bool last = (x == n - 1) || ((int)(kb[x + 1] >> 16) != ai);
                    gi = first ? 0 : max(gi, k - prev);
                    lo = first ? k : lo;
                    prev = k;
                    if (last) {
                        dp_aisle(v, a.g, ai - pa, lo, k, gi);
                        pa = ai;
                    }
                }
                mv_long_commit(M, i, sshape_cost(a.g, m, (int)(kl >> 16), (int)(kl & 0xFFFFu)), dp_final(v));
            }
        }
        if (m <= MVL_RMAX && ++have == cols) run_dps();
        __syncwarp();
    }
    run_dps();
}

// moves that ended with a non-zero status report zero deltas
__global__ void k_mv_finish(MoveArgs M) {
    pdl_trigger();
    pdl_wait();
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < M.n_moves; m += gridDim.x * blockDim.x) {
        if (M.mstatus[m] != 0) {
            M.delta[2 * m] = 0;
            M.delta[2 * m + 1] = 0;
        }
    }
}

int grid_of(int64_t n, int threads, int cap = 8192) {
    int64_t g = (n + threads - 1) / threads;
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

// occupancy bits of every plan's slotting (relocation moves): bit l of plan
// p set when a SKU of p sits at location l (ids outside the layout skipped)
__global__ void k_occupancy(const int32_t* slot_map, int64_t stride, int32_t n_plans, int32_t n_sku, int32_t n_loc,
                            uint32_t* used) {
    const int64_t total = (int64_t)n_plans * n_sku;
    const int words = (n_loc + 31) >> 5;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = i / n_sku, s = i - p * n_sku;
        const int loc = slot_map[p * stride + s];
        if ((unsigned)loc < (unsigned)n_loc) atomicOr(&used[p * words + (loc >> 5)], 1u << (loc & 31));
    }
}

}  // namespace

// The moves' short kernels, a dozen in a row: each waits for the one before it
// as its first statement (pdl_wait) and is launched beside its tail.  The two
// large ones (k_mv_eval, k_task_features) are launched the ordinary way and
// trigger nothing early: beside another kernel's blocks they start with that
// kernel's split of L1 and shared memory, and later blocks would take theirs
// (the plain step 635 us instead of 574).
cudaError_t launch_moves_prepare(const MoveArgs& M, int num_sms, cudaStream_t s, bool reuse_index) {
    const EvalArgs& a = M.a;
    if (reuse_index) {
        // the order -> tour table, the tours' line counts and the SKU ->
        // orders index of the same plans are in place: only the moves' checks,
        // task counts and their scan
        launch_dependent(k_mv_count, grid_of(M.n_moves, 256), 256, 0, s, M);
        const int64_t n = (int64_t)M.n_moves + 1;
        const int nb = (int)((n + SCAN_T - 1) / SCAN_T);
        launch_dependent(k_scan_blocks, nb, SCAN_T, 0, s, M.task_off, n, M.scan_aux);
        launch_dependent(k_scan_top, 1, SCAN_T, 0, s, M.scan_aux, nb);
        launch_dependent(k_scan_add, nb, SCAN_T, 0, s, M.task_off, n, M.scan_aux);
        return cudaGetLastError();
    }
    const bool per_plan = a.n_orders <= MVT_MAX_ORDERS;
    if (!per_plan &&
        cudaMemsetAsync(M.order_tour, 0xFF, sizeof(int32_t) * (size_t)a.n_plans * (size_t)a.n_orders, s) != cudaSuccess)
        return cudaGetLastError();
    if (cudaMemsetAsync(M.sku_cur, 0, sizeof(int32_t) * ((size_t)a.n_sku + 1), s) != cudaSuccess)
        return cudaGetLastError();
    if (per_plan) {
        // tours outside every plan's range (malformed plan offsets, flagged)
        // keep the "bad tour" line count
        if (a.n_tours > 0 && cudaMemsetAsync(M.tour_lines, 0xFF, sizeof(int32_t) * (size_t)a.n_tours, s) != cudaSuccess)
            return cudaGetLastError();
        const int grid = a.n_plans < num_sms * 8 ? a.n_plans : num_sms * 8;
        if (grid > 0) k_mv_tours_plan<<<grid, MVT_THREADS, sizeof(int32_t) * (size_t)a.n_orders, s>>>(M);
    } else if (a.n_tours > 0) {
        k_mv_tours<<<grid_of(a.n_tours, 256), 256, 0, s>>>(M);
    }
    if (a.n_lines > 0) launch_dependent(k_mv_sku_count, grid_of(a.n_lines, 256), 256, 0, s, M);
    if (a.n_sku > 0) launch_dependent(k_mv_sku_alloc, (a.n_sku + SKU_ALLOC_T - 1) / SKU_ALLOC_T, SKU_ALLOC_T, 0, s, M);
    if (a.n_orders > 0) launch_dependent(k_mv_sku_fill, grid_of(a.n_orders, 256), 256, 0, s, M);
    launch_dependent(k_mv_count, grid_of(M.n_moves, 256), 256, 0, s, M);
    // exclusive scan of n_moves + 1 task counts
    const int64_t n = (int64_t)M.n_moves + 1;
    const int nb = (int)((n + SCAN_T - 1) / SCAN_T);
    launch_dependent(k_scan_blocks, nb, SCAN_T, 0, s, M.task_off, n, M.scan_aux);
    launch_dependent(k_scan_top, 1, SCAN_T, 0, s, M.scan_aux, nb);
    launch_dependent(k_scan_add, nb, SCAN_T, 0, s, M.task_off, n, M.scan_aux);
    return cudaGetLastError();
}

// 32 warps an SM: enough to hide the lists' gathers, and up to 32 moves a
// warp beyond that (16,384 kept moves 51 us with 32 moves a warp throughout)
cudaError_t launch_moves_fill(const MoveArgs& M, int num_sms, cudaStream_t s) {
    if (M.n_moves <= 0) return cudaSuccess;
    const int64_t warps = (int64_t)num_sms * 32, u = (M.n_moves + warps - 1) / warps;
    const int unit = u > 32 ? 32 : (int)u;
    launch_dependent(k_mv_fill, grid_of((M.n_moves + unit - 1) / unit * 32, 256), 256, 0, s, M, unit);
    return cudaGetLastError();
}

cudaError_t launch_moves_eval(const MoveArgs& M, int num_sms, cudaStream_t s) {
    const cudaError_t f = launch_moves_fill(M, num_sms, s);
    if (f != cudaSuccess) return f;
    if (M.n_tasks > 0) {
        int per_sm = 0;
        cudaError_t e = rows_per_sm(k_mv_eval, &per_sm);
        if (e != cudaSuccess) return e;
        const int64_t grid = (int64_t)per_sm * num_sms;
        const int unit = row_unit(M.n_tasks, grid * ROW_WARPS);
        const int64_t want = (M.n_tasks + (int64_t)unit * ROW_WARPS - 1) / (unit * ROW_WARPS);
        k_mv_eval<<<(int)(grid < want ? grid : want), ROW_THREADS, ROW_SMEM, s>>>(M, unit);
    }
    return cudaGetLastError();
}

// Every CTA of k_mv_long that fits the chip, and as many columns a warp as it
// can have tasks (at most a lane's each).
cudaError_t moves_long_shape(int64_t n_tasks, int num_sms, int* grid, int* cols, size_t* bytes) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_mv_long, LONG_WARPS * 32, 0);
    if (e != cudaSuccess) return e;
    *grid = num_sms * (per_sm > 0 ? per_sm : 1);
    const int64_t warps = (int64_t)*grid * LONG_WARPS, most = (n_tasks + warps - 1) / warps;
    *cols = most < 32 ? (int)most : 32;
    *bytes = sizeof(uint2) * (size_t)MVL_RMAX * (size_t)*cols * (size_t)warps;
    return cudaSuccess;
}

cudaError_t launch_moves_long(const MoveArgs& M, int grid, cudaStream_t s) {
    if (M.n_tasks > 0) launch_dependent(k_mv_long, grid, LONG_WARPS * 32, 0, s, M);
    if (M.n_moves > 0) launch_dependent(k_mv_finish, grid_of(M.n_moves, 256), 256, 0, s, M);
    return cudaGetLastError();
}

}  // namespace wh

// ---------------------------------------------------------- local search
namespace wh {
namespace {

// One CTA per plan: the move with the most negative optimal-cost delta among
// the plan's moves of status 0 (ties: lowest index) is applied in place.
__global__ void k_ls_apply(LsArgs L) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ int32_t seg[];
    __shared__ long long s_best;
    __shared__ int s_pos[2];
    const EvalArgs& a = L.a;
    const int tid = threadIdx.x, T = blockDim.x;
    for (int p = blockIdx.x; p < a.n_plans; p += gridDim.x) {
        if (tid < 32) {
            long long best = 0x7fffffffffffffffll;
            for (int k = tid; k < L.moves_per_plan; k += 32) {
                const int64_t m = (int64_t)p * L.moves_per_plan + k;
                const long long d = L.delta[2 * m + 1];
                if (L.status[m] == 0 && d < 0 && L.moves[m].w == p) best = min(best, d * 256 + k);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, o));
            if (tid == 0) {
                s_best = best;
                s_pos[0] = s_pos[1] = -1;
            }
        }
        __syncthreads();
        const long long best = s_best;
        const int k = best == 0x7fffffffffffffffll ? -1 : (int)(((best % 256) + 256) % 256);
        if (tid == 0) L.applied[p] = k;
        if (k >= 0) {
            const int4 mv = L.moves[(int64_t)p * L.moves_per_plan + k];
            const int t0 = a.plan_tour_off[p], t1 = a.plan_tour_off[p + 1];
            const int s0 = a.tour_off[t0], s1 = a.tour_off[t1];
            int32_t* order_seq = const_cast<int32_t*>(a.order_seq);
            int32_t* tour_off = const_cast<int32_t*>(a.tour_off);
            if (mv.x == 0 || mv.x == 1) {
                for (int q = s0 + tid; q < s1; q += T) {
                    const int o = order_seq[q];
                    if (o == mv.y) s_pos[0] = q;
                    if (mv.x == 0 && o == mv.z) s_pos[1] = q;
                }
                __syncthreads();
                const int ia = s_pos[0];
                if (mv.x == 0) {
                    if (tid == 0 && ia >= 0 && s_pos[1] >= 0) {
                        order_seq[ia] = mv.z;
                        order_seq[s_pos[1]] = mv.y;
                    }
                } else if (ia >= 0) {
                    // tour holding position ia: largest t with tour_off[t] <= ia
                    int lo = t0, hi = t1 - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (tour_off[mid] <= ia) lo = mid; else hi = mid - 1;
                    }
                    const int ta = lo, tb = t0 + mv.z;
                    const int end = tour_off[tb + 1];
                    const int r0 = tb > ta ? ia : end, r1 = tb > ta ? end : ia + 1;   // range that moves
                    if (r1 - r0 <= L.seg_cap) {
                        for (int q = r0 + tid; q < r1; q += T) seg[q - r0] = order_seq[q];
                        __syncthreads();
                        if (tb > ta) {
                            for (int q = r0 + tid; q < r1 - 1; q += T) order_seq[q] = seg[q - r0 + 1];
                            if (tid == 0) order_seq[r1 - 1] = mv.y;
                            for (int t = ta + 1 + tid; t <= tb; t += T) tour_off[t] -= 1;
                        } else {
                            for (int q = r0 + 1 + tid; q < r1; q += T) order_seq[q] = seg[q - r0 - 1];
                            if (tid == 0) order_seq[r0] = mv.y;
                            for (int t = tb + 1 + tid; t <= ta; t += T) tour_off[t] += 1;
                        }
                    } else if (tid == 0) {
                        flag(a.status, WH_STATUS_BAD_OFFSET);
                        L.applied[p] = -1;
                    }
                }
            } else if (mv.x == 2 && tid == 0) {
                int32_t* smap = const_cast<int32_t*>(a.slot_map) + (int64_t)p * a.slot_stride;
                const int32_t x = smap[mv.y];
                smap[mv.y] = smap[mv.z];
                smap[mv.z] = x;
            } else if (mv.x == 3 && tid == 0) {
                // relocation: the SKU's entry and the plan's occupancy bits
                int32_t* smap = const_cast<int32_t*>(a.slot_map) + (int64_t)p * a.slot_stride;
                const int32_t old = smap[mv.y];
                smap[mv.y] = mv.z;
                if (a.loc_used) {
                    uint32_t* used = a.loc_used + (int64_t)p * ((a.g.n_loc + 31) >> 5);
                    if ((unsigned)old < (unsigned)a.g.n_loc) used[old >> 5] &= ~(1u << (old & 31));
                    used[mv.z >> 5] |= 1u << (mv.z & 31);
                }
            }
            // costs: the changed tours take their tasks' new costs, the plan its delta
            if (L.task_cost && L.applied[p] == k) {
                const int64_t m = (int64_t)p * L.moves_per_plan + k;
                for (int64_t i = L.task_off[m] + tid; i < L.task_off[m + 1]; i += T) {
                    const int2 c = L.task_cost[i];
                    if (c.x < 0) continue;
                    const int t = L.tasks[i].y;
                    if (L.tour_s) L.tour_s[t] = c.x;
                    if (L.tour_rr) L.tour_rr[t] = c.y;
                    if (L.tour_changed) L.tour_changed[t] = 1;
                }
                if (tid == 0) {
                    if (L.plan_s) L.plan_s[p] += L.delta[2 * m];
                    if (L.plan_rr) L.plan_rr[p] += L.delta[2 * m + 1];
                }
            }
        }
        __syncthreads();
    }
}

// Features of every task's changed tour, one task per warp (WarpFeat): its
// orders by the lanes, the added one last; the SKU-swap rule that picks the
// counted task of a tour reduces over the lanes.  Marks in task_cost which
// tasks count (rows of non-counted tasks are written too and ignored by the
// selection).
constexpr int TF_THREADS = 256;

// One changed tour per warp.  Its orders are taken 32 at a time (one per
// lane: id, line range); then the lanes walk the round's lines flat, 32 at a
// time, each lane finding its line's order from the orders' start offsets (a
// bitmask of order starts within the 32-line window), so all lanes gather
// slot-map entries together whatever the orders' sizes.
__global__ void __launch_bounds__(TF_THREADS) k_task_features(MoveArgs M, FeatConst c, uint4* X) {
    __shared__ WarpFeat ws[TF_THREADS / 32];
    __shared__ int s_lb[TF_THREADS / 32][32], s_off[TF_THREADS / 32][33], s_o[TF_THREADS / 32][32],
        s_rank[TF_THREADS / 32][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    WarpFeat& w = ws[wid];
    int* lbs = s_lb[wid];
    int* offs = s_off[wid];
    int* ords = s_o[wid];
    int* rank_to_k = s_rank[wid];
    wf_init(w, lane);
    const EvalArgs& a = M.a;
    const unsigned lt_mask = (1u << lane) - 1u;
    const int64_t n_warps = (int64_t)gridDim.x * (TF_THREADS / 32);
    for (int64_t i = (int64_t)blockIdx.x * (TF_THREADS / 32) + wid; i < M.n_tasks; i += n_warps) {
        const int4 tk = M.tasks[i];
        bool ok = false, primary = false, over = false;
        uint32_t n_lines = 0;
        if (tk.y >= 0 && tk.y < a.n_tours) {
            const int4 mv = M.moves[tk.x];
            const bool swap = mv.x >= 2;   // SKU moves: swap or relocation
            const int32_t* map = a.slot_map + (int64_t)mv.w * a.slot_stride;
            const int q0 = a.tour_off[tk.y], q1 = a.tour_off[tk.y + 1];
            const int add = (!swap && tk.z >= 0) ? tk.z : -1;
            const int rem = (!swap && tk.w >= 0) ? tk.w : -1;
            bool bad = !(q0 >= 0 && q1 >= q0 && (int64_t)q1 <= a.n_seq);
            int hit_min = 0x7fffffff;
            bool own_has_s1 = false;
            const int q_end = bad ? q0 : (add >= 0 ? q1 + 1 : q1);
            for (int qb = q0; qb < q_end; qb += 32) {
                // this round's orders, one per lane (none: count 0)
                const int q = qb + lane;
                int o = -1, lb = 0, cnt = 0;
                if (q < q_end) {
                    o = q < q1 ? a.order_seq[q] : add;
                    if (q < q1 && o == rem) {
                        o = -1;
                    } else {
                        int le;
                        const int cc = order_lines_checked(a, o, lb, le);
                        if (cc < 0) bad = true;
                        else cnt = cc;
                    }
                }
                const int incl = warp_inclusive_scan(cnt);
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                const unsigned nonempty = __ballot_sync(0xffffffffu, cnt > 0);
                lbs[lane] = lb;
                offs[lane] = incl - cnt;
                ords[lane] = o;
                if (cnt > 0) rank_to_k[__popc(nonempty & lt_mask)] = lane;
                __syncwarp();
                // the round's lines, 32 at a time: line p belongs to the
                // nonempty order whose start is the last one <= p
                int before = 0;   // nonempty orders starting before this window
                for (int p0 = 0; p0 < total; p0 += 32) {
                    const int start = offs[lane];
                    const bool head = cnt > 0 && start >= p0 && start < p0 + 32;
                    const unsigned hm = __reduce_or_sync(0xffffffffu, head ? 1u << (start - p0) : 0u);
                    const int p = p0 + lane;
                    if (p < total && !bad) {
                        const int r = before + __popc(hm & (lt_mask | (1u << lane))) - 1;
                        const int k = rank_to_k[r];
                        const int ok_ = ords[k];
                        const int l = lbs[k] + (p - offs[k]);
                        const int sk = a.line_sku[l];
                        if ((unsigned)sk >= (unsigned)a.n_sku) {
                            bad = true;
                        } else {
                            if (swap && sku_hit(sk, mv)) {
                                hit_min = min(hit_min, ok_);
                                if (ok_ == tk.z && sk == mv.y) own_has_s1 = true;
                            }
                            const int loc = task_loc(map, sk, mv);
                            if ((unsigned)loc >= (unsigned)a.g.n_loc) bad = true;
                            else {
                                over |= !wf_insert(w, loc_key(a.g, loc));
                                ++n_lines;
                            }
                        }
                    }
                    before += __popc(hm);
                }
                __syncwarp();
            }
            ok = !__any_sync(0xffffffffu, bad);
            hit_min = __reduce_min_sync(0xffffffffu, hit_min);
            own_has_s1 = __any_sync(0xffffffffu, own_has_s1);
            primary = !swap || (hit_min == tk.z && (tk.w == -2 || !own_has_s1));
        }
        over = __any_sync(0xffffffffu, over);
        n_lines = __reduce_add_sync(0xffffffffu, n_lines);
        if (lane == 0) M.task_cost[i] = (ok && primary && !over) ? make_int2(0, 0) : make_int2(-1, -1);
        wf_finish(w, c, lane, n_lines, X + i * 24);
    }
}

// Predicted delta of every move (sum over its counted tasks, in order), then
// per plan the `keep` moves with the lowest predicted delta (ties: lowest
// index); unfilled places get an invalid move that scores status 3.
constexpr int SCORE_SERIAL = 12;

__global__ void k_screen_score(ScreenArgs S) {
    pdl_trigger();
    pdl_wait();
    const MoveArgs& M = S.M;
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // one move per lane; a move of more than SCORE_SERIAL tasks is scored by the
    // whole warp: lanes load 32 tasks' terms at once, and every lane adds
    // them up in task order, so the sum is the serial one
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < M.n_moves; base += stride) {
        const int64_t m = base + lane;
        float sc = 3.0e38f;
        int64_t i0 = 0, i1 = 0;
        if (m < M.n_moves && M.mstatus[m] == 0) {
            sc = 0.0f;
            i0 = M.task_off[m];
            i1 = M.task_off[m + 1];
        }
        const bool lng = i1 - i0 > SCORE_SERIAL;
        if (!lng)
            for (int64_t i = i0; i < i1; i += 4) {
                // counted task: an order move, or the first task of its tour
                // for a SKU swap; four tasks' loads in flight
                int t[4];
                float yt[4], yo[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    t[u] = i + u < i1 ? M.tasks[i + u].y : -1;
                    if (i + u < i1 && M.task_cost[i + u].x < 0) t[u] = -1;
                    yt[u] = i + u < i1 ? S.y_task[i + u] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) yo[u] = t[u] >= 0 ? S.y_tour[t[u]] : 0.0f;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (t[u] >= 0) sc += yt[u] - yo[u];
            }
        unsigned longs = __ballot_sync(0xffffffffu, lng);
        while (longs) {
            const int src = __ffs(longs) - 1;
            longs &= longs - 1;
            const int64_t b = __shfl_sync(0xffffffffu, i0, src), e = __shfl_sync(0xffffffffu, i1, src);
            float acc = 0.0f;
            for (int64_t c0 = b; c0 < e; c0 += 128) {
                // 128 tasks' terms in flight (a popular SKU's move has
                // hundreds of tasks, and the longest sets the kernel's time)
                int t[4];
                float term[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int64_t i = c0 + 32 * u + lane;
                    t[u] = i < e && M.task_cost[i].x >= 0 ? M.tasks[i].y : -1;
                    term[u] = i < e ? S.y_task[i] : 0.0f;
                }
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (t[u] >= 0) term[u] -= S.y_tour[t[u]];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const unsigned cm = __ballot_sync(0xffffffffu, t[u] >= 0);
#pragma unroll 8
                    for (int j = 0; j < 32; ++j) {
                        const float tj = __shfl_sync(0xffffffffu, term[u], j);
                        if ((cm >> j) & 1u) acc += tj;
                    }
                }
            }
            if (lane == src) sc = acc;
        }
        if (m < M.n_moves) S.score[m] = sc;
    }
}

__global__ void k_screen_select(ScreenArgs S) {
    pdl_trigger();
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int n_plans = S.M.a.n_plans;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < n_plans; p += warps) {
        uint32_t taken[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // up to 256 moves per plan
        for (int j = 0; j < S.keep; ++j) {
            float best = 3.0e38f;
            int bk = 0x7fffffff;
            for (int k = lane; k < S.moves_per_plan; k += 32) {
                if (taken[k >> 5] >> (k & 31) & 1u) continue;
                const float v = S.score[p * S.moves_per_plan + k];
                if (v < best || (v == best && k < bk)) { best = v; bk = k; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float ov = __shfl_xor_sync(0xffffffffu, best, o);
                const int ok = __shfl_xor_sync(0xffffffffu, bk, o);
                if (ov < best || (ov == best && ok < bk)) { best = ov; bk = ok; }
            }
            int4 out = make_int4(9, 0, 0, (int)p);
            if (best < 1.0e38f && bk < S.moves_per_plan) {
                out = S.M.moves[p * S.moves_per_plan + bk];
                taken[bk >> 5] |= 1u << (bk & 31);
            }
            if (lane == 0) S.kept[p * S.keep + j] = out;
        }
    }
}

}  // namespace

cudaError_t launch_task_features(const MoveArgs& M, const FeatConst& c, void* X, int num_sms, cudaStream_t s) {
    if (M.n_tasks == 0) return cudaSuccess;
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_task_features, TF_THREADS, 0);
    if (e != cudaSuccess) return e;
    int64_t grid = (int64_t)per_sm * num_sms;
    const int64_t want = (M.n_tasks + TF_THREADS / 32 - 1) / (TF_THREADS / 32);
    if (grid > want) grid = want;
    if (grid < 1) grid = 1;
    k_task_features<<<(int)grid, TF_THREADS, 0, s>>>(M, c, static_cast<uint4*>(X));
    return cudaGetLastError();
}

cudaError_t launch_screen_select(const ScreenArgs& S, cudaStream_t s) {
    launch_dependent(k_screen_score, grid_of(S.M.n_moves, 256), 256, 0, s, S);
    launch_dependent(k_screen_select, grid_of((int64_t)S.M.a.n_plans * 32, 256), 256, 0, s, S);
    return cudaGetLastError();
}

cudaError_t launch_ls_apply(const LsArgs& L, cudaStream_t s) {
    const size_t smem = sizeof(int32_t) * (size_t)L.seg_cap;
    cudaError_t e = cudaFuncSetAttribute(k_ls_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int grid = L.a.n_plans < 65536 ? L.a.n_plans : 65536;
    if (grid < 1) grid = 1;
    launch_dependent(k_ls_apply, grid, 256, smem, s, L);
    return cudaGetLastError();
}

}  // namespace wh

namespace wh {
cudaError_t launch_occupancy(const int32_t* slot_map, int64_t stride, int32_t n_plans, int32_t n_sku, int32_t n_loc,
                             uint32_t* used, int num_sms, cudaStream_t st) {
    const size_t words = (size_t)((n_loc + 31) >> 5) * (size_t)n_plans;
    cudaError_t e = cudaMemsetAsync(used, 0, words * sizeof(uint32_t), st);
    if (e != cudaSuccess || n_plans == 0 || n_sku == 0) return e;
    const int64_t total = (int64_t)n_plans * n_sku;
    const int64_t want = (total + 255) / 256;
    const int grid = (int)(want < (int64_t)num_sms * 16 ? want : (int64_t)num_sms * 16);
    k_occupancy<<<grid, 256, 0, st>>>(slot_map, stride, n_plans, n_sku, n_loc, used);
    return cudaGetLastError();
}
}  // namespace wh
