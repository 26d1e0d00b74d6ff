// Plan evaluation with one CTA per plan, for plans that each have their own
// slotting and for layouts whose keys need 32 bits.
//
// k_eval_short walks each tour's orders straight into the plan's slotting in
// global memory: chains of dependent loads with few warps to hide them, 32
// keys or more a thread in registers, and a separate pass of one warp a tour
// for tours of more than 64 lines or 32 aisles.  Here a CTA takes a plan
// through short phases of few registers each:
//   count      a thread per tour: its orders checked and counted, a row of
//              shared memory for its keys and every order's place in it;
//   translate  a thread per order-book line, in line order: SKU (coalesced),
//              its location under the plan's slotting (eight independent
//              gathers in flight) and the key written to the order's place;
//   sort       2, 4 or 8 lanes a tour with 16 keys each: a merge-exchange
//              network in the lane, bitonic merges across lanes by shuffles;
//   cost       a thread per tour, ordered by line count: one pass over the
//              sorted row, a DP step where an aisle ends (no record slots,
//              so no limit on a tour's aisles).
#include "row_core.cuh"

namespace wh {
namespace {

constexpr int PL_THREADS = 256;
constexpr int PL_MAXN = ROW_MAXN;   // longer tours go to the long-tour pass

// Line count of tour t, its orders checked: -1 for invalid offsets or ids
// (flagged), PL_MAXN + 1 for a tour that the long-tour pass takes.  Four
// order ids in flight.
__device__ __forceinline__ int count_lines(const EvalArgs& a, const uint8_t* s_cnt, int t, int& q0, int& q1) {
    q0 = __ldg(a.tour_off + t);
    q1 = __ldg(a.tour_off + t + 1);
    if (q0 < 0 || q1 < q0 || (int64_t)q1 > a.n_seq) {
        flag(a.status, WH_STATUS_BAD_OFFSET);
        return -1;
    }
    int n = 0;
    bool bad = false;
    for (int q = q0; q < q1; q += 4) {
        int o[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) o[u] = q + u < q1 ? __ldg(a.order_seq + q + u) : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if ((unsigned)o[u] < (unsigned)a.n_orders) n += s_cnt[o[u]];
            else bad |= q + u < q1;
        }
        n = min(n, PL_MAXN + 1);
    }
    if (bad) {
        flag(a.status, WH_STATUS_BAD_ORDER);
        return -1;
    }
    return n;
}

// sum over the warp's lanes of values 0 <= v < 2^31
__device__ __forceinline__ long long warp_sum31(int v) {
    const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)v >> 16);
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0xFFFFu);
    return ((long long)hi << 16) + lo;
}

// LIST: tours of a plan taken per round (each round translates the order book
// anew); CTAS: per SM.
template <bool SHARED_MAP, int LIST, int CTAS>
__global__ void __launch_bounds__(PL_THREADS, CTAS) k_eval_plan(EvalArgs a) {
    constexpr int T = PL_THREADS, PL_U = LIST / T;
    extern __shared__ __align__(16) uint32_t rows[];   // keys, then per order: place, line count, seen bit
    __shared__ int s_bin[PL_MAXN + 1];        // tours of every line count, then their first place in the list
    __shared__ uint16_t s_list[LIST];      // the round's tours by falling line count
    __shared__ uint16_t s_base[LIST];      // their rows, by tour
    __shared__ uint8_t s_n[LIST];          // their line counts, by tour
    __shared__ int s_total, s_unit, s_rows;
    __shared__ bool s_untidy;
    const int tid = threadIdx.x, lane = tid & 31;
    uint32_t* s_dst32 = rows + a.n_lines;     // first place of an order's lines, 16 bits each (0xFFFF: none)
    uint16_t* s_dst = reinterpret_cast<uint16_t*>(s_dst32);
    const int n_dst = (a.n_orders + 1) >> 1, n_seen = (a.n_orders + 31) >> 5;
    uint32_t* s_seen = s_dst32 + n_dst;
    uint8_t* s_cnt = reinterpret_cast<uint8_t*>(s_seen + n_seen);
    const bool need_rr = (a.mask & WH_ROUTE_OPTIMAL) != 0;
    const bool want_s = (a.mask & WH_ROUTE_SSHAPE) != 0;

    // (no early trigger: the long-tour kernel's blocks would take the shared
    // memory that is this one's L1)
    pdl_wait();
    // line counts, up to 255 (an order of more than PL_MAXN lines makes its
    // tour a long one); an order book with malformed offsets has no line ->
    // order table to go by: every tour goes to the long-tour pass
    // (2,000 plans of 4,000 orders: 207 us also with an order of 300 lines in
    // the book, 304 with it in a tour of every plan, 222 with an order twice in
    // every plan; 640, 953 and 656 with all tours handed over for it)
    bool odd = false;
    for (int o = tid; o < a.n_orders; o += T) {
        const int lb = a.order_off[o], le = a.order_off[o + 1];
        const bool ok = lb >= 0 && le >= lb && le <= a.n_lines;
        s_cnt[o] = ok ? (uint8_t)min(le - lb, 255) : 0;
        odd |= !ok;
    }
    if (tid == 0) s_untidy = (__ldcg(a.status) & WH_STATUS_BAD_OFFSET) != 0;
    odd = __syncthreads_or(odd);

    // Malformed plan offsets (k_prep has flagged them; or another call whose
    // bit nobody has read) must still leave every tour with one plan, the first
    // that ends behind it or else the last, as k_eval_short has it: a plan
    // begins at the largest end of those before.
    const bool untidy = s_untidy;
    int begin = 0, seen = 0;   // the largest of plan offsets 1 .. seen - 1
    for (int plan = blockIdx.x; plan < a.n_plans; plan += gridDim.x) {
        const int32_t* map = SHARED_MAP ? nullptr : a.slot_map + (int64_t)plan * a.slot_stride;
        int t0 = a.plan_tour_off[plan], t1 = a.plan_tour_off[plan + 1];
        if (untidy) {
            for (; seen <= plan; ++seen) begin = max(begin, seen > 0 ? a.plan_tour_off[seen] : 0);
            t0 = min(begin, a.n_tours);
            t1 = plan == a.n_plans - 1 ? a.n_tours : min(max(begin, t1), a.n_tours);
        }
        for (int tb = t0; tb < t1; tb += LIST) {
            const int nt = min(LIST, t1 - tb);
            for (int i = tid; i <= PL_MAXN; i += T) s_bin[i] = 0;
            for (int i = tid; i < n_dst; i += T) s_dst32[i] = 0xFFFFFFFFu;
            for (int i = tid; i < n_seen; i += T) s_seen[i] = 0u;
            if (tid == 0) s_unit = s_rows = 0;
            __syncthreads();
            // ---- count
            int at[PL_U];   // line count << 16 | place in its bin, -1: not scored here
#pragma unroll
            for (int u = 0; u < PL_U; ++u) {
                const int i = tid + u * T;
                at[u] = -1;
                if (i >= nt) continue;
                int q0, q1;
                const int n = count_lines(a, s_cnt, tb + i, q0, q1);
                if (n < 0) {
                    if (a.tour_s) a.tour_s[tb + i] = -1;
                    if (a.tour_rr) a.tour_rr[tb + i] = -1;
                    continue;
                }
                // the long-tour pass takes tours of too many lines, tours that
                // want an order which another place has already, and the tours
                // that the rows have no room for then
                const int base = !odd && n <= PL_MAXN ? atomicAdd(&s_rows, n) : a.n_lines + 1;
                if (base + n <= a.n_lines) {
                    s_n[i] = (uint8_t)n;
                    s_base[i] = (uint16_t)base;
                    at[u] = n << 16 | atomicAdd(&s_bin[n], 1);
                    int pos = base;
                    bool taken = false;
                    for (int q = q0; q < q1; q += 4) {
                        int o[4];
#pragma unroll
                        for (int v = 0; v < 4; ++v) o[v] = q + v < q1 ? __ldg(a.order_seq + q + v) : -1;
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            if (o[v] < 0) continue;
                            const int cnt = s_cnt[o[v]];
                            const uint32_t bit = cnt > 0 ? 1u << (o[v] & 31) : 0u;
                            if (atomicOr(&s_seen[o[v] >> 5], bit) & bit) taken = true;
                            else s_dst[o[v]] = (uint16_t)pos;
                            pos += cnt;
                        }
                    }
                    if (!taken) continue;
                    s_n[i] = 0;   // it keeps its place in the list, as a tour of no lines
                }
                const int slot = atomicAdd(a.long_count, 1);
                if (slot < a.long_cap) {
                    a.long_list[3 * slot] = 0;
                    a.long_list[3 * slot + 1] = tb + i;
                    a.long_list[3 * slot + 2] = plan;
                } else {
                    flag(a.status, WH_STATUS_LONG_OVERFLOW);
                    if (a.tour_s) a.tour_s[tb + i] = -1;
                    if (a.tour_rr) a.tour_rr[tb + i] = -1;
                }
            }
            __syncthreads();
            if (odd) continue;   // (every tour handed over)
            // the bins' first places in the list: most lines first
            if (tid < 32) {
                constexpr int B = (PL_MAXN + 32) / 32;
                int v[B], sum = 0;
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    const int b = PL_MAXN - (B * lane + u);
                    v[u] = b >= 0 ? s_bin[b] : 0;
                    sum += v[u];
                }
                const int incl = warp_inclusive_scan(sum);
                int pos = incl - sum;
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    const int b = PL_MAXN - (B * lane + u);
                    if (b >= 0) s_bin[b] = pos;
                    pos += v[u];
                }
                if (lane == 31) s_total = incl;
            }
            // ---- translate
            for (int l0 = tid; l0 < a.n_lines; l0 += 8 * T) {
                uint32_t sk[8], at_o[8];
                int loc[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int l = l0 + u * T;
                    sk[u] = l < a.n_lines ? (SHARED_MAP ? a.line_key[l] : (uint32_t)__ldg(a.line_sku + l)) : 0u;
                    at_o[u] = l < a.n_lines ? a.line_ord[l] : 0xFFFFFFFFu;
                }
                if constexpr (!SHARED_MAP) {
#pragma unroll
                    for (int u = 0; u < 8; ++u) loc[u] = sk[u] < (uint32_t)a.n_sku ? __ldg(map + sk[u]) : 0;
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (at_o[u] == 0xFFFFFFFFu) continue;   // past the end, or in no order
                    const uint32_t d = s_dst[at_o[u] >> 8];
                    if (d == 0xFFFFu) continue;             // in none of the round's tours
                    uint32_t k = sk[u];
                    if constexpr (!SHARED_MAP) {
                        k = loc_key(a.g, loc[u]);
                        if ((uint32_t)loc[u] >= (uint32_t)a.g.n_loc) k = KEY_BAD;
                        if (sk[u] >= (uint32_t)a.n_sku) k = KEY_BAD_SKU;
                    }
                    rows[d + (at_o[u] & 0xFFu)] = k;
                }
            }
            __syncthreads();
#pragma unroll
            for (int u = 0; u < PL_U; ++u)
                if (at[u] >= 0) s_list[s_bin[at[u] >> 16] + (at[u] & 0xFFFF)] = (uint16_t)(tid + u * T);
            __syncthreads();
            // ---- sort: units of a warp's tours, the longest first
            const int total = s_total, c8 = s_bin[64], c4 = s_bin[32];   // tours over 64 and over 32 lines
            const int u8n = (c8 + 3) >> 2, u4n = u8n + ((c4 - c8 + 7) >> 3), un = u4n + ((total - c4 + 15) >> 4);
            for (;;) {
                int u = lane == 0 ? atomicAdd(&s_unit, 1) : 0;
                u = __shfl_sync(0xffffffffu, u, 0);
                if (u >= un) break;
                const int G = u < u8n ? 8 : u < u4n ? 4 : 2;
                const int i0 = G == 8 ? 4 * u : G == 4 ? c8 + 8 * (u - u8n) : c4 + 16 * (u - u4n);
                sort_rows(G, rows, s_list, s_base, s_n, i0, G == 8 ? c8 : G == 4 ? c4 : total, lane);
            }
            __syncthreads();
            // ---- cost
            const DPConst c = dp_const(a.g);
            for (int i0 = tid & ~31; i0 < total; i0 += T) {
                const bool on = i0 + lane < total;
                const int k = on ? s_list[i0 + lane] : 0, t = tb + k, n = on ? s_n[k] : 0;
                const uint32_t* row = rows + (on ? s_base[k] : 0);
                int cs, cr;
                row_costs(a.g, c, row, n, need_rr, cs, cr);
                const bool kbad = n > 0 && row[n - 1] >= KEY_BAD_SKU;
                if (kbad) {
                    if constexpr (!SHARED_MAP)   // under a shared slotting k_prep has flagged the line
                        for (int p = n - 1; p >= 0 && row[p] >= KEY_BAD_SKU; --p)
                            flag(a.status, row[p] == KEY_BAD ? WH_STATUS_BAD_LOC : WH_STATUS_BAD_SKU);
                    if (a.tour_s) a.tour_s[t] = -1;
                    if (a.tour_rr) a.tour_rr[t] = -1;
                } else if (on) {
                    if (a.tour_s && want_s) a.tour_s[t] = cs;
                    if (a.tour_rr && need_rr) a.tour_rr[t] = cr;
                }
                const bool ok = on && !kbad;
                const long long ss = warp_sum31(ok ? cs : 0), sr = warp_sum31(ok ? cr : 0);
                if (lane == 0) {
                    if (a.plan_s && want_s && ss)
                        atomicAdd(reinterpret_cast<unsigned long long*>(&a.plan_s[plan]), (unsigned long long)ss);
                    if (a.plan_rr && need_rr && sr)
                        atomicAdd(reinterpret_cast<unsigned long long*>(&a.plan_rr[plan]), (unsigned long long)sr);
                }
            }
            __syncthreads();   // the rows are about to be rewritten
        }
    }
}

size_t plan_smem_bytes(const EvalArgs& a) {
    return sizeof(uint32_t) * ((size_t)a.n_lines + ((size_t)a.n_orders + 1) / 2 + ((size_t)a.n_orders + 31) / 32) +
           (((size_t)a.n_orders + 15) & ~(size_t)15);
}

// Four CTAs an SM and lists of 512 tours instead of three and 1,024 (launch_eval_plan).
bool four_ctas(const EvalArgs& a) {
    return plan_smem_bytes(a) <= (a.slot_stride == 0 ? 53 : 40) * 1024 && a.n_tours <= 448ll * a.n_plans;
}

// k_eval_short walks what the plans hold; here every plan has the whole order
// book translated, again for every round of its tours, and a thread for every
// tour.  Microseconds of either beyond what both take, as they were measured
// over 792 shapes (books of 600 to 4,000 orders, plans that hold 32 orders to
// all of them in tours of 1 to 24, 16 to 2,000 plans; own slottings of 200,000
// and of 8,000 locations and shared ones): k_eval_short's chain of loads per
// line or its lines' throughput, this kernel's latency for a book and its
// tours or its throughput.
bool short_is_faster(const EvalArgs& a) {
    const bool own = a.slot_stride != 0;
    const double plans = a.n_plans, book = a.n_lines, tours = a.n_tours / plans;
    const double held = a.n_orders > 0 ? book * ((double)a.n_seq / a.n_orders) / plans : 0.0, lines = held / tours;
    const double rounds = 1 + (int)(tours / (four_ctas(a) ? 512 : 1024));
    const double chain = (!own ? 0.6 : key16_ok(a.g) ? 1.8 : 1.0) * lines;
    const double walk = (own ? 25e-6 : 14.5e-6) * plans * held;
    const double latency = (own ? 0.7e-3 : 0.5e-3) * rounds * book + 18e-3 * tours + 0.18 * lines;
    const double work = own ? rounds * (13e-3 + 5e-6 * book) + 2.5e-6 * held + 23e-6 * tours
                            : rounds * (13e-3 + 0.6e-6 * book) + 5e-6 * held + 30e-6 * tours;
    const double both = 16.0;
    return both + (latency > plans * work ? latency : plans * work) > 1.1 * (both + (chain > walk ? chain : walk));
}

}  // namespace

// Measured against k_eval_short + k_eval_long (us a call, GB300; orders x
// tours a plan x lines a tour):
//   own slottings    4,000 x 167 x 59, 500 aisles: 16 plans 58 -> 32,
//                    500 plans 167 -> 68, 2,000 plans 516 -> 202
//                    4,000 x 200 x 49, 40 aisles: 16 plans 58 -> 28,
//                    2,000 plans 238 -> 156
//                    300 x 38 x 20: 500 plans 33 -> 19, 2,000 plans 40 -> 50
//                    400 x 17 x 59: 500 plans 54 -> 23, 2,000 plans 82 -> 77
//   shared, 32-bit   4,000 x 167 x 59: 16 plans 46 -> 29, 2,000 plans 334 -> 145
//                    400 x 17 x 59: 152 plans 37 -> 19, 2,000 plans 50 -> 72
//                    3,000 x 375 x 20: 64 plans 25 -> 29, 152 plans 29 -> 27,
//                    2,000 plans 206 -> 99
//   own, 4,000 orders in the book, 500 aisles
//                    all held, a tour each: 16 plans 18 -> 105, 600 plans 204 -> 271
//                    128 held, a tour each: 2,000 plans 42 -> 124
//                    512 held, 8 a tour: 16 plans 38 -> 26, 2,000 plans 80 -> 134
//                    1,000 held, 24 a tour: 16 plans 67 -> 33, 600 plans 86 -> 76
// So: many plans of few tours (a CTA's threads idle, and one tour per thread
// fills the chip anyway), few plans of short tours under a shared slotting
// (k_eval_short has no latency of gathers or of a long-tour pass there) and
// short tours or small parts of a large book where that tells (short_is_faster)
// stay.  With the last of them left out, the 792 shapes take on average 18 %
// more than the faster of the two, with it 2 %.
// Three CTAs an SM take order books of up to 67 KB; a shared slotting with
// 16-bit keys is k_eval_short's best case (half the sort, one gather).
bool eval_plan_applies(const EvalArgs& a, int num_sms) {
    if (sshape_kernel_applies(a) || a.n_tours == 0 || a.n_lines > 0xFFFE || plan_smem_bytes(a) > 67 * 1024) return false;
    if (a.n_plans > 4 * num_sms && a.n_tours / a.n_plans < 64) return false;
    if (a.slot_stride == 0) {
        if (key16_ok(a.g)) return false;
        if (a.n_plans < num_sms &&
            (double)a.n_lines * (double)a.n_seq <= 32.0 * (double)a.n_orders * (double)a.n_tours)
            return false;
    }
    return !short_is_faster(a);
}

// Three CTAs an SM (60 KB an order book at paper scale; what is left of the
// 228 KB is the L1 that the gathers go through; 320 threads a CTA took the
// same time), or four with lists of 512 tours where four books leave that much
// too and few plans need a second round.  At paper scale four CTAs left the L1
// 3 KB and took 1,019 us instead of 745; 2,000 plans of 3,000 orders in 300
// aisles 141 -> 126 us, under a shared slotting (no gathers) 113 -> 99.
cudaError_t launch_eval_plan(const EvalArgs& a, int num_sms, cudaStream_t s) {
    const size_t smem = plan_smem_bytes(a);
    const bool shared = a.slot_stride == 0;
    const bool four = four_ctas(a);
    auto kern = shared ? (four ? k_eval_plan<true, 512, 4> : k_eval_plan<true, 1024, 3>)
                       : (four ? k_eval_plan<false, 512, 4> : k_eval_plan<false, 1024, 3>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int grid = a.n_plans;
    if (grid > num_sms) {
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PL_THREADS, smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
        if (grid > per_sm * num_sms) grid = per_sm * num_sms;
    }
    // beside k_prep's blocks an SM keeps their split of L1 and shared memory:
    // no matter with a block an SM (16 plans 35 -> 32 us), but not with more
    if (grid <= num_sms) return launch_dependent(kern, grid, PL_THREADS, smem, s, a);
    kern<<<grid, PL_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace wh
