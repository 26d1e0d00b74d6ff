// Explicit optimal routes: for listed tours, the order in which a picker
// visits the tour's pick points along a shortest closed walk from the depot
// (the picking sequence the paper's case study asks for, Sec. 5 and Sec. 6),
// with its length.
//
// One tour per warp, its state in shared memory.  The lanes gather the tour's
// keys, sort them and drop repeats; lane 0 runs the Ratliff-Rosenthal DP in the
// same reduced 5-class form as the evaluation kernels, keeping the state before
// every visited aisle; the lanes then find, an aisle each, which arrival
// (source class and horizontal edge pattern over the aisle gaps) gave every
// class's minimum.  Backtracking from the cheapest final class fixes the
// route's subgraph: the horizontal edges between consecutive pick aisles
// (front, back: 0, 1 or 2 each) and every pick aisle's vertical option
// (traverse, double traverse, largest gap left out, from the front, from the
// back).  The subgraph has even degrees and one component; Hierholzer's
// algorithm (lane 0) walks it from the depot, and the picks are emitted in
// walking order: along a traversed aisle in the walking direction, on a spur
// (the out-and-back pieces of the gap, front and back options) when its end
// node is first reached.  The walk's length equals the DP's, so the emitted
// sequence, taken with shortest paths between consecutive points, is an
// optimal route.
//
// What bounds it: the latency of lane 0's serial parts, hidden by the warps of
// an SM (20 fit its shared memory).  Paper-scale tours of one plan (166):
// 56 us, of 64 plans 144 us, of 1,024 plans 1.94 ms; one tour per thread with
// its arrays in local memory took 743 us, 860 us and 2.44 ms.
#include "tour_core.cuh"

namespace wh {

namespace {

constexpr int RT_MAXL = ROUTE_MAX_POINTS;   // distinct pick points per tour, and so pick aisles
constexpr int RT_WARPS = 4;                 // tours per block
constexpr int RT_CHUNK = 256;               // lines gathered at a time

// one tour's state
struct RtWarp {
    uint32_t key[RT_MAXL + RT_CHUNK];   // the distinct points so far, then a chunk of lines
    uint2 rec[RT_MAXL];                 // per pick aisle: aisle << 16 | lo, hi << 16 | largest gap
    uint16_t beg[RT_MAXL + 2];          // first point of every pick aisle, then the number of points
    uint32_t dec[RT_MAXL];              // per class: arrival code and source class, 6 bits each
    uint8_t cls[RT_MAXL];               // the route's class after every pick aisle
    union {
        int state[RT_MAXL][5];          // DP state before every pick aisle (until dec is known)
        struct {
            uint16_t node[6 * RT_MAXL + 2];   // the walk's stack: (aisle + 1) * 2 + back, the depot 0
            uint32_t left[RT_MAXL + 2];       // [aisle + 1] edges not walked yet and what is emitted (RT_*)
            uint16_t fs_end[RT_MAXL], bs_beg[RT_MAXL];
        } walk;
    };
};

// walk.left: copies of the front edge into the aisle, of the back edge, of its
// traversal (two bits each), then the ends visited and the aisle emitted
constexpr int RT_VERT = 4, RT_SEEN = 6;
constexpr uint32_t RT_CROSSED = 1u << 8;

// arrival codes: (source class, horizontal pattern front/back)
enum { H_UU11 = 0, H_E020 = 1, H_EE20 = 2, H_OE02 = 3, H_EE02 = 4, H_EE22 = 5, H_E222 = 6 };
// classes
enum { C_UU = 0, C_E0 = 1, C_OE = 2, C_EE = 3, C_E2 = 4 };
// vertical options
enum { V_T = 1, V_D = 2, V_G = 3, V_F = 4, V_B = 5 };

__device__ __forceinline__ int h_src(int h) {
    return h == H_UU11 ? C_UU : h == H_E020 ? C_E0 : h == H_OE02 ? C_OE : h == H_E222 ? C_E2 : C_EE;
}
__device__ __forceinline__ int h_front(int h) {
    return h == H_UU11 ? 1 : (h == H_E020 || h == H_EE20 || h == H_EE22 || h == H_E222) ? 2 : 0;
}
__device__ __forceinline__ int h_back(int h) {
    return h == H_UU11 ? 1 : (h == H_OE02 || h == H_EE02 || h == H_EE22 || h == H_E222) ? 2 : 0;
}
__device__ __forceinline__ int vert_of(int cls, int h) {
    switch (cls) {
        case C_UU: return h == H_UU11 ? V_G : V_T;
        case C_EE: return h == H_UU11 ? V_T : (h == H_EE22 ? V_G : V_D);
        case C_E0: return V_F;
        case C_OE: return V_B;
        default: return V_G;
    }
}

// first argmin over candidates (value, code)
__device__ __forceinline__ void take(int& best, int& code, int val, int c) {
    if (val < best) {
        best = val;
        code = c;
    }
}

// The arrival code of every class after one pick aisle, from the state before
// it (dp_aisle_rel's form): the first minimum in a fixed order of the
// candidates, with its source class, 6 bits per class.
__device__ uint32_t arrival_codes(const DP5& v, const DPConst& k, int d, int lo, int hi, int gi) {
    const int h2 = k.p2 * d;
    int hv[7];
    hv[H_UU11] = v.uu;
    hv[H_E020] = v.e0;
    hv[H_EE20] = v.ee;
    hv[H_OE02] = v.oe;
    hv[H_EE02] = v.ee;
    hv[H_EE22] = v.ee + h2;
    hv[H_E222] = v.e2 + h2;
    const int cB = k.cb0 - lo * k.s2, cF = k.cf0 + hi * k.s2, cT = k.y, cD = k.y2;
    const int cG = min(min(cB, k.y2 - gi * k.s2), cF);
    const int big = 0x7fffffff;
    int uu = big, ee = big, e0 = big, oe = big, e2 = big;
    int kuu = 0, kee = 0, ke0 = 0, koe = 0, ke2 = 0;
    take(uu, kuu, hv[H_UU11] + cG, H_UU11);
    take(uu, kuu, hv[H_E020] + cT, H_E020);
    take(uu, kuu, hv[H_EE20] + cT, H_EE20);
    take(uu, kuu, hv[H_OE02] + cT, H_OE02);
    take(uu, kuu, hv[H_EE02] + cT, H_EE02);
    take(uu, kuu, hv[H_E222] + cT, H_E222);
    take(uu, kuu, hv[H_EE22] + cT, H_EE22);
    take(ee, kee, hv[H_UU11] + cT, H_UU11);
    take(ee, kee, hv[H_E020] + cD, H_E020);
    take(ee, kee, hv[H_EE20] + cD, H_EE20);
    take(ee, kee, hv[H_OE02] + cD, H_OE02);
    take(ee, kee, hv[H_EE02] + cD, H_EE02);
    take(ee, kee, hv[H_E222] + cD, H_E222);
    take(ee, kee, hv[H_EE22] + cG, H_EE22);
    take(e0, ke0, hv[H_E020] + cF, H_E020);
    take(e0, ke0, hv[H_EE20] + cF, H_EE20);
    take(oe, koe, hv[H_OE02] + cB, H_OE02);
    take(oe, koe, hv[H_EE02] + cB, H_EE02);
    take(e2, ke2, hv[H_E020] + cG, H_E020);
    take(e2, ke2, hv[H_EE20] + cG, H_EE20);
    take(e2, ke2, hv[H_OE02] + cG, H_OE02);
    take(e2, ke2, hv[H_EE02] + cG, H_EE02);
    take(e2, ke2, hv[H_E222] + cG, H_E222);
    auto entry = [](int code, int cls) { return (uint32_t)(code | (h_src(code) << 3)) << (6 * cls); };
    return entry(kuu, C_UU) | entry(ke0, C_E0) | entry(koe, C_OE) | entry(kee, C_EE) | entry(ke2, C_E2);
}

// The tour's lines [base, base + RT_CHUNK) as keys at out[0 ..), lanes over
// orders, then over lines; returns the tour's lines.  bad: status bits of what
// is invalid, the same in every lane.
__device__ __forceinline__ int gather_lines(const EvalArgs& a, const int32_t* map, int q0, int q1, int base,
                                            uint32_t* out, int lane, uint32_t& bad) {
    int n = 0;
    for (int qb = q0; qb < q1; qb += 32) {
        const int q = qb + lane;
        int lb = 0, cnt = 0;
        if (q < q1) {
            const int o = a.order_seq[q];
            if ((unsigned)o >= (unsigned)a.n_orders) {
                bad |= WH_STATUS_BAD_ORDER;
            } else {
                lb = a.order_off[o];
                const int le = a.order_off[o + 1];
                if (lb < 0 || le < lb || le > a.n_lines) bad |= WH_STATUS_BAD_OFFSET;
                else cnt = le - lb;
            }
        }
        const int incl = warp_inclusive_scan(cnt), at = n + incl - cnt - base;
        for (int l = max(0, -at); l < cnt && at + l < RT_CHUNK; ++l) out[at + l] = (uint32_t)(lb + l);
        n += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    const int m = min(n - base, RT_CHUNK);
    for (int x = lane; x < m; x += 32) {
        const int s = a.line_sku[out[x]];
        const int loc = (unsigned)s < (unsigned)a.n_sku ? map[s] : -1;
        if ((unsigned)loc >= (unsigned)a.g.n_loc) bad |= WH_STATUS_BAD_LOC;
        else out[x] = loc_key(a.g, loc);
    }
    __syncwarp();
    bad = __reduce_or_sync(0xffffffffu, bad);
    return n;
}

__global__ void __launch_bounds__(RT_WARPS * 32) k_routes(EvalArgs a, const int32_t* tours, int32_t n,
                                                          int32_t max_points, int32_t* points, int32_t* n_points,
                                                          int32_t* length) {
    __shared__ RtWarp s_tour[RT_WARPS];
    const int lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * RT_WARPS + (threadIdx.x >> 5);
    if (i >= n) return;   // (warps share nothing)
    const Geo& g = a.g;
    RtWarp& W = s_tour[threadIdx.x >> 5];
    int32_t* out = points + i * max_points;
    if (lane == 0) {
        n_points[i] = -1;
        length[i] = -1;
    }
    auto fail = [&](uint32_t bits) {
        if (lane == 0) flag(a.status, bits);
    };
    const int t = tours[i];
    if ((unsigned)t >= (unsigned)a.n_tours) return fail(WH_STATUS_BAD_OFFSET);
    const int plan = a.slot_stride != 0 ? warp_find_plan(a, t, lane) : 0;
    const int32_t* map = a.slot_map + (int64_t)plan * a.slot_stride;
    const int q0 = a.tour_off[t], q1 = a.tour_off[t + 1];
    if (q0 < 0 || q1 < q0 || (int64_t)q1 > a.n_seq) return fail(WH_STATUS_BAD_OFFSET);
    // the tour's distinct pick points (aisle << 16 | slot), ascending: chunks
    // of lines joined to the points so far, sorted, repeats dropped
    int np = 0;
    for (int base = 0, lines = 1; base < lines; base += RT_CHUNK) {
        uint32_t bad = 0;
        lines = gather_lines(a, map, q0, q1, base, W.key + np, lane, bad);
        if (bad) return fail(bad);
        const int have = np + min(lines - base, RT_CHUNK);
        if (have == 0) break;
        warp_sort_buffer(W.key, have, lane);
        np = 0;
        uint32_t before = KEY_NONE;
        for (int x0 = 0; x0 < have; x0 += 32) {
            const uint32_t k = x0 + lane < have ? W.key[x0 + lane] : KEY_NONE;
            uint32_t left = __shfl_up_sync(0xffffffffu, k, 1);
            if (lane == 0) left = before;
            before = __shfl_sync(0xffffffffu, k, 31);
            const bool keep = x0 + lane < have && k != left;
            const unsigned km = __ballot_sync(0xffffffffu, keep);
            __syncwarp();
            if (keep) W.key[np + __popc(km & ((1u << lane) - 1u))] = k;   // at or before its place
            np += __popc(km);
            __syncwarp();
        }
        if (np > RT_MAXL) return fail(WH_STATUS_TOUR_TOO_LONG);
    }
    if (np > max_points) return fail(WH_STATUS_TOUR_TOO_LONG);
    if (np == 0) {
        if (lane == 0) {
            n_points[i] = 0;
            length[i] = 0;
        }
        return;
    }
    // pick aisles and their records
    int m = 0;
    for (int x0 = 0; x0 < np; x0 += 32) {
        const int x = x0 + lane;
        const bool first = x < np && (x == 0 || (W.key[x - 1] >> 16) != (W.key[x] >> 16));
        const unsigned fm = __ballot_sync(0xffffffffu, first);
        if (first) W.beg[m + __popc(fm & ((1u << lane) - 1u))] = (uint16_t)x;
        m += __popc(fm);
    }
    if (lane == 0) W.beg[m] = (uint16_t)np;
    __syncwarp();
    for (int j = lane; j < m; j += 32) {
        const int b0 = W.beg[j], b1 = W.beg[j + 1];
        const uint32_t k0 = W.key[b0], k1 = W.key[b1 - 1];
        uint32_t gi = 0;
        for (int x = b0 + 1; x < b1; ++x) gi = max(gi, W.key[x] - W.key[x - 1]);
        W.rec[j] = make_uint2(k0, (k1 << 16) | gi);
    }
    __syncwarp();
    const DPConst kc = dp_const(g);
    int len = 0, cls = C_EE;
    if (lane == 0) {
        DP5 v;
        dp_init(v);
        int pa = 0;
        uint2 r = W.rec[0];
        for (int j = 0; j < m; ++j) {
            const uint2 rn = j + 1 < m ? W.rec[j + 1] : r;
            int* st = W.state[j];
            st[0] = v.uu; st[1] = v.e0; st[2] = v.oe; st[3] = v.ee; st[4] = v.e2;
            const int ai = (int)(r.x >> 16);
            dp_aisle_rel(v, kc, ai - pa, (int)(r.x & 0xFFFFu), (int)(r.y >> 16), (int)(r.y & 0xFFFFu));
            pa = ai;
            r = rn;
        }
        int best = v.ee;
        if (v.e0 < best) { best = v.e0; cls = C_E0; }
        if (v.oe < best) { best = v.oe; cls = C_OE; }
        len = best + kc.p2 * pa;
    }
    __syncwarp();
    for (int j = lane; j < m; j += 32) {
        const int* st = W.state[j];
        DP5 v;
        v.uu = st[0]; v.e0 = st[1]; v.oe = st[2]; v.ee = st[3]; v.e2 = st[4];
        const uint2 r = W.rec[j];
        const int pa = j > 0 ? (int)(W.rec[j - 1].x >> 16) : 0;
        W.dec[j] = arrival_codes(v, kc, (int)(r.x >> 16) - pa, (int)(r.x & 0xFFFFu), (int)(r.y >> 16),
                                           (int)(r.y & 0xFFFFu));
    }
    __syncwarp();   // the states are done with: the walk's arrays take their place
    // backtrack: the class after every pick aisle (the table's reads do not
    // wait for it)
    int ok = 1;
    if (lane == 0) {
        uint32_t d = W.dec[m - 1];
        for (int j = m - 1; j >= 0; --j) {
            const uint32_t dn = j > 0 ? W.dec[j - 1] : 0u;
            W.cls[j] = (uint8_t)cls;
            cls = (int)(d >> (6 * cls + 3)) & 7;
            d = dn;
        }
        ok = cls == C_E0;   // the walk starts at the depot, on the front
        if (h_back((int)(W.dec[0] >> (6 * W.cls[0])) & 7) != 0) ok = 0;
    }
    __syncwarp();   // lane 0's classes are read by every lane (a shuffle orders no memory)
    ok = __shfl_sync(0xffffffffu, ok, 0);
    if (!ok) return fail(WH_STATUS_BAD_OFFSET);
    // per pick aisle, the edges into it from the left (front, back: 0..2 each)
    // and its vertical option, with the
    // spurs of the gap / front / back options: the front spur covers points
    // [beg, fs_end), the back spur [bs_beg, end) of the aisle; and the edges
    int n_edges = 0;
    for (int j = lane; j < m; j += 32) {
        const int b0 = W.beg[j], b1 = W.beg[j + 1], c = W.cls[j];
        const int h = (int)(W.dec[j] >> (6 * c)) & 7, vo = vert_of(c, h);
        int fs = b0, bs = b1;
        if (vo == V_F) {
            fs = b1;
        } else if (vo == V_B) {
            bs = b0;
        } else if (vo == V_G) {
            // leave out the largest of the front gap, the inner gaps and the
            // back gap (the DP's choice; ties give the same length)
            const int lo = (int)(W.key[b0] & 0xFFFFu), hi = (int)(W.key[b1 - 1] & 0xFFFFu);
            const int gfront = g.h + lo * g.S, gback = g.Y - (g.h + hi * g.S);
            int gin = 0, split = b0;   // largest inner gap: between points split - 1 and split
            for (int x = b0 + 1; x < b1; ++x) {
                const int dgap = ((int)(W.key[x] & 0xFFFFu) - (int)(W.key[x - 1] & 0xFFFFu)) * g.S;
                if (dgap > gin) { gin = dgap; split = x; }
            }
            if (gfront >= gin && gfront >= gback) {
                bs = b0;          // everything from the back
            } else if (gback >= gin) {
                fs = b1;          // everything from the front
            } else {
                fs = bs = split;
            }
        }
        W.walk.fs_end[j] = (uint16_t)fs;
        W.walk.bs_beg[j] = (uint16_t)bs;
        const int hf = h_front(h), hb = h_back(h), nv = vo == V_T ? 1 : vo == V_D ? 2 : 0;
        W.walk.left[j + 1] = (uint32_t)(hf | (hb << 2) | (nv << RT_VERT));
        n_edges += hf + hb + nv;
    }
    if (lane == 0) W.walk.left[0] = W.walk.left[m + 1] = 0u;
    n_edges = (int)__reduce_add_sync(0xffffffffu, (unsigned)n_edges);
    __syncwarp();
    if (lane != 0) return;
    // The route's multigraph: the depot (aisle -1), and every pick aisle's
    // front and back end; parallel edges are alike, so only their numbers are
    // kept.  Hierholzer from the depot, at every node an edge to the left
    // first, then to the right, then the aisle.  Nodes are popped in the order
    // of an Euler circuit (the reverse of the usual output, itself a circuit
    // from the depot); consecutive pops are neighbours in the graph (the two
    // ends of one aisle: along it).  Picks are emitted while walking it: along
    // an aisle the first time it is traversed, in the walking direction; a
    // spur's points the first time its end node is reached.
    int w = 0, n_pop = 0, prev = -1, sp = 1;
    int u = 0;                                                        // (aisle + 1) * 2 + back
    uint32_t here = W.walk.left[0], right = W.walk.left[1];           // of u's aisle and the next
    W.walk.node[0] = 0;
    while (sp > 0) {
        const int j1 = u >> 1, sh = (u & 1) * 2;
        if ((here >> sh) & 3u) {
            W.walk.left[j1] = here - (1u << sh);
            right = here - (1u << sh);
            u -= 2;
            here = W.walk.left[j1 - 1];
        } else if ((right >> sh) & 3u) {
            here = right - (1u << sh);
            W.walk.left[j1 + 1] = here;
            u += 2;
            right = W.walk.left[j1 + 2];
        } else if ((here >> RT_VERT) & 3u) {
            here -= 1u << RT_VERT;
            W.walk.left[j1] = here;
            u ^= 1;
        } else {
            // no edge is left at u: it leaves the stack
            const int x = u, j = j1 - 1;
            --sp;
            if (x > 0) {
                const int b0 = W.beg[j], b1 = W.beg[j + 1];
                uint32_t now = here;
                if (prev == (x ^ 1) && !(now & RT_CROSSED)) {
                    now |= RT_CROSSED;
                    if (prev < x) {   // front -> back: deeper picks later
                        for (int y = b0; y < b1; ++y) out[w++] = (int32_t)W.key[y];
                    } else {
                        for (int y = b1 - 1; y >= b0; --y) out[w++] = (int32_t)W.key[y];
                    }
                }
                const uint32_t seen = 1u << (RT_SEEN + (x & 1));
                if (!(now & seen)) {
                    now |= seen;
                    if (!(x & 1)) {   // front end: up to the gap
                        for (int y = b0; y < W.walk.fs_end[j]; ++y) out[w++] = (int32_t)W.key[y];
                    } else {          // back end: down to the gap
                        for (int y = b1 - 1; y >= W.walk.bs_beg[j]; --y) out[w++] = (int32_t)W.key[y];
                    }
                }
                W.walk.left[j1] = now;
            }
            prev = x;
            ++n_pop;
            if (sp > 0) {
                u = W.walk.node[sp - 1];
                here = W.walk.left[u >> 1];
                right = W.walk.left[(u >> 1) + 1];
            }
            continue;
        }
        W.walk.node[sp++] = (uint16_t)u;
    }
    if (n_pop != n_edges + 1 || prev != 0 || w != np) return fail(WH_STATUS_BAD_OFFSET);
    n_points[i] = np;
    length[i] = len;
}

}  // namespace

cudaError_t launch_routes(const EvalArgs& a, const int32_t* tours, int32_t n, int32_t max_points, int32_t* points,
                          int32_t* n_points, int32_t* length, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_routes<<<(n + RT_WARPS - 1) / RT_WARPS, RT_WARPS * 32, 0, s>>>(a, tours, n, max_points, points, n_points, length);
    return cudaGetLastError();
}

}  // namespace wh
