// Seed-and-grow batch formation on the GPU: the orders are partitioned into
// picker tours by the exact optimal route length (the paper's clustering of
// orders and suggestion of which orders are picked together, Sec. 5 and
// Sec. 6).  One CTA per slotting runs the greedy:
//   seed - the unassigned order whose tour alone is longest (ties: lowest id);
//   grow - add the fitting unassigned order that lengthens the tour least
//          (ties: lowest id) until the order or line capacity is reached or
//          no order fits;
// until every order is in a tour.
//
// The current tour lives in shared memory as one 256-bit pick-depth mask per
// aisle and the sorted list of its aisles with their records (shallowest,
// deepest, the two largest gaps between consecutive picks), and, for every
// position of that list, the 5-class DP's state before it (F) and the cost to
// go from it (G, the same min-plus steps run backwards).  A candidate's length
// is then the DP from F at its first aisle over the aisles up to its last,
// closed with G: steps only where the candidate changes the tour, not one per
// aisle of it.
//
// Candidates are scored lazily.  The optimal length of a pick set never falls
// when picks are added, so the length with any part of a candidate, or with an
// earlier, smaller state of the same tour, bounds its length now from below.
// A tour's first growth step bounds every order by up to three of its lines
// taken one at a time (one DP step each); after that an order's bound is its last score in
// this tour.  Each step scores the candidate of the lowest bound, and then, if
// others are bounded below that score, those: the choice (least length, ties
// to the lowest id) is the one of scoring them all.
//
// What bounds it: the latency of a growth step (six barriers, the two serial
// chains of F and G, two rounds of candidate DPs), one CTA per slotting.
// Mid-size, 4,000 orders under 304 slottings: 24 ms; scoring every
// candidate over all of the tour's aisles in every step took 226 ms.
#include "tour_core.cuh"

namespace wh {

namespace {

constexpr int BG_THREADS = 512;
constexpr int BG_QUEUE = 1024;   // candidates queued for a step's second round; more are scored in place

// the DP state before a list position, or the costs to go from it
struct __align__(16) BgVec {
    int v[8];   // five used
};

struct BgShared {
    uint16_t* key;       // [n_lines] aisle << 8 | slot under this slotting
    int32_t* off;        // [n_orders + 1]; the top bit of off[o] marks an assigned order
    int32_t* bound;      // [n_orders] by position in rem: a lower bound of the tour's length with that order
    uint32_t* mask;      // [A][8] the tour's pick-depth bits per aisle (zero: none)
    uint2* list;         // [A] the tour's aisles, ascending: aisle << 24 | lo << 16 | hi << 8 | gap and where
                         //     that (largest) gap begins << 8 | the largest of the others
    uint16_t* first;     // [A] entries of list before the aisle
    BgVec* F;            // [A + 1] relative-form DP state before list entry j (dp_aisle_rel)
    BgVec* G;            // [A] cost to go from a state at list entry j, per class and crossing
    uint16_t* rem;       // [n_orders] the unassigned orders, compacted (any order)
    uint16_t* by_len;    // [n_orders] orders by their tour alone, longest first, ties by id
};

constexpr int BG_OFF_MASK = 0x7fffffff;

// shallowest / deepest set slot and the largest gap between consecutive set
// slots of a 256-bit mask (at least one bit set)
__device__ __forceinline__ void mask_stats(const uint32_t (&m)[8], int& lo, int& hi, int& gap) {
    lo = -1;
    hi = -1;
    gap = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        uint32_t b = m[w];
        while (b) {
            const int k = 32 * w + __ffs(b) - 1;
            b &= b - 1;
            if (lo < 0) lo = k;
            else gap = max(gap, k - hi);
            hi = k;
        }
    }
}

__device__ __forceinline__ void load_mask(const uint32_t* p, uint32_t (&m)[8]) {
    const uint4 x = *reinterpret_cast<const uint4*>(p), y = *reinterpret_cast<const uint4*>(p + 4);
    m[0] = x.x; m[1] = x.y; m[2] = x.z; m[3] = x.w;
    m[4] = y.x; m[5] = y.y; m[6] = y.z; m[7] = y.w;
}

__device__ __forceinline__ void put_state(BgVec* p, const DP5& v) {
    *reinterpret_cast<int4*>(p->v) = make_int4(v.uu, v.e0, v.oe, v.ee);
    p->v[4] = v.e2;
}

__device__ __forceinline__ DP5 get_state(const BgVec* p) {
    const int4 x = *reinterpret_cast<const int4*>(p->v);
    DP5 v;
    v.uu = x.x; v.e0 = x.y; v.oe = x.z; v.ee = x.w; v.e2 = p->v[4];
    return v;
}

// One backward step of dp_aisle_rel: with the cost to go g per class after
// the aisle, the cost to go from the state before it, held per term of that
// step: uu; min(e0, ee); min(oe, ee); ee and e2, each plus 2P per aisle crossed.
__device__ __forceinline__ DP5 back_step(const DP5& g, const DPConst& c, int lo, int hi, int gi) {
    const int cB = c.cb0 - lo * c.s2, cF = c.cf0 + hi * c.s2;
    const int cG = __vimin3_s32(cB, c.y2 - gi * c.s2, cF);
    const int yu = g.uu + c.y;
    const int m = __viaddmin_s32(g.ee, c.y2, __viaddmin_s32(g.e2, cG, yu));
    DP5 r;
    r.uu = __viaddmin_s32(g.uu, cG, g.ee + c.y);
    r.e0 = __viaddmin_s32(g.e0, cF, m);
    r.oe = __viaddmin_s32(g.oe, cB, m);
    r.ee = __viaddmin_s32(g.ee, cG, yu);
    r.e2 = m;
    return r;
}

// the same terms as classes of a state d aisles to the left
__device__ __forceinline__ DP5 back_cross(const DP5& t, const DPConst& c, int d) {
    DP5 g;
    g.uu = t.uu;
    g.e0 = t.e0;
    g.oe = t.oe;
    g.ee = __viaddmin_s32(t.ee, c.p2 * d, min(t.e0, t.oe));
    g.e2 = t.e2 + c.p2 * d;
    return g;
}

// Shallowest, deepest and largest gap of a listed aisle with one more pick k:
// only a pick inside the largest gap can shrink it.
__device__ __forceinline__ void add_pick(uint2 r, int k, int& lo, int& hi, int& gap) {
    lo = (int)(r.x >> 16) & 0xFF;
    hi = (int)(r.x >> 8) & 0xFF;
    gap = (int)(r.x & 0xFFu);
    const int from = (int)(r.y >> 8), to = from + gap;
    if (k < lo) {
        gap = max(gap, lo - k);
        lo = k;
    } else if (k > hi) {
        gap = max(gap, k - hi);
        hi = k;
    } else if (k > from && k < to) {
        gap = __vimax3_s32((int)(r.y & 0xFFu), k - from, to - k);
    }
}

// length of the tour from the state v after aisle pa, list entries j .. nt - 1 to go
__device__ __forceinline__ int close_with(const BgShared& S, const DPConst& c, const DP5& v, int pa, int j, int nt) {
    if (j >= nt) return dp_final(v) + c.p2 * pa;
    const DP5 t = get_state(S.G + j);
    const int x = c.p2 * ((int)(S.list[j].x >> 24) - pa);
    const int far_ = min(v.ee + t.ee, v.e2 + t.e2) + x;
    const int near_ = __vimin3_s32(v.uu + t.uu, min(v.e0, v.ee) + t.e0, min(v.oe, v.ee) + t.oe);
    return min(near_, far_) + c.p2 * (int)(S.list[nt - 1].x >> 24);
}

constexpr uint32_t BG_PAST = 0xFFFFFFFFu;   // aisle 255: past every aisle

// Optimal length of the tour (nt list entries) plus one pick.
__device__ __forceinline__ int cost_with_pick(const BgShared& S, const DPConst& c, int nt, uint32_t k) {
    const int a = (int)(k >> 8);
    int j = S.first[a];
    DP5 v = get_state(S.F + j);
    const int pa = j > 0 ? (int)(S.list[j - 1].x >> 24) : 0;
    int lo = (int)(k & 0xFFu), hi = lo, gap = 0;
    if (j < nt) {
        const uint2 r = S.list[j];
        if ((int)(r.x >> 24) == a) {
            add_pick(r, (int)(k & 0xFFu), lo, hi, gap);
            ++j;
        }
    }
    dp_aisle_rel(v, c, a - pa, lo, hi, gap);
    return close_with(S, c, v, a, j, nt);
}

// Optimal length of the tour (nt list entries) plus the order of lines
// [io, le), sorted in S.key; an order of no lines leaves the tour's length.
__device__ __forceinline__ int cost_with(const BgShared& S, const DPConst& c, int nt, int io, int le) {
    if (io >= le) return nt > 0 ? close_with(S, c, get_state(S.F + nt), (int)(S.list[nt - 1].x >> 24), nt, nt) : 0;
    uint32_t k = S.key[io];
    int j = S.first[k >> 8];
    DP5 v = get_state(S.F + j);
    int pa = j > 0 ? (int)(S.list[j - 1].x >> 24) : 0;
    uint2 r = j < nt ? S.list[j] : make_uint2(BG_PAST, 0u);
    for (bool more = true; more;) {
        const int ao = (int)(k >> 8), at = (int)(r.x >> 24);
        int a = at, lo = (int)(r.x >> 16) & 0xFF, hi = (int)(r.x >> 8) & 0xFF, gap = (int)(r.x & 0xFFu);
        if (ao <= at) {
            // the order's picks of this aisle, with the tour's if it has any
            a = ao;
            const int i0 = io, k0 = (int)(k & 0xFFu);
            int prev = k0, inner = 0;
            do {
                inner = max(inner, (int)(k & 0xFFu) - prev);
                prev = (int)(k & 0xFFu);
                ++io;
                more = io < le;
                if (more) k = S.key[io];
            } while (more && (int)(k >> 8) == ao);
            if (at != ao) {
                lo = k0;
                hi = prev;
                gap = inner;
            } else if (k0 == prev) {
                add_pick(r, k0, lo, hi, gap);
            } else {
                uint32_t m[8];
                load_mask(S.mask + 8 * ao, m);
                for (int i = i0; i < io; ++i) {
                    const uint32_t x = S.key[i] & 0xFFu, bit = 1u << (x & 31u);
#pragma unroll
                    for (int w = 0; w < 8; ++w) m[w] |= (x >> 5) == (uint32_t)w ? bit : 0u;
                }
                mask_stats(m, lo, hi, gap);
            }
        }
        if (at == a) {
            ++j;
            r = j < nt ? S.list[j] : make_uint2(BG_PAST, 0u);
        }
        dp_aisle_rel(v, c, a - pa, lo, hi, gap);
        pa = a;
    }
    return close_with(S, c, v, pa, j, nt);
}

__device__ __forceinline__ unsigned long long warp_min_u64(unsigned long long x) {
    const unsigned hi = (unsigned)(x >> 32), mh = __reduce_min_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_min_sync(0xffffffffu, hi == mh ? (unsigned)x : 0xffffffffu);
    return ((unsigned long long)mh << 32) | ml;
}

// orders by tour length, ties by id
__device__ __forceinline__ unsigned long long bg_rank(int length, int o) {
    return ((unsigned long long)(uint32_t)length << 32) | (uint32_t)o;
}

// One warp adds the order of lines [lb, le) to the tour: mask bits, and the
// list with its records (32 lines at a time; new aisles merged into the list
// by their rank among the old and the new ones).  Returns the list's length.
__device__ int insert_order(const BgShared& S, int nt, int lb, int le, int lane) {
    for (int l0 = lb; l0 < le; l0 += 32) {
        const int l = l0 + lane;
        const bool in = l < le;
        const uint32_t k = in ? S.key[l] : 0xFFFFu;
        const int ai = (int)(k >> 8);
        const int before = __shfl_up_sync(0xffffffffu, ai, 1);
        const bool head = in && (lane == 0 || before != ai);   // first line of its aisle here
        int at = 0, hi = nt;                                   // list position of the aisle
        if (l0 == lb) {
            if (head && nt > 0) at = S.first[ai];
        } else if (head)
            while (at < hi) {
                const int mid = (at + hi) >> 1;
                if ((int)(S.list[mid].x >> 24) < ai) at = mid + 1; else hi = mid;
            }
        const bool fresh = head && (at == nt || (int)(S.list[at].x >> 24) != ai);
        if (in) atomicOr(&S.mask[8 * ai + ((k & 0xFFu) >> 5)], 1u << (k & 31u));
        const unsigned fm = __ballot_sync(0xffffffffu, fresh);
        if (fm) {
            // old entries move right by the new aisles below them, last ones first
            for (int b = (nt - 1) & ~31; b >= 0; b -= 32) {
                const uint2 e = b + lane < nt ? S.list[b + lane] : make_uint2(0u, 0u);
                int shift = 0;
                for (unsigned f = fm; f; f &= f - 1) shift += __shfl_sync(0xffffffffu, ai, __ffs(f) - 1) < (int)(e.x >> 24);
                __syncwarp();
                if (b + lane < nt) S.list[b + lane + shift] = e;
                __syncwarp();
            }
            nt += __popc(fm);
        }
        at += __popc(fm & ((1u << lane) - 1u));   // keys are sorted: the new aisles of lower lanes lie below
        __syncwarp();
        // records of the aisles with new picks, four at a time, a lane per mask word
        for (unsigned hm = __ballot_sync(0xffffffffu, head); hm;) {
            int src = -1;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (u == (lane >> 3)) src = __ffs(hm) - 1;
                hm &= hm - 1;
            }
            const int aisle = __shfl_sync(0xffffffffu, ai, src & 31), at_h = __shfl_sync(0xffffffffu, at, src & 31);
            uint32_t b = src >= 0 ? S.mask[8 * aisle + (lane & 7)] : 0u;
            const int base = 32 * (lane & 7);
            // the last pick of the words before this one (a running maximum)
            int upto = b ? base + 31 - __clz(b) : -1;
#pragma unroll
            for (int d = 1; d < 8; d <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, upto, d, 8);
                if ((lane & 7) >= d) upto = max(upto, x);
            }
            int prev = __shfl_up_sync(0xffffffffu, upto, 1, 8);
            if ((lane & 7) == 0) prev = -1;
            const int hi_pick = __shfl_sync(0xffffffffu, upto, 7, 8);
            int lo_pick = b && prev < 0 ? base + __ffs(b) - 1 : 0x7fffffff;
            int g1 = 0, from = 0, g2 = 0;   // largest gap, where it begins, the largest of the others
            for (; b; b &= b - 1) {
                const int k = base + __ffs(b) - 1;
                if (prev >= 0) {
                    const int d = k - prev;
                    if (d > g1) {
                        g2 = g1;
                        g1 = d;
                        from = prev;
                    } else {
                        g2 = max(g2, d);
                    }
                }
                prev = k;
            }
            __syncwarp();
#pragma unroll
            for (int d = 1; d < 8; d <<= 1) {
                const int h1 = __shfl_xor_sync(0xffffffffu, g1, d, 8), hf = __shfl_xor_sync(0xffffffffu, from, d, 8);
                const int h2 = __shfl_xor_sync(0xffffffffu, g2, d, 8);
                lo_pick = min(lo_pick, __shfl_xor_sync(0xffffffffu, lo_pick, d, 8));
                g2 = __vimax3_s32(g2, h2, min(g1, h1));
                from = h1 > g1 ? hf : from;
                g1 = max(g1, h1);
            }
            if (src >= 0 && (lane & 7) == 0)
                S.list[at_h] = make_uint2(((uint32_t)aisle << 24) | ((uint32_t)lo_pick << 16) |
                                              ((uint32_t)hi_pick << 8) | (uint32_t)g1,
                                          ((uint32_t)from << 8) | (uint32_t)g2);
        }
        __syncwarp();
    }
    return nt;
}

__global__ void __launch_bounds__(BG_THREADS) k_batch_grow(BatchGrowArgs B) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long red[2 * (BG_THREADS / 32)], s_win;
    __shared__ uint16_t s_queue[BG_QUEUE];
    __shared__ int s_nt, s_nq, s_at, s_most;
    const EvalArgs& a = B.a;
    const Geo& g = a.g;
    const DPConst dc = dp_const(g);
    constexpr int T = BG_THREADS, NW = T / 32;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_orders = a.n_orders, n_lines = a.n_lines, A = g.A;
    const int p = blockIdx.x;
    // carve shared memory (sizes match batch_grow_launch_bytes)
    unsigned char* q = smem;
    BgShared S;
    S.F = reinterpret_cast<BgVec*>(q);
    q += sizeof(BgVec) * (size_t)(A + 1);
    S.G = reinterpret_cast<BgVec*>(q);
    q += sizeof(BgVec) * (size_t)A;
    S.mask = reinterpret_cast<uint32_t*>(q);
    q += 32 * (size_t)A;
    S.list = reinterpret_cast<uint2*>(q);
    q += 8 * (size_t)A;
    S.off = reinterpret_cast<int32_t*>(q);
    q += 4 * (size_t)(n_orders + 1);
    S.bound = reinterpret_cast<int32_t*>(q);
    q += 4 * (size_t)n_orders;
    S.first = reinterpret_cast<uint16_t*>(q);
    q += 2 * (size_t)A;
    S.key = reinterpret_cast<uint16_t*>(q);
    q += 2 * (size_t)n_lines;
    S.rem = reinterpret_cast<uint16_t*>(q);
    q += 2 * (size_t)n_orders;
    S.by_len = reinterpret_cast<uint16_t*>(q);

    const int32_t* map = a.slot_map + (int64_t)p * a.slot_stride;
    int32_t* tour_off = B.tour_off + (int64_t)p * (n_orders + 1);
    int32_t* order_seq = B.order_seq + (int64_t)p * n_orders;
    bool bad = false;
    for (int o = tid; o <= n_orders; o += T) S.off[o] = a.order_off[o];
    for (int l = tid; l < n_lines; l += T) {
        const int s = a.line_sku[l];
        const int loc = (unsigned)s < (unsigned)a.n_sku ? map[s] : -1;
        if ((unsigned)loc >= (unsigned)g.n_loc) {
            bad = true;
            S.key[l] = 0;
        } else {
            S.key[l] = (uint16_t)key16_of(loc_key(g, loc));
        }
    }
    for (int i = tid; i < 8 * A; i += T) S.mask[i] = 0u;
    for (int i = tid; i < A; i += T) S.first[i] = 0;
    for (int o = tid; o < n_orders; o += T) {
        S.rem[o] = (uint16_t)o;
        S.by_len[o] = (uint16_t)o;
    }
    if (tid == 0) {
        DP5 v;
        dp_init(v);
        put_state(S.F, v);
        s_most = 0;
    }
    if (__syncthreads_or(bad)) {
        if (tid == 0) {
            flag(a.status, WH_STATUS_BAD_LOC);
            B.n_tours[p] = -1;
        }
        return;
    }
    // each order's keys ascending (aisle, slot), once; the most lines of an order
    for (int o = tid; o < n_orders; o += T) {
        const int lb = S.off[o], le = S.off[o + 1];
        if (le - lb > s_most) atomicMax(&s_most, le - lb);
        for (int i = lb + 1; i < le; ++i) {
            const uint16_t k = S.key[i];
            int j = i;
            while (j > lb && S.key[j - 1] > k) {
                S.key[j] = S.key[j - 1];
                --j;
            }
            S.key[j] = k;
        }
    }
    __syncthreads();
    // every order's tour alone (the tour is empty, rem holds every order at
    // its own id), and the orders by it, longest first, ties by id: a bitonic
    // network of ascending merges whose entries past n_orders stand for +inf
    for (int o = tid; o < n_orders; o += T) S.bound[o] = cost_with(S, dc, 0, S.off[o], S.off[o + 1]);
    __syncthreads();
    auto exchange = [&](int x, int y) {   // x < y
        if (y >= n_orders) return;
        const int ox = S.by_len[x], oy = S.by_len[y];
        const int lx = S.bound[ox], ly = S.bound[oy];
        if (ly > lx || (ly == lx && oy < ox)) {
            S.by_len[x] = (uint16_t)oy;
            S.by_len[y] = (uint16_t)ox;
        }
    };
    for (int k = 2; k < 2 * n_orders; k <<= 1) {
        for (int x = tid; x < n_orders; x += T)
            if ((x & (k >> 1)) == 0) exchange(x, x ^ (k - 1));
        __syncthreads();
        for (int j = k >> 2; j > 0; j >>= 1) {
            for (int x = tid; x < n_orders; x += T)
                if ((x & j) == 0) exchange(x, x | j);
            __syncthreads();
        }
    }

    int done = 0, tours = 0, head = 0, nrem = n_orders;
    if (tid == 0) tour_off[0] = 0;
    while (done < n_orders) {
        // seed: the longest order alone that is left
        while (S.off[S.by_len[head]] < 0) ++head;
        int o_add = S.by_len[head++];
        for (int i = tid; i < nrem; i += T)
            if ((int)S.rem[i] == o_add) s_at = i;
        __syncthreads();
        bool mine = tid == T - 1;   // the thread that takes o_add off the list
        int at = s_at, nt = 0;
        int count = 0, lines = 0;
        for (;;) {
            // o_add joins the tour (warp 0) and leaves the unassigned list
            // (its finder; the last entry takes its place)
            const int lb = S.off[o_add] & BG_OFF_MASK, le = S.off[o_add + 1] & BG_OFF_MASK;
            if (warp == 0) {
                const int n = insert_order(S, nt, lb, le, lane);
                if (lane == 0) {
                    s_nt = n;
                    order_seq[done] = o_add;
                }
            }
            --nrem;
            if (mine) {
                S.rem[at] = S.rem[nrem];
                S.bound[at] = S.bound[nrem];
            }
            ++done;
            ++count;
            lines += le - lb;
            __syncthreads();
            if (mine) S.off[o_add] |= ~BG_OFF_MASK;
            if (B.max_orders > 0 && count >= B.max_orders) break;
            // the DP before and to go from every list entry, one warp each,
            // and the list position of every aisle
            nt = s_nt;
            if (tid == 0) {
                DP5 v;
                dp_init(v);
                int pa = 0;
                uint32_t r = nt > 0 ? S.list[0].x : 0u;
                for (int j = 0; j < nt; ++j) {
                    const uint32_t rn = j + 1 < nt ? S.list[j + 1].x : 0u;
                    const int ai = (int)(r >> 24);
                    dp_aisle_rel(v, dc, ai - pa, (int)(r >> 16) & 0xFF, (int)(r >> 8) & 0xFF, (int)(r & 0xFFu));
                    put_state(S.F + j + 1, v);
                    pa = ai;
                    r = rn;
                }
            } else if (tid == 32) {
                DP5 g5;   // past the last aisle: dp_final's classes
                g5.uu = g5.e2 = INF;
                g5.e0 = g5.oe = g5.ee = 0;
                uint32_t r = nt > 0 ? S.list[nt - 1].x : 0u;
                for (int j = nt - 1; j >= 0; --j) {
                    const uint32_t rp = j > 0 ? S.list[j - 1].x : 0u;
                    const DP5 t = back_step(g5, dc, (int)(r >> 16) & 0xFF, (int)(r >> 8) & 0xFF, (int)(r & 0xFFu));
                    put_state(S.G + j, t);
                    g5 = back_cross(t, dc, (int)(r >> 24) - (int)(rp >> 24));
                    r = rp;
                }
            } else if (warp >= 2) {
                for (int ai = tid - 64; ai < A; ai += T - 64) {
                    int x = 0, y = nt;
                    while (x < y) {
                        const int mid = (x + y) >> 1;
                        if ((int)(S.list[mid].x >> 24) < ai) x = mid + 1; else y = mid;
                    }
                    S.first[ai] = (uint16_t)x;
                }
            }
            __syncthreads();
            // grow: the fitting order that leaves the tour shortest
            auto fits = [&](int o) {
                return B.max_lines <= 0 || lines + (S.off[o + 1] & BG_OFF_MASK) - S.off[o] <= B.max_lines;
            };
            unsigned long long best = ~0ull;
            at = -1;
            auto score = [&](int i) {   // the unassigned order at position i, which fits
                const int o = S.rem[i];
                const int c = cost_with(S, dc, nt, S.off[o], S.off[o + 1] & BG_OFF_MASK);
                S.bound[i] = c;
                const unsigned long long v = bg_rank(c, o);
                if (v < best) {
                    best = v;
                    at = i;
                }
            };
            // no order makes the tour shorter than it is
            const int cur = cost_with(S, dc, nt, 0, 0);
            if (count == 1) {
                // the tour's first growth step: bounds from the order's first,
                // middle and last line
                for (int i = tid; i < nrem; i += T) {
                    const int o = S.rem[i], lb = S.off[o], le = S.off[o + 1] & BG_OFF_MASK;
                    int v = 0;
                    if (lb < le) {
                        v = cost_with_pick(S, dc, nt, S.key[lb]);
                        if (lb + 2 < le) v = max(v, cost_with_pick(S, dc, nt, S.key[(lb + le) >> 1]));
                        if (lb + 1 < le) v = max(v, cost_with_pick(S, dc, nt, S.key[le - 1]));
                    }
                    S.bound[i] = v;
                }
            }
            // the two lowest bounds: the lowest is scored, and where the score
            // lies above the second, every order bounded below the score is
            unsigned long long low = ~0ull, next = ~0ull;
            int il = -1;
            const bool all_fit = B.max_lines <= 0 || lines + s_most <= B.max_lines;
            for (int i = tid; i < nrem; i += T) {
                const int o = S.rem[i];
                const unsigned long long v = bg_rank(max(S.bound[i], cur), o);
                if (v >= next || !(all_fit || fits(o))) continue;
                if (v < low) {
                    next = low;
                    low = v;
                    il = i;
                } else {
                    next = v;
                }
            }
            {
                const unsigned long long m1 = warp_min_u64(low), m2 = warp_min_u64(low == m1 ? next : low);
                if (lane == 0) {
                    red[warp] = m1;
                    red[NW + warp] = m2;
                }
            }
            if (tid == 0) s_nq = 0;
            __syncthreads();
            {
                const unsigned long long x = lane < NW ? red[lane] : ~0ull, y = lane < NW ? red[NW + lane] : ~0ull;
                const unsigned long long m1 = warp_min_u64(x);
                next = warp_min_u64(x == m1 ? y : x);
                if (m1 == ~0ull) break;   // nothing fits
                if (low == m1) {
                    score(il);
                    s_win = best;
                }
            }
            __syncthreads();
            unsigned long long win = s_win;
            if (next < win) {
                for (int i0 = warp * 32; i0 < nrem; i0 += T) {
                    const int i = i0 + lane;
                    bool take = false;
                    if (i < nrem) {
                        const int o = S.rem[i];
                        take = bg_rank(max(S.bound[i], cur), o) < win && (all_fit || fits(o));   // (not the one scored)
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, take);
                    if (!m) continue;
                    int slot = 0;
                    if (lane == 0) slot = atomicAdd(&s_nq, __popc(m));
                    slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(m & ((1u << lane) - 1u));
                    if (take) {
                        if (slot < BG_QUEUE) s_queue[slot] = (uint16_t)i;
                        else score(i);
                    }
                }
                __syncthreads();
                const int nq = min(s_nq, BG_QUEUE);
                // neighbouring entries to different warps: few entries run at a lane each
                for (int x = lane * NW + warp; x < nq; x += T) score(s_queue[x]);
                const unsigned long long wb = warp_min_u64(best);
                if (lane == 0) red[warp] = wb;
                __syncthreads();
                win = warp_min_u64(lane < NW ? red[lane] : ~0ull);
            }
            o_add = (int)(win & 0xFFFFFFFFull);
            mine = best == win;
        }
        // close the tour: clear its masks
        ++tours;
        if (tid == 0) tour_off[tours] = done;
        const int na = s_nt;
        for (int i = tid; i < na * 8; i += T) S.mask[8 * (S.list[i >> 3].x >> 24) + (i & 7)] = 0u;
        __syncthreads();
    }
    if (tid == 0) B.n_tours[p] = tours;
}

// shared memory of a launch: the order book, the unassigned list, the bounds,
// and per aisle a depth mask, a list entry, its DP state and its cost to go
size_t batch_grow_launch_bytes(int n_orders, int n_lines, int A) {
    return sizeof(BgVec) * (2 * (size_t)A + 1) + 42 * (size_t)A + 12 * (size_t)n_orders + 4 + 2 * (size_t)n_lines + 16;
}

}  // namespace

// the documented size that a call is accepted by (12 B per order, 2 B per
// line, 38 B per aisle); a launch adds 68 B per aisle to it
size_t batch_grow_smem_bytes(int n_orders, int n_lines, int A) {
    return 4 * (size_t)(n_orders + 1) + 4 * (size_t)n_orders + 32 * (size_t)A + 4 * (size_t)A + 2 * (size_t)n_lines +
           2 * (size_t)A + 4 * (size_t)n_orders + 16;
}

cudaError_t launch_batch_grow(const BatchGrowArgs& B, int n_maps, cudaStream_t s) {
    if (n_maps <= 0) return cudaSuccess;
    const size_t smem = batch_grow_launch_bytes(B.a.n_orders, B.a.n_lines, B.a.g.A);
    cudaError_t e = cudaFuncSetAttribute(k_batch_grow, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_batch_grow<<<n_maps, BG_THREADS, smem, s>>>(B);
    return cudaGetLastError();
}

}  // namespace wh
