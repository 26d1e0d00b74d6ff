// K-means slotting on the GPU (subproblem 3 of Sec. 5: products placed by
// picking frequency, an unsupervised K-means classification deciding which
// are stored together; subroutine 4 then scores the placement with the
// evaluator).  All arithmetic is integer, so the result is exact:
//   features  co_s = sum over every line of s of (T_o - r_s), T_o the sum of
//             the sign rows of the order's lines (= the co-occurrence row of
//             s projected on the sign directions); x_s = trunc(co_s * 1024 /
//             isqrt(|co_s|^2)), last coordinate freq_weight * bitlen(freq_s);
//   seeding   the given SKUs, or K-means++ (Arthur & Vassilvitskii 2007) from
//             the caller's draws: next seed = first SKU whose running sum of
//             D^2 exceeds u mod sum D^2;
//   Lloyd     nearest centroid (ties: lowest), centroid = member mean rounded
//             to the nearest integer (halves up), empty clusters kept;
//   zones     clusters by picks (heavier first), SKUs by picks inside, the
//             r-th SKU at the r-th location in aisle-major order.
// Distances fit int32: |x_j| <= 1024 for the 31 sketch coordinates and
// 0 <= x_31 <= 32 * 256, so a squared distance is below 31 * 2048^2 + 8192^2
// < 2^31; centroids are means of rows and obey the same bounds.
//
// A SKU that no order asks for has an all-zero row, and most of a catalogue is
// such SKUs (45,000 of 50,000 at paper scale): they share one distance to
// every seed and centroid and one nearest cluster, so seeding and Lloyd rounds
// run over the list of ordered SKUs and count the others.
//
// What bounds it: latency.  Paper scale (50,000 SKUs, k = 256, 20 rounds):
// 1.01 ms a call, against 4.79 ms with a launch per seed over all SKUs (2.5 ms),
// Lloyd rounds over all SKUs (1.3 ms) and the zones' ranks found by counting
// pairs (0.65 ms): seeding 0.55 ms, Lloyd rounds 0.3, features and zones 0.1.
#include <cooperative_groups.h>

#include "tour_core.cuh"

namespace wh {

namespace {

constexpr int KM_T = 256;

__device__ __forceinline__ void load_row(const int32_t* p, int32_t (&v)[KM_DIM]) {
    const int4* q = reinterpret_cast<const int4*>(p);
#pragma unroll
    for (int i = 0; i < KM_DIM / 4; ++i) {
        const int4 w = q[i];
        v[4 * i] = w.x;
        v[4 * i + 1] = w.y;
        v[4 * i + 2] = w.z;
        v[4 * i + 3] = w.w;
    }
}

__device__ __forceinline__ void load_signs(const int8_t* p, int32_t (&r)[KM_DIM]) {
    const int4* q = reinterpret_cast<const int4*>(p);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int4 w = q[i];
        const int32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) r[16 * i + 4 * b + c] = (int32_t)(int8_t)((uint32_t)ws[b] >> (8 * c));
    }
}

__device__ __forceinline__ int32_t sqdist32(const int32_t (&x)[KM_DIM], const int32_t* c) {
    int32_t d = 0;
#pragma unroll
    for (int j = 0; j < KM_DIM; ++j) {
        const int32_t e = x[j] - c[j];
        d += e * e;
    }
    return d;
}

__device__ __forceinline__ long long floor_div(long long a, long long b) {   // b > 0
    long long q = a / b;
    if ((a % b) != 0 && a < 0) --q;
    return q;
}

// features, step 1: co-occurrence sketch and pick counts (integer atomics,
// so the sums do not depend on the order of the updates)
__global__ void k_km_cooc(KmArgs A) {
    for (int o = blockIdx.x * blockDim.x + threadIdx.x; o < A.n_orders; o += gridDim.x * blockDim.x) {
        const int lb = A.order_off[o], le = A.order_off[o + 1];
        if (lb < 0 || le < lb || le > A.n_lines) {
            flag(A.status, WH_STATUS_BAD_OFFSET);
            continue;
        }
        int32_t T[KM_DIM];
#pragma unroll
        for (int j = 0; j < KM_DIM; ++j) T[j] = 0;
        bool bad = false;
        for (int l = lb; l < le; ++l) {
            const int s = A.line_sku[l];
            if ((unsigned)s >= (unsigned)A.n_sku) {
                bad = true;
                continue;
            }
            int32_t r[KM_DIM];
            load_signs(A.signs + (int64_t)s * KM_DIM, r);
#pragma unroll
            for (int j = 0; j < KM_SKETCH; ++j) T[j] += r[j];
        }
        if (bad) flag(A.status, WH_STATUS_BAD_SKU);
        for (int l = lb; l < le; ++l) {
            const int s = A.line_sku[l];
            if ((unsigned)s >= (unsigned)A.n_sku) continue;
            int32_t r[KM_DIM];
            load_signs(A.signs + (int64_t)s * KM_DIM, r);
            atomicAdd(&A.freq[s], 1);
            unsigned long long* co = reinterpret_cast<unsigned long long*>(A.co + (int64_t)s * KM_DIM);
#pragma unroll
            for (int j = 0; j < KM_SKETCH; ++j) {
                const int32_t v = T[j] - r[j];
                if (v != 0) atomicAdd(co + j, (unsigned long long)(long long)v);
            }
        }
    }
}

__device__ __forceinline__ long long isqrt_ll(long long v) {
    long long r = (long long)sqrt((double)v);
    while (r > 0 && r * r > v) --r;
    while ((r + 1) * (r + 1) <= v) ++r;
    return r;
}

// features, step 2: the blocks' ordered SKUs and the largest pick count; a
// SKU never ordered has the zero row
__global__ void __launch_bounds__(KM_T) k_km_count(KmArgs A) {
    const int s = blockIdx.x * KM_T + threadIdx.x;
    const int f = s < A.n_sku ? A.freq[s] : 0;
    const int n_act = __syncthreads_count(f > 0);
    const unsigned fm = __reduce_max_sync(0xffffffffu, (unsigned)f);
    if (threadIdx.x == 0) A.bcount[blockIdx.x] = n_act;
    if ((threadIdx.x & 31) == 0 && fm > 0) atomicMax(A.max_freq, fm);
    if (s < A.n_sku && f == 0) {
        int4* out = reinterpret_cast<int4*>(A.x + (int64_t)s * KM_DIM);
#pragma unroll
        for (int i = 0; i < KM_DIM / 4; ++i) out[i] = make_int4(0, 0, 0, 0);
    }
}

// features, step 3, one ordered SKU per warp, a coordinate per lane: normalise
// the sketch, append the frequency coordinate
__global__ void __launch_bounds__(KM_T) k_km_features(KmArgs A) {
    const int na = *A.n_active, lane = threadIdx.x & 31;
    for (int i = (int)((blockIdx.x * KM_T + threadIdx.x) >> 5); i < na; i += (int)(gridDim.x * (KM_T / 32))) {
        const int s = A.active[i];
        const long long c = lane < KM_SKETCH ? A.co[(int64_t)s * KM_DIM + lane] : 0;
        long long nn = c * c;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, d);
        const long long n = isqrt_ll(nn);
        int32_t x = n > 0 ? (int32_t)(c * KM_SCALE / n) : 0;
        if (lane == KM_SKETCH) x = A.fw * (32 - __clz(A.freq[s]));
        A.x[(int64_t)s * KM_DIM + lane] = x;
    }
}

// the ordered SKUs' ids, ascending: every block adds up the counts of the
// blocks before it and writes its own at that place
__global__ void __launch_bounds__(KM_T) k_km_compact(KmArgs A) {
    __shared__ int s_before, s_warp[KM_T / 32];
    if (threadIdx.x == 0) s_before = 0;
    __syncthreads();
    int part = 0;
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += KM_T) part += A.bcount[b];
    part = (int)__reduce_add_sync(0xffffffffu, (unsigned)part);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0 && part) atomicAdd(&s_before, part);
    const int s = blockIdx.x * KM_T + threadIdx.x;
    const bool act = s < A.n_sku && A.freq[s] > 0;
    const unsigned m = __ballot_sync(0xffffffffu, act);
    if (lane == 0) s_warp[w] = __popc(m);
    __syncthreads();
    int at = s_before + __popc(m & ((1u << lane) - 1u));
    for (int i = 0; i < w; ++i) at += s_warp[i];
    if (act) A.active[at] = s;
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == KM_T - 1) *A.n_active = at + (act ? 1 : 0);
}

// seeds given: copy them (range-checked)
__global__ void k_km_seed_copy(KmArgs A) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= A.k) return;
    int s = A.init[c];
    if ((unsigned)s >= (unsigned)A.n_sku) {
        flag(A.status, WH_STATUS_BAD_SKU);
        s = 0;
    }
    A.seeds[c] = s;
}

__global__ void k_km_pp_first(KmArgs A) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        A.seeds[0] = (int32_t)(A.u[0] % (unsigned long long)A.n_sku);
        *A.done = 0u;
    }
}

__device__ __forceinline__ long long block_sum_ll(long long v, long long* red) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) red[w] = v;
    __syncthreads();
    long long t = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += red[i];
    return t;
}

// inclusive block scan of int64 values
__device__ __forceinline__ long long block_scan_ll(long long v, long long* red) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    long long x = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    __syncthreads();
    if (lane == 31) red[w] = x;
    __syncthreads();
    long long before = 0;
    for (int i = 0; i < w; ++i) before += red[i];
    return before + x;
}

// K-means++ round c >= 1: fold seed c-1 into D, then the last block to finish
// draws seed c from the running sums of D (in SKU order)
__global__ void __launch_bounds__(KM_T) k_km_pp_round(KmArgs A, int c) {
    __shared__ long long red[KM_T / 32];
    __shared__ bool last;
    __shared__ long long s_target, s_before;
    __shared__ int s_block, s_pick;
    const int s = blockIdx.x * KM_T + threadIdx.x;
    const int ctr = A.seeds[c - 1];
    long long dm = 0;
    if (s < A.n_sku) {
        int32_t x[KM_DIM], y[KM_DIM];
        load_row(A.x + (int64_t)s * KM_DIM, x);
        load_row(A.x + (int64_t)ctr * KM_DIM, y);
        const long long d = sqdist32(x, y);
        dm = min(A.dmin[s], d);
        A.dmin[s] = dm;
    }
    const long long bs = block_sum_ll(dm, red);
    if (threadIdx.x == 0) {
        A.bsum[blockIdx.x] = bs;
        __threadfence();
        const unsigned t = atomicAdd(A.done, 1u);
        last = t == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the block holding the draw: every thread sums a contiguous run of the
    // block sums, a block scan of the runs gives each run's start, and the
    // thread whose run covers the target finds the block inside it
    const int nb = (int)gridDim.x, per = (nb + KM_T - 1) / KM_T;
    const int b0 = min((int)threadIdx.x * per, nb), b1 = min(b0 + per, nb);
    long long part = 0;
    for (int b = b0; b < b1; ++b) part += __ldcg(A.bsum + b);
    const long long incl = block_scan_ll(part, red);
    __shared__ long long s_total;
    if (threadIdx.x == KM_T - 1) s_total = incl;
    if (threadIdx.x == 0) s_pick = -1;
    __syncthreads();
    const long long tot = s_total;
    if (tot == 0) {
        if (threadIdx.x == 0) s_pick = (int)(A.u[c] % (unsigned long long)A.n_sku);
    } else {
        const long long target = (long long)(A.u[c] % (unsigned long long)tot);
        const long long excl = incl - part;
        if (part > 0 && excl <= target && target < incl) {
            long long run = excl;
            int b = b0;
            for (; b < b1; ++b) {
                const long long v = __ldcg(A.bsum + b);
                if (run + v > target) break;
                run += v;
            }
            s_block = b;
            s_before = run;
            s_target = target;
        }
    }
    __syncthreads();
    if (s_pick < 0) {
        const int q = s_block * KM_T + threadIdx.x;
        const long long v = q < A.n_sku ? __ldcg(A.dmin + q) : 0;
        const long long incl = s_before + block_scan_ll(v, red);
        // the first SKU whose running sum exceeds the target
        const bool hit = q < A.n_sku && incl > s_target && incl - v <= s_target;
        if (hit) s_pick = q;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        A.seeds[c] = s_pick >= 0 ? s_pick : A.n_sku - 1;
        *A.done = 0u;
    }
}

// K-means++ seeding in one launch by a cluster of eight CTAs, each holding an
// eighth of the ordered SKUs (a contiguous run of ids) in shared memory as
// 16-bit rows with their D^2; a SKU never ordered has the zero row and the one
// D^2 of all of them, so the runs between ordered SKUs enter the running sums
// by their length.  A round folds the last seed into D^2, scans the sums
// inside each CTA, exchanges the CTAs' totals, and the CTA that the draw falls
// into finds the SKU and hands its row to all eight.  Two cluster barriers a
// round (2.2 us a round; a launch per seed took 9.8; 1,024 threads a CTA 2.6).  Used where the
// ordered SKUs fit (at most min(SKUs, order lines) of them); the launch per
// seed above serves larger books.
constexpr int PP_CTAS = 8;
constexpr int PP_T = 512;
constexpr int PP_ROW_BYTES = 64 + 3 * 4;

__global__ void __cluster_dims__(PP_CTAS, 1, 1) __launch_bounds__(PP_T, 1) k_km_pp_cluster(KmArgs A, int cap) {
    namespace cg = cooperative_groups;
    extern __shared__ __align__(16) unsigned char pp_smem[];
    __shared__ long long s_tot[2][PP_CTAS], s_warp[PP_T / 32], s_target;
    __shared__ __align__(16) int32_t s_y[2][KM_DIM];
    __shared__ int s_pick, s_row, s_owner;
    uint4* xs = reinterpret_cast<uint4*>(pp_smem);                    // [4][cap]: eight coordinates a piece
    int32_t* norm = reinterpret_cast<int32_t*>(xs + 4 * (size_t)cap);  // [cap] |x|^2
    int32_t* dmin = norm + cap;                                        // [cap]
    int32_t* ids = dmin + cap;                                         // [cap]
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int na = *A.n_active;
    const int i0 = (int)((int64_t)na * rank / PP_CTAS), cnt = (int)((int64_t)na * (rank + 1) / PP_CTAS) - i0;
    // this CTA's run of SKU ids [r0, r1): from its first ordered SKU (CTA 0:
    // from 0) to the next CTA's
    const int r0 = rank == 0 ? 0 : i0 < na ? A.active[i0] : A.n_sku;
    const int r1 = rank == PP_CTAS - 1 || i0 + cnt >= na ? A.n_sku : A.active[i0 + cnt];
    for (int r = tid; r < cnt; r += PP_T) {
        const int s = A.active[i0 + r];
        int32_t x[KM_DIM];
        load_row(A.x + (int64_t)s * KM_DIM, x);
        int32_t nn = 0;
#pragma unroll
        for (int j = 0; j < KM_DIM; ++j) nn += x[j] * x[j];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint32_t v[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) v[h] = ((uint32_t)x[8 * q + 2 * h] & 0xFFFFu) | ((uint32_t)x[8 * q + 2 * h + 1] << 16);
            xs[(size_t)q * cap + r] = make_uint4(v[0], v[1], v[2], v[3]);
        }
        norm[r] = nn;
        dmin[r] = 0x7fffffff;
        ids[r] = s;
    }
    const int s0 = (int)(A.u[0] % (unsigned long long)A.n_sku);
    if (rank == 0 && tid == 0) A.seeds[0] = s0;
    if (tid < KM_DIM) s_y[0][tid] = A.x[(int64_t)s0 * KM_DIM + tid];
    cl.sync();   // (also: every CTA has started before another writes into its shared memory)
    const int per = (cnt + PP_T - 1) / PP_T;
    const int b0 = min(tid * per, cnt), b1 = min(b0 + per, cnt);
    int32_t dz = 0x7fffffff;   // D^2 of every SKU that is never ordered
    for (int c = 1; c < A.k; ++c) {
        const int par = c & 1;
        const int32_t* y = s_y[par ^ 1];
        const unsigned long long u = A.u[c];
        int32_t yn = 0;
#pragma unroll
        for (int j = 0; j < KM_DIM; ++j) yn += y[j] * y[j];
        dz = min(dz, yn);
        int prev = b0 > 0 ? ids[b0 - 1] + 1 : r0;
        long long part = 0;
        for (int r = b0; r < b1; ++r) {
            int32_t dot = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 v = xs[(size_t)q * cap + r];
                const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    dot += (int32_t)(int16_t)vv[h] * y[8 * q + 2 * h] + ((int32_t)vv[h] >> 16) * y[8 * q + 2 * h + 1];
            }
            const int32_t d = min(dmin[r], norm[r] + yn - 2 * dot);
            dmin[r] = d;
            const int s = ids[r];
            part += (long long)(s - prev) * dz + d;
            prev = s + 1;
        }
        if (tid == PP_T - 1) part += (long long)(r1 - (cnt > 0 ? ids[cnt - 1] + 1 : r0)) * dz;
        // inclusive block scan
        long long incl = part;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const long long v = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += v;
        }
        if (lane == 31) s_warp[w] = incl;
        __syncthreads();
        if (w == 0) {
            const long long own = lane < PP_T / 32 ? s_warp[lane] : 0;
            long long v = own;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const long long t = __shfl_up_sync(0xffffffffu, v, d);
                if (lane >= d) v += t;
            }
            if (lane < PP_T / 32) s_warp[lane] = v - own;
            const long long tot = __shfl_sync(0xffffffffu, v, 31);
            if (lane < PP_CTAS) *cl.map_shared_rank(&s_tot[par][rank], lane) = tot;
        }
        cl.sync();
        if (tid == 0) {
            long long before = 0, total = 0;
            for (int j = 0; j < PP_CTAS; ++j) {
                before += j < rank ? s_tot[par][j] : 0;
                total += s_tot[par][j];
            }
            if (total == 0) {
                // every D^2 is zero: the draw modulo the SKU count
                s_pick = (int)(u % (unsigned long long)A.n_sku);
                s_owner = s_pick >= r0 && s_pick < r1 ? 1 : 0;
                int lo = 0, hi = cnt;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (ids[mid] < s_pick) lo = mid + 1; else hi = mid;
                }
                s_row = lo < cnt && ids[lo] == s_pick ? lo : -1;
            } else {
                const long long target = (long long)(u % (unsigned long long)total) - before;
                s_target = target;
                s_owner = target >= 0 && target < s_tot[par][rank] ? 2 : 0;
            }
        }
        __syncthreads();
        if (s_owner) {
            const long long excl = s_warp[w] + incl - part, target = s_target;
            if (s_owner == 2 && part > 0 && excl <= target && target < excl + part) {
                // the first SKU of this thread's run whose running sum exceeds the target
                long long rem = target - excl;
                int pick = -1, row = -1;
                prev = b0 > 0 ? ids[b0 - 1] + 1 : r0;
                for (int r = b0; r < b1; ++r) {
                    const int s = ids[r];
                    const long long zeros = (long long)(s - prev) * dz;
                    if (rem < zeros) break;
                    rem -= zeros;
                    prev = s + 1;
                    if (rem < dmin[r]) {
                        pick = s;
                        row = r;
                        break;
                    }
                    rem -= dmin[r];
                }
                s_pick = row >= 0 ? pick : prev + (int)(rem / dz);
                s_row = row;
            }
            __syncthreads();
            if (w == 0) {
                const int row = s_row;
                int32_t v = 0;
                if (row >= 0) {
                    const uint32_t* q = reinterpret_cast<const uint32_t*>(&xs[(size_t)(lane >> 3) * cap + row]);
                    const uint32_t pair = q[(lane & 7) >> 1];
                    v = (lane & 1) ? ((int32_t)pair >> 16) : (int32_t)(int16_t)pair;
                }
                for (int j = 0; j < PP_CTAS; ++j) *cl.map_shared_rank(&s_y[par][lane], j) = v;
                if (lane == 0) A.seeds[c] = s_pick;
            }
        }
        cl.sync();
    }
}

__global__ void k_km_gather(KmArgs A) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= A.k * KM_DIM) return;
    const int c = i / KM_DIM, j = i % KM_DIM;
    A.cent[i] = A.x[(int64_t)A.seeds[c] * KM_DIM + j];
}

// |c|^2 - 2 x.c: the squared distance less |x|^2, a constant per row, so the
// nearest centroid and its ties are the same; fits int32 by the same bounds
__device__ __forceinline__ int32_t dist_less_norm(const int32_t (&x)[KM_DIM], const int32_t* c, int32_t cn) {
    int32_t dot = 0;
#pragma unroll
    for (int j = 0; j < KM_DIM; ++j) dot += x[j] * c[j];
    return cn - 2 * dot;
}

// One Lloyd round (mode 0) or the final assignment (mode 1) over the ordered
// SKUs: eight threads a row, each an eighth of the centroids from shared
// memory (rows padded to 36 words: the eight read eight different bank
// groups); the block's member sums meet in shared memory first (one cluster
// can hold most rows, and a row's 32 atomics on it would all meet in one
// line).  Block 0 adds the never-ordered SKUs to their cluster's count; after
// the final assignment the last block to finish (an atomic ticket, no wait)
// ranks the clusters by weight.  15 us a round with the update at paper scale
// (k = 256); 21 before each launch was made beside the tail of the one before
// and blocks without rows left at once; 66 over all SKUs, one thread a row.
constexpr int LL_SUB = 8;
constexpr int LL_ROWS = KM_T / LL_SUB;
constexpr int LL_STRIDE = KM_DIM + 4;

__global__ void __launch_bounds__(KM_T) k_km_lloyd(KmArgs A, int mode) {
    extern __shared__ __align__(16) int32_t sm[];
    __shared__ int s_zero;
    __shared__ bool s_last;
    const int K = A.k, tid = threadIdx.x;
    int32_t* cent = sm;                      // [K][36]
    int32_t* cnorm = cent + K * LL_STRIDE;   // [K] |c|^2
    int32_t* pcnt = cnorm + K;               // [K] the block's members
    int32_t* psum = pcnt + K;                // [K][32] and their sums (mode 0)
    pdl_trigger();
    if (mode == 0)
        for (int i = tid; i < K * KM_DIM; i += KM_T) psum[i] = 0;
    for (int c = tid; c < K; c += KM_T) pcnt[c] = 0;
    pdl_wait();
    const int na = *A.n_active;
    // the grid is sized for the most SKUs that can be ordered
    if (mode == 0 && blockIdx.x > 0 && (int)blockIdx.x * LL_ROWS >= na) return;
    for (int i = tid; i < K * KM_DIM; i += KM_T) cent[(i / KM_DIM) * LL_STRIDE + i % KM_DIM] = A.cent[i];
    __syncthreads();
    for (int c = tid; c < K; c += KM_T) {
        int32_t nn = 0;
#pragma unroll
        for (int j = 0; j < KM_DIM; ++j) nn += cent[c * LL_STRIDE + j] * cent[c * LL_STRIDE + j];
        cnorm[c] = nn;
    }
    __syncthreads();
    if (tid < 32) {
        // the zero row's cluster: the smallest |c|^2, ties to the lowest
        int32_t bd = 0x7fffffff;
        int best = 0x7fffffff;
        for (int c = tid; c < K; c += 32)
            if (cnorm[c] < bd) {
                bd = cnorm[c];
                best = c;
            }
        const int32_t m = __reduce_min_sync(0xffffffffu, bd);
        best = __reduce_min_sync(0xffffffffu, bd == m ? best : 0x7fffffff);
        if (tid == 0) s_zero = best;
    }
    __syncthreads();
    const int sub = tid & (LL_SUB - 1);
    for (int g = blockIdx.x; g * LL_ROWS < na; g += gridDim.x) {
        const int i = g * LL_ROWS + tid / LL_SUB;
        const bool in = i < na;
        const int s = A.active[in ? i : na - 1];
        int32_t x[KM_DIM];
        load_row(A.x + (int64_t)s * KM_DIM, x);
        int best = 0x7fffffff;
        int32_t bd = 0x7fffffff;
        for (int c = sub; c < K; c += LL_SUB) {
            const int32_t d = dist_less_norm(x, cent + c * LL_STRIDE, cnorm[c]);
            if (d < bd || best == 0x7fffffff) {
                bd = d;
                best = c;
            }
        }
#pragma unroll
        for (int d = 1; d < LL_SUB; d <<= 1) {
            const int32_t od = __shfl_xor_sync(0xffffffffu, bd, d);
            const int ob = __shfl_xor_sync(0xffffffffu, best, d);
            if (ob != 0x7fffffff && (best == 0x7fffffff || od < bd || (od == bd && ob < best))) {
                bd = od;
                best = ob;
            }
        }
        if (!in) continue;
        if (mode == 0) {
            // (a block adds up at most 2^16 rows of |x_j| <= 2^13)
#pragma unroll
            for (int j = 0; j < KM_DIM; ++j)
                if ((j >> 2) == sub && x[j] != 0) atomicAdd(&psum[best * KM_DIM + j], x[j]);
        } else if (sub == 0) {
            A.assign[s] = best;
            atomicAdd(reinterpret_cast<unsigned long long*>(A.weight) + best, (unsigned long long)A.freq[s]);
        }
        if (sub == 0) atomicAdd(&pcnt[best], 1);
    }
    __syncthreads();
    if (mode == 0) {
        for (int i = tid; i < K * KM_DIM; i += KM_T)
            if (psum[i]) atomicAdd(reinterpret_cast<unsigned long long*>(A.sum) + i, (unsigned long long)(long long)psum[i]);
        for (int c = tid; c < K; c += KM_T) {
            const int n = pcnt[c] + (blockIdx.x == 0 && c == s_zero ? A.n_sku - na : 0);
            if (n) atomicAdd(&A.cnt[c], n);
        }
        return;
    }
    for (int s = blockIdx.x * KM_T + tid; s < A.n_sku; s += gridDim.x * KM_T)
        if (A.freq[s] == 0) A.assign[s] = s_zero;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(A.done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // cluster ranks (heavier first, ties lowest id)
    long long* wt = reinterpret_cast<long long*>(sm);
    for (int c = tid; c < K; c += KM_T) wt[c] = __ldcg(A.weight + c);
    __syncthreads();
    for (int c = tid; c < K; c += KM_T) {
        int r = 0;
        for (int d = 0; d < K; ++d) r += (wt[d] > wt[c]) || (wt[d] == wt[c] && d < c);
        A.rank[c] = r;
    }
}

// centroids from the member sums and counts, which are cleared for the next
// round (a block holds whole clusters)
__global__ void __launch_bounds__(KM_T) k_km_update(KmArgs A) {
    pdl_trigger();
    pdl_wait();
    const int i = blockIdx.x * KM_T + threadIdx.x;
    const bool in = i < A.k * KM_DIM;
    const long long n = in ? A.cnt[i / KM_DIM] : 0;
    if (n > 0) {
        const long long num = 2 * A.sum[i] + n, den = 2 * n;
        if (num >= -0x7fffffffll && num <= 0x7fffffffll && den <= 0x7fffffffll) {
            int q = (int)num / (int)den;
            if ((int)num % (int)den != 0 && num < 0) --q;
            A.cent[i] = q;
        } else {
            A.cent[i] = (int32_t)floor_div(num, den);
        }
    }
    __syncthreads();
    if (in) A.sum[i] = 0;
    if (in && i % KM_DIM == 0) A.cnt[i / KM_DIM] = 0;
}

// Zones: the SKUs sorted by (cluster rank, picks descending, id) with a stable
// radix sort from id order, eight bits a pass: the pick counts' bytes (as many
// as the largest count has) and then the ranks.  A pass counts the digits of
// every tile of 1,024 SKUs, scans the counts digit by digit, and scatters; the
// last one writes the r-th SKU's location.  54 us at paper scale; finding
// every SKU's rank by counting the smaller keys of its cluster took 680 (a
// cluster of 44,000 never-ordered SKUs).
constexpr int RS_TILE = 1024;

struct RsPass {
    int byte;   // of the pick count; -1: the cluster's rank
    int done;   // passes over lower bytes before this one
};

// false: the byte is zero in every count, the pass leaves the order as it is
__device__ __forceinline__ bool rs_needed(const KmArgs& A, RsPass p) {
    return p.byte <= 0 || (*A.max_freq >> (8 * p.byte)) != 0u;
}

// the order after the passes before p: NULL stands for id order
__device__ __forceinline__ const int32_t* rs_source(const KmArgs& A, RsPass p) {
    int n = p.done;
    while (n > 1 && (*A.max_freq >> (8 * (n - 1))) == 0u) --n;   // passes that ran
    return n == 0 ? nullptr : (n & 1) ? A.order_a : A.order_b;
}

__device__ __forceinline__ int rs_digit(const KmArgs& A, RsPass p, int s) {
    return p.byte < 0 ? A.rank[A.assign[s]] : 255 - ((A.freq[s] >> (8 * p.byte)) & 255);
}

__global__ void __launch_bounds__(RS_TILE) k_km_rs_count(KmArgs A, RsPass p) {
    __shared__ int hist[256];
    if (!rs_needed(A, p)) return;
    const int32_t* src = rs_source(A, p);
    if (threadIdx.x < 256) hist[threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * RS_TILE + threadIdx.x;
    if (i < A.n_sku) atomicAdd(&hist[rs_digit(A, p, src ? src[i] : i)], 1);
    __syncthreads();
    if (threadIdx.x < 256) A.rs_count[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = hist[threadIdx.x];
}

// one block: exclusive scan of the 256 * tiles counts, in place
__global__ void __launch_bounds__(1024) k_km_rs_scan(KmArgs A, RsPass p, int64_t n) {
    __shared__ int s_warp[32];
    if (!rs_needed(A, p)) return;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    int carry = 0;
    for (int64_t base = 0; base < n; base += 4096) {
        const int64_t i = base + 4 * tid;
        int v[4], t = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            v[u] = i + u < n ? A.rs_count[i + u] : 0;
            t += v[u];
        }
        int x = t;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
        __syncthreads();
        if (lane == 31) s_warp[w] = x;
        __syncthreads();
        int y = s_warp[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int z = __shfl_up_sync(0xffffffffu, y, d);
            if (lane >= d) y += z;
        }
        const int below = __shfl_sync(0xffffffffu, y, w > 0 ? w - 1 : 0);
        int run = carry + (w > 0 ? below : 0) + x - t;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (i + u < n) A.rs_count[i + u] = run;
            run += v[u];
        }
        carry += __shfl_sync(0xffffffffu, y, 31);
    }
}

__global__ void __launch_bounds__(RS_TILE) k_km_rs_scatter(KmArgs A, RsPass p) {
    __shared__ uint16_t cnt[RS_TILE / 32][256];   // per warp, then what the warps before it hold
    if (!rs_needed(A, p)) return;
    const int32_t* src = rs_source(A, p);
    int32_t* dst = src == A.order_a ? A.order_b : A.order_a;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int i = tid; i < RS_TILE / 32 * 256; i += RS_TILE) (&cnt[0][0])[i] = 0;
    __syncthreads();
    const int i = blockIdx.x * RS_TILE + tid;
    const bool in = i < A.n_sku;
    const int s = in ? (src ? src[i] : i) : 0;
    const int d = in ? rs_digit(A, p, s) : 256 + lane;
    const unsigned same = __match_any_sync(0xffffffffu, d);
    const int below = __popc(same & ((1u << lane) - 1u));
    if (in && below == 0) cnt[w][d] = (uint16_t)__popc(same);
    __syncthreads();
    if (tid < 256) {
        int run = 0;
#pragma unroll
        for (int v = 0; v < RS_TILE / 32; ++v) {
            const int c = cnt[v][tid];
            cnt[v][tid] = (uint16_t)run;
            run += c;
        }
    }
    __syncthreads();
    if (!in) return;
    const int r = A.rs_count[(int64_t)d * gridDim.x + blockIdx.x] + cnt[w][d] + below;
    if (p.byte >= 0) {
        dst[r] = s;
    } else {
        // the r-th location in aisle-major order
        const int L = A.g.L, aisle = r / (2 * L), q = r % (2 * L);
        A.slot_map[s] = (aisle * 2 + (q & 1)) * L + (q >> 1);
    }
}

}  // namespace

// ordered SKUs a seeding cluster holds
int kmeans_pp_rows() { return (220 * 1024 / PP_ROW_BYTES) * PP_CTAS; }

cudaError_t launch_kmeans(const KmArgs& A, cudaStream_t s) {
    const int n = A.n_sku, K = A.k;
    const int gb = (n + KM_T - 1) / KM_T;
    const int most = n < A.n_lines ? n : A.n_lines;   // ordered SKUs at most
    cudaError_t e;
    // features (the counters and sums that start at zero lie together)
    if ((e = cudaMemsetAsync(A.zeroed, 0, A.zeroed_bytes, s)) != cudaSuccess) return e;
    if (A.n_orders > 0) k_km_cooc<<<(A.n_orders + KM_T - 1) / KM_T, KM_T, 0, s>>>(A);
    k_km_count<<<gb, KM_T, 0, s>>>(A);
    k_km_compact<<<gb, KM_T, 0, s>>>(A);
    const int rows8 = (most + KM_T / 32 - 1) / (KM_T / 32);
    k_km_features<<<rows8 < 1 ? 1 : rows8 < 2048 ? rows8 : 2048, KM_T, 0, s>>>(A);
    // seeds
    if (A.init) {
        k_km_seed_copy<<<(K + KM_T - 1) / KM_T, KM_T, 0, s>>>(A);
    } else if (!A.dmin) {
        const int cap = (most + PP_CTAS - 1) / PP_CTAS + 1;
        const size_t smem = (size_t)PP_ROW_BYTES * cap;
        if ((e = cudaFuncSetAttribute(k_km_pp_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
            cudaSuccess)
            return e;
        k_km_pp_cluster<<<PP_CTAS, PP_T, smem, s>>>(A, cap);
    } else {
        k_km_pp_first<<<1, 32, 0, s>>>(A);
        if ((e = cudaMemsetAsync(A.dmin, 0x7F, sizeof(long long) * (size_t)n, s)) != cudaSuccess) return e;
        for (int c = 1; c < K; ++c) k_km_pp_round<<<gb, KM_T, 0, s>>>(A, c);
    }
    k_km_gather<<<(K * KM_DIM + KM_T - 1) / KM_T, KM_T, 0, s>>>(A);
    // Lloyd rounds, the final assignment and the clusters' ranks
    const size_t smem = sizeof(int32_t) * (size_t)K * (LL_STRIDE + 2 + KM_DIM);
    if ((e = cudaFuncSetAttribute(k_km_lloyd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    int grid = (most + LL_ROWS - 1) / LL_ROWS;
    grid = grid < 1 ? 1 : grid > 1216 ? 1216 : grid;   // up to eight blocks an SM
    for (int it = 0; it < A.iters; ++it) {
        if ((e = launch_dependent(k_km_lloyd, grid, KM_T, smem, s, A, 0)) != cudaSuccess) return e;
        if ((e = launch_dependent(k_km_update, (K * KM_DIM + KM_T - 1) / KM_T, KM_T, 0, s, A)) != cudaSuccess) return e;
    }
    if ((e = launch_dependent(k_km_lloyd, grid, KM_T, smem, s, A, 1)) != cudaSuccess) return e;
    // zones
    const int tiles = (n + RS_TILE - 1) / RS_TILE;
    int passes = 1;
    while (passes < 4 && (A.n_lines >> (8 * passes)) != 0) ++passes;
    for (int q = 0; q <= passes; ++q) {
        const RsPass p{q < passes ? q : -1, q};
        k_km_rs_count<<<tiles, RS_TILE, 0, s>>>(A, p);
        k_km_rs_scan<<<1, 1024, 0, s>>>(A, p, (int64_t)256 * tiles);
        k_km_rs_scatter<<<tiles, RS_TILE, 0, s>>>(A, p);
    }
    return cudaGetLastError();
}

}  // namespace wh
