// Generated exact kNN relation consumed by a neighbour sum (paper Section 4.9, generated kNN).
//
// The paper's kernel scans every source for every query and skips the sort of a tile that cannot
// improve the retained keys.  Here the cell directory of the radius relation orders the search
// instead, which keeps the result exact (keys are compared, never approximated) and removes the
// quadratic scan on inputs of roughly even density:
//
//   knn_cells_kernel  a warp per share of the points in cell order, a cell (a slice of a dense one) at a time.  The points are binned with a cell edge a little above a
//                     search radius h chosen so that a ball of radius h holds about 2k points on
//                     average.  Every point closer than h to a query of the cell lies in the
//                     27-cell stencil, so a query that finds k keys <= h^2 there is finished: no
//                     point outside the stencil can have a smaller key.  The stencil is staged in
//                     shared memory (candidates farther than h from the bounding box of the
//                     cell's points are dropped), one candidate per lane is tested against four
//                     queries, accepted keys are compacted into per-query lists by ballots, and a
//                     list that fills up is cut back to its k smallest keys, which also tightens
//                     that query's acceptance threshold.
//   knn_rings_kernel  one warp per query that found fewer than k keys within h (sparse regions,
//                     tiny inputs): it walks cubic shells of cells outwards and stops when the
//                     k-th key is no larger than the squared distance to the unexplored region, or
//                     when the whole grid has been visited.
//
// Keys are (fp32 squared distance by direct differences in a fixed operation order, source index),
// held as one 64-bit integer (distance bits above the index: squared distances are never negative,
// so their bit patterns order like the values).  The k smallest of a list are found in two steps: a list of
// more than 32 entries is trimmed to at most 32 by a distance that k entries do not exceed (guessed from the
// list's length, counts grow with the cube of the distance, and corrected by counting ballots); then every lane
// counts the entries closer than its own, which is that entry's place in the row.  Equal distances and k > 24 go
// through the general form, a bitonic network of shuffles over 32 keys at a time and merges, which orders
// whole keys.  (131,072 uniform points, k = 16, one feature: 552 warp instructions per query here and 40 in the rings kernel.)
#include "radius_test.cuh"
#include <type_traits>

namespace tiga {

constexpr int KQB = 4;                             // queries per batch (cells kernel)
constexpr int KNN_STAGE_CAP = 192;                 // staged candidates per chunk
constexpr int KNN_QCAP = 96;                       // list entries per query (cells kernel)
constexpr int KNN_QSTRIDE = KNN_QCAP + 2;          // even: entries are read two at a time
constexpr int KNN_TRIM = 32;                       // entries a trimmed list has at most (one per lane)
constexpr int KNN_COUNT_K = 24;                    // largest k that counting serves: a trimmed list has k to KNN_TRIM entries
constexpr int KNN_RING_CAP = 128;                  // list entries of the rings kernel
constexpr int KNN_STAGE_BYTES = (KNN_STAGE_CAP + STAGE_PAD) * 16;
constexpr int KNN_LIST_BYTES = (KQB * KNN_QSTRIDE * 8 + 15) / 16 * 16;
constexpr int KNN_MISC_BYTES = KQB * 16 + KQB * 4 * 2 + 80;     // queries, list lengths, thresholds, range offsets of the stencil
constexpr int KNN_PER_WARP = KNN_STAGE_BYTES + KNN_LIST_BYTES + KNN_MISC_BYTES;
static_assert(KNN_PER_WARP % 16 == 0 && KNN_LIST_BYTES % 16 == 0, "the stage and the queries are accessed as 16-byte vectors");
constexpr int RING_WARPS = 4, RING_THREADS = 32 * RING_WARPS;
constexpr int KNN_RING_BLOCKS = 148 * 16;          // a query's shells are one chain of latencies: a warp each as far as they go (148 x 4, 10, 16: 60 k clustered points 719, 694, 690 us; 1 M, k = 4 957, 938, 903)
constexpr double KNN_BALL_FACTOR = 2.0;            // expected points within the search radius, in units of k

typedef unsigned long long knn_key;                // (bits of d2) << 32 | source index
constexpr knn_key KNN_NO_KEY = ~0ull;

struct KnnParams {
    RadiusParams rp;        // points, features, plan
    int k;
    float h2;               // square of the search radius: the cells kernel accepts keys <= h2
    float prune2;           // staging drops candidates farther than this (squared) from the cell's points
    float hmin;             // smallest cell edge, shortened by 2^-10 (guarantee of the rings kernel)
    float* out;
    int32_t* nbr;
    float* nbr_d2;
    int32_t* queue;         // queries the cells kernel could not finish
};

// the key's squared distance: operation order fixed, nothing contracted
static __device__ __forceinline__ float key_d2(const float qx, const float qy, const float qz,
                                               const float cx, const float cy, const float cz) {
    const float dx = __fsub_rn(qx, cx), dy = __fsub_rn(qy, cy), dz = __fsub_rn(qz, cz);
    return __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
}

static __device__ __forceinline__ int key_index(const knn_key v) { return (int)(unsigned)(v & 0xffffffffull); }
static __device__ __forceinline__ float key_dist(const knn_key v) { return __uint_as_float((unsigned)(v >> 32)); }

// sorts 32 keys, one per lane, ascending by lane (bitonic network)
static __device__ __forceinline__ knn_key sort32(knn_key v, const int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const knn_key o = __shfl_xor_sync(0xffffffffu, v, stride);
            const bool take_min = ((lane & stride) == 0) == ((lane & size) == 0);
            v = ((v < o) == take_min) ? v : o;
        }
    }
    return v;
}

// a, b sorted ascending by lane: returns the 32 smallest of both, sorted
static __device__ __forceinline__ knn_key merge_low32(const knn_key a, const knn_key b, const int lane) {
    const knn_key br = __shfl_sync(0xffffffffu, b, 31 - lane);
    knn_key c = a < br ? a : br;                              // the 32 smallest as a bitonic sequence
#pragma unroll
    for (int stride = 16; stride > 0; stride >>= 1) {
        const knn_key o = __shfl_xor_sync(0xffffffffu, c, stride);
        c = ((c < o) == ((lane & stride) == 0)) ? c : o;
    }
    return c;
}

// two independent groups of 32 keys sorted side by side (the shuffles of one hide behind the other's)
static __device__ __forceinline__ void sort32x2(knn_key& a, knn_key& b, const int lane) {
#pragma unroll
    for (int size = 2; size <= 32; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            const knn_key oa = __shfl_xor_sync(0xffffffffu, a, stride);
            const knn_key ob = __shfl_xor_sync(0xffffffffu, b, stride);
            const bool take_min = ((lane & stride) == 0) == ((lane & size) == 0);
            a = ((a < oa) == take_min) ? a : oa;
            b = ((b < ob) == take_min) ? b : ob;
        }
    }
}

// The 32 smallest keys of lq[0, n), sorted, lane t holding the t-th (KNN_NO_KEY beyond n).
// List entries are (index, d2) pairs, which read as one little-endian 64-bit key.
static __device__ __noinline__ knn_key select_sorted(const float2* lq, const int n, const int lane) {
    const knn_key* l64 = reinterpret_cast<const knn_key*>(lq);
    if (n <= 32) return sort32(lane < n ? l64[lane] : KNN_NO_KEY, lane);
    knn_key best = l64[lane];
    knn_key v = 32 + lane < n ? l64[32 + lane] : KNN_NO_KEY;
    sort32x2(best, v, lane);
    best = merge_low32(best, v, lane);
    for (int base = 64; base < n; base += 32) {
        v = sort32(base + lane < n ? l64[base + lane] : KNN_NO_KEY, lane);
        best = merge_low32(best, v, lane);
    }
    return best;
}

// Trims lq[0, n), n <= 96, to the entries with d2 <= t for a t that at least k and at most KNN_TRIM of them satisfy; tau bounds
// the distances in the list.  Returns the new length and sets tau = t, or returns n when no such t was found (many
// equal distances).
static __device__ __forceinline__ int trim_list(float2* lq, const int n, const int k, float& tau, const int lane) {
    constexpr unsigned FULL = 0xffffffffu;
    const float far = __int_as_float(0x7f800000);
    float2 e[3];
#pragma unroll
    for (int g = 0; g < 3; ++g) e[g] = 32 * g + lane < n ? lq[32 * g + lane] : make_float2(0.f, far);
    const float target = 0.5f * (float)(k + KNN_TRIM);
    float lo = 0.f, hi = tau, at = tau;
    int c = n;
    unsigned m[3];
    for (int it = 0; it < 8; ++it) {
        // counts grow like the cube of the distance: d2 ~ count^(2/3)
        float t = at * fast_exp2(0.6666667f * __log2f(target / (float)(c > 0 ? c : 1)));
        if (!(t > lo && t < hi)) t = 0.5f * (lo + hi);
        at = t;
        c = 0;
#pragma unroll
        for (int g = 0; g < 3; ++g) { m[g] = __ballot_sync(FULL, e[g].y <= t); c += __popc(m[g]); }
        if (c >= k && c <= KNN_TRIM) {
            const unsigned lt = (1u << lane) - 1u;
            int pos = 0;
#pragma unroll
            for (int g = 0; g < 3; ++g) {
                if ((m[g] >> lane) & 1u) lq[pos + __popc(m[g] & lt)] = e[g];
                pos += __popc(m[g]);
            }
            __syncwarp();
            tau = t;
            return c;
        }
        if (c < k) lo = t; else hi = t;
    }
    return n;
}

// Writes the row of query i from its m selected entries: lanes with sel hold source id, distance and place in the row.
// ids: room for 32 ids (features of eight and more are gathered by groups of lanes, several rows at a time).
static __device__ __forceinline__ void emit_row(const KnnParams& P, const int i, const bool sel, const int id, const float d2, const int place, const int m,
                                                int* ids, const int lane) {
    constexpr unsigned FULL = 0xffffffffu;
    const int k = P.k, F = P.rp.F;
    if (sel) {
        if (P.nbr) P.nbr[(size_t)i * k + place] = id;
        if (P.nbr_d2) P.nbr_d2[(size_t)i * k + place] = d2;
    }
    const float* feat = P.rp.feat;
    if (F >= 8) {
        __syncwarp();
        if (sel) ids[place] = checked(id, P.rp.n, CHECK_POINT);
        __syncwarp();
        // 8, 16 or 32 lanes span a row, the warp's groups take rows in turn; four rows in flight per lane (one at a time:
        // F = 64, k = 16, 1 M points 2770 instead of 1633 us; F = 8 998 and 906)
        const int lg = F <= 8 ? 3 : F <= 16 ? 4 : 5, fl = lane & ((1 << lg) - 1), g = lane >> lg, step = 32 >> lg;
        for (int f = fl; f - fl < F; f += 1 << lg) {
            const bool in = f < F;
            float acc = 0.f;
            for (int t = g; t < m; t += 4 * step) {
                float x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = in && t + u * step < m ? __ldg(feat + (size_t)ids[t + u * step] * F + f) : 0.f;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (t + u * step < m) acc += x[u];
            }
            for (int o = 1 << lg; o < 32; o <<= 1) acc += __shfl_xor_sync(FULL, acc, o);
            if (g == 0 && in) P.out[(size_t)i * F + f] = acc;
        }
    } else {
        const size_t row = sel ? (size_t)checked(id, P.rp.n, CHECK_POINT) * F : 0;
        for (int f = 0; f < F; ++f) {
            float x = sel ? __ldg(feat + row + f) : 0.f;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
            if (lane == 0) P.out[(size_t)i * F + f] = x;
        }
    }
}

// the row of query i from m <= k keys in order, one per lane; missing entries are -1 and +inf
static __device__ __forceinline__ void emit_sorted(const KnnParams& P, const int i, const knn_key top, const int m, int* ids, const int lane) {
    const bool v = lane < m;
    if (lane >= m && lane < P.k) {
        if (P.nbr) P.nbr[(size_t)i * P.k + lane] = -1;
        if (P.nbr_d2) P.nbr_d2[(size_t)i * P.k + lane] = __int_as_float(0x7f800000);
    }
    emit_row(P, i, v, v ? key_index(top) : -1, key_dist(top), lane, m, ids, lane);
}

// Selects and writes the row of query i from its list of n >= k entries, none farther than tau (squared).
// tied: the warp's last query had equal distances, so this one is ordered by whole keys at once (points on a lattice: counting
// first and then sorting, 64,000 points, k = 8 and 16, 105 and 95 us instead of 95 and 85 us).
static __device__ __forceinline__ void select_and_emit(const KnnParams& P, const int i, float2* lq, int n, float tau, bool& tied, const int lane) {
    constexpr unsigned FULL = 0xffffffffu;
    const int k = P.k;
    if (k <= KNN_COUNT_K && n > KNN_TRIM) n = trim_list(lq, n, k, tau, lane);
    if (k <= KNN_COUNT_K && n <= KNN_TRIM && !tied) {
        const float2 own = lane < n ? lq[lane] : make_float2(0.f, __int_as_float(0x7f800000));
        int place = 0;
        const float4* l4 = reinterpret_cast<const float4*>(lq);
        int j = 0;
        for (; j + 4 <= n; j += 4) {
            const float4 a = l4[j >> 1], b = l4[(j >> 1) + 1];
            place += (a.y < own.y ? 1 : 0) + (a.w < own.y ? 1 : 0) + (b.y < own.y ? 1 : 0) + (b.w < own.y ? 1 : 0);
        }
        for (; j < n; ++j) place += lq[j].y < own.y ? 1 : 0;
        // equal distances share a place: then the general form orders them by index
        const unsigned taken = __reduce_or_sync(FULL, lane < n ? 1u << place : 0u);
        if (__popc(taken) == n) {
            emit_row(P, i, lane < n && place < k, __float_as_int(own.x), own.y, place, k, reinterpret_cast<int*>(lq), lane);
            return;
        }
    }
    const knn_key top = select_sorted(lq, n, lane);
    const float before = __shfl_up_sync(FULL, key_dist(top), 1);
    tied = __any_sync(FULL, lane > 0 && lane < n && key_dist(top) == before);
    emit_sorted(P, i, top, k, reinterpret_cast<int*>(lq), lane);
}

// ------------------------------------------------------------------------------ cells kernel
// queries [qs0, qe0) of one cell (the whole cell, or a slice of a dense one)
// SU: groups of 32 candidates staged per step.  A step that no longer fits the stage is taken again, and above k = 20 the
// stencil keeps more candidates (about 9 k) than the stage holds, for every batch of queries anew: short steps there (one
// feature, 1 M points, k = 24, 25, 32: 1428, 1349, 1816 us with four groups, 1288, 1238, 1672 us with two; k = 16 783 and 816 us).
template <int SU>
__device__ __forceinline__ void knn_cell_slice(const KnnParams& P, const int (&c)[3], const int qs0, const int qe0, bool& tied, unsigned char* s_raw) {
    const RadiusParams& p = P.rp;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;

    unsigned char* base = s_raw + (size_t)wib * KNN_PER_WARP;
    float4* stage = reinterpret_cast<float4*>(base);                                      // x, y, z, point id
    float2* list = reinterpret_cast<float2*>(base + KNN_STAGE_BYTES);                     // (point id, d2) per query
    float4* s_q = reinterpret_cast<float4*>(base + KNN_STAGE_BYTES + KNN_LIST_BYTES);
    int* s_n = reinterpret_cast<int*>(s_q + KQB);
    float* s_tau = reinterpret_cast<float*>(s_n + KQB);
    const unsigned lt_mask = (1u << lane) - 1u;
    const int k = P.k;

    // ---- the stencil as nine ranges of the cell-ordered points: the x neighbours are contiguous
    int* s_delta = reinterpret_cast<int*>(s_tau + KQB);
    const RunStencil sten(p, c, 1, s_delta);
    const int total = sten.total;

    // ---- bounding box of the cell's points, one register per lane (lane d: low, lane 3 + d: high)
    float bb;
    {
        float blo[3] = {FAR_AWAY, FAR_AWAY, FAR_AWAY}, bhi[3] = {-FAR_AWAY, -FAR_AWAY, -FAR_AWAY};
        for (int q = qs0 + lane; q < qe0; q += 32) {
            const float4 pq = p.spos[q];
            blo[0] = fminf(blo[0], pq.x); bhi[0] = fmaxf(bhi[0], pq.x);
            blo[1] = fminf(blo[1], pq.y); bhi[1] = fmaxf(bhi[1], pq.y);
            blo[2] = fminf(blo[2], pq.z); bhi[2] = fmaxf(bhi[2], pq.z);
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) { blo[d] = warp_min(blo[d]); bhi[d] = warp_max(bhi[d]); }
        bb = lane == 0 ? blo[0] : lane == 1 ? blo[1] : lane == 2 ? blo[2] : lane == 3 ? bhi[0] : lane == 4 ? bhi[1] : bhi[2];
    }

    // ---- stages kept candidates starting at flattened stencil position v0 until the next step might not fit or the stencil
    //      ends; returns the next position, the kept count in ns.  `before` counts the ranges that began before v0 (-1 at 0).
    auto stage_from = [&](int v0, int& before, int& ns) -> int {
        static_assert(KNN_STAGE_CAP >= 32 * SU, "a step fits an empty stage");
        int nst = 0;
        while (v0 < total) {
            const int step = total - v0 < 32 * SU ? total - v0 : 32 * SU, before0 = before;
            float4 c4[SU];
            unsigned kept[SU];
#pragma unroll
            for (int u = 0; u < SU; ++u) {                    // all loads of the step first
                c4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (32 * u >= step) continue;
                const int src = sten.source(v0 + 32 * u, before, s_delta);
                if (v0 + 32 * u + lane < total) c4[u] = __ldg(p.spos + checked(src, p.n, CHECK_SLOT));
            }
            const float lx = __shfl_sync(FULL, bb, 0), ly = __shfl_sync(FULL, bb, 1), lz = __shfl_sync(FULL, bb, 2);
            const float hx = __shfl_sync(FULL, bb, 3), hy = __shfl_sync(FULL, bb, 4), hz = __shfl_sync(FULL, bb, 5);
            int all = nst;
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                kept[u] = 0u;
                if (32 * u >= step) continue;
                const float ex = fmaxf(fmaxf(lx - c4[u].x, c4[u].x - hx), 0.f);
                const float ey = fmaxf(fmaxf(ly - c4[u].y, c4[u].y - hy), 0.f);
                const float ez = fmaxf(fmaxf(lz - c4[u].z, c4[u].z - hz), 0.f);
                kept[u] = __ballot_sync(FULL, v0 + 32 * u + lane < total && fmaf(ez, ez, fmaf(ey, ey, ex * ex)) <= P.prune2);
                all += __popc(kept[u]);
            }
            if (all > KNN_STAGE_CAP) { before = before0; break; }     // taken again with an empty stage
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                if ((kept[u] >> lane) & 1u) stage[nst + __popc(kept[u] & lt_mask)] = c4[u];
                nst += __popc(kept[u]);
            }
            v0 += 32 * SU;
        }
        if (lane < STAGE_PAD) stage[nst + lane] = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, __int_as_float(-1));
        __syncwarp();
        ns = nst;
        return v0;
    };

    int ns = 0, before = -1;
    const bool single = stage_from(0, before, ns) >= total;           // the whole (pruned) stencil fits: staged once

    for (int qb0 = qs0; qb0 < qe0; qb0 += KQB) {
        const int nq = (qe0 - qb0 < KQB) ? qe0 - qb0 : KQB;
        __syncwarp();
        if (lane < KQB) {
            // absent queries sit far away with a negative threshold: they accept nothing
            const float4 pq = lane < nq ? p.spos[qb0 + lane] : make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, __int_as_float(-2));
            s_q[lane] = pq;
            s_n[lane] = 0;
            s_tau[lane] = lane < nq ? P.h2 : -1.f;
        }
        __syncwarp();
        int qcnt[KQB];
        float tq[KQB];
#pragma unroll
        for (int q = 0; q < KQB; ++q) { qcnt[q] = 0; tq[q] = s_tau[q]; }

        // all queries of the batch against the ns staged candidates
        auto scan = [&](const int ns_, auto width) {
            constexpr int NQ = decltype(width)::value;             // queries tested per trip (a short batch tests four)
            for (int cbase = 0; cbase < ns_; cbase += 32) {
                const float4 pj = stage[cbase + lane];
                int mx = 0;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    const float4 qv = s_q[q];
                    const float d2 = key_d2(qv.x, qv.y, qv.z, pj.x, pj.y, pj.z);
                    const bool ok = d2 <= tq[q] && __float_as_int(pj.w) != __float_as_int(qv.w);
                    const unsigned m = __ballot_sync(FULL, ok);
                    if (ok) list[q * KNN_QSTRIDE + qcnt[q] + __popc(m & lt_mask)] = make_float2(pj.w, d2);
                    qcnt[q] += __popc(m);
                    mx = qcnt[q] > mx ? qcnt[q] : mx;
                }
                if (mx > KNN_QCAP - 32) {
                    // a list may overflow on the next trip: trim every long list; what bounds the entries left
                    // becomes that query's threshold (later equal keys are resolved by index)
                    __syncwarp();
                    if (lane == 0) {
#pragma unroll
                        for (int q = 0; q < KQB; ++q) s_n[q] = qcnt[q];
                    }
                    __syncwarp();
                    for (int q = 0; q < nq; ++q) {
                        const int n = s_n[q];
                        if (n > (k <= KNN_COUNT_K ? KNN_TRIM : k)) {
                            float2* lq = list + q * KNN_QSTRIDE;
                            float tau = s_tau[q];
                            const int left = k <= KNN_COUNT_K ? trim_list(lq, n, k, tau, lane) : n;
                            if (left < n) {
                                if (lane == 0) { s_n[q] = left; s_tau[q] = tau; }
                            } else {
                                const knn_key top = select_sorted(lq, n, lane);
                                __syncwarp();
                                if (lane < k) reinterpret_cast<knn_key*>(lq)[lane] = top;
                                if (lane == k - 1) { s_n[q] = k; s_tau[q] = key_dist(top); }
                            }
                            __syncwarp();
                        }
                    }
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < KQB; ++q) { qcnt[q] = s_n[q]; tq[q] = s_tau[q]; }
                }
            }
        };

        if (single) {
            if (nq <= KQB / 2) scan(ns, std::integral_constant<int, KQB / 2>{});
            else scan(ns, std::integral_constant<int, KQB>{});
        } else {
            before = -1;
            for (int v = 0; v < total;) {
                int ns2;
                v = stage_from(v, before, ns2);
                scan(ns2, std::integral_constant<int, KQB>{});
                __syncwarp();
            }
        }

        // ---- finish the batch: k keys within h settle a query, otherwise it is handed on
        __syncwarp();
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < KQB; ++q) s_n[q] = qcnt[q];
        }
        __syncwarp();
        for (int q = 0; q < nq; ++q) {
            const int n = s_n[q];
            const int i = __float_as_int(s_q[q].w);
            if (n < k) {
                if (lane == 0) P.queue[atomicAdd(p.queue_n, 1)] = i;
            } else {
                select_and_emit(P, i, list + q * KNN_QSTRIDE, n, s_tau[q], tied, lane);
            }
        }
    }
}

// one warp per unit of points; cells are not joined (the search radius already gives a cell about k / 2 points)
template <int SU>
__global__ void __launch_bounds__(TRAV_THREADS, 32 / TRAV_WARPS) knn_cells_kernel(const __grid_constant__ KnnParams P) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    bool tied = false;
    auto work = [&](const int (&cell)[3], int, const int qs, const int qe) { knn_cell_slice<SU>(P, cell, qs, qe, tied, s_raw); };
    walk_unit(P.rp, blockIdx.x * TRAV_WARPS + (threadIdx.x >> 5), 1, work);
}

// ------------------------------------------------------------------------------ rings kernel
__global__ void __launch_bounds__(RING_THREADS) knn_rings_kernel(const __grid_constant__ KnnParams P) {
    const RadiusParams& p = P.rp;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ float2 s_list[RING_WARPS][KNN_RING_CAP + 32];

    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    float2* list = s_list[wib];
    const unsigned lt_mask = (1u << lane) - 1u;
    const int k = P.k;
    const int nqueue = *p.queue_n;
    const int nwarps = gridDim.x * RING_WARPS;
    const int nx = p.nc[0], ny = p.nc[1], nz = p.nc[2];
    const int smax = max(nx, max(ny, nz));

    for (int t = blockIdx.x * RING_WARPS + wib; t < nqueue; t += nwarps) {
        const int i = P.queue[t];
        const float qx = p.pos[3 * (size_t)i], qy = p.pos[3 * (size_t)i + 1], qz = p.pos[3 * (size_t)i + 2];
        const int cid = p.cell[i];
        const int cx = cid % nx, cy = (cid / nx) % ny, cz = cid / (nx * ny);
        int cnt = 0;
        float tau = 3.0e38f;
        __syncwarp();

        // cuts the list back to its (at most k) smallest keys, sorted; k keys set the threshold
        auto cut = [&]() {
            const knn_key top = select_sorted(list, cnt, lane);
            __syncwarp();
            cnt = cnt < k ? cnt : k;
            if (lane < cnt) reinterpret_cast<knn_key*>(list)[lane] = top;
            if (cnt == k) tau = key_dist(__shfl_sync(FULL, top, k - 1));
            __syncwarp();
        };

        // Rows of cells beyond the k-th key found so far are skipped (with shells read in full, 131 k points, k = 16 174 instead of 159 us, 60 k
        // clustered points 816 instead of 719).  Squared distance of a coordinate in cell `own` from the cells [a, b] of dimension d, short of it by at least 2^-10 of a cell
        auto beyond = [&](const float v, const int own, const int a, const int b, const int d) {
            if (own >= a && own <= b) return 0.f;
            const float gap = fmaxf((float)a * p.hcell[d] - v, v - (float)(b + 1) * p.hcell[d]) - p.hcell[d] * (1.f / 1024.f) - 4e-7f * p.len[d];
            return gap > 0.f ? gap * gap : 0.f;
        };
        for (int s = 0; s <= smax; ++s) {
            const int z0 = max(cz - s, 0), z1 = min(cz + s, nz - 1);
            const int y0 = max(cy - s, 0), y1 = min(cy + s, ny - 1);
            const int x0 = max(cx - s, 0), x1 = min(cx + s, nx - 1);
            const int wy = y1 - y0 + 1, nrow = (z1 - z0 + 1) * wy;
            // the (y, z) rows of the shell, sixteen at a time: every lane resolves one contiguous run of
            // cell-ordered points (a face row is one run over the whole x range, an inner row has its two
            // end cells), then the runs are walked as one flat sequence so that all loads are independent
            for (int rbase = 0; rbase < nrow; rbase += 16) {
                const int rr = rbase + (lane >> 1), side = lane & 1;
                int ra = 0, rlen = 0;
                if (rr < nrow) {
                    const int z = z0 + rr / wy, y = y0 + rr % wy;
                    const int row = (z * ny + y) * nx;
                    const bool face = z - cz == s || cz - z == s || y - cy == s || cy - y == s;
                    int xa = -1, xb = -1;                                  // cells [xa, xb]
                    if (face) { if (side == 0) { xa = x0; xb = x1; } }
                    else if (side == 0) { if (cx - s >= 0) xa = xb = cx - s; }
                    else if (s > 0 && cx + s < nx) xa = xb = cx + s;
                    if (xa >= 0 && beyond(qx, cx, xa, xb, 0) + beyond(qy, cy, y, y, 1) + beyond(qz, cz, z, z, 2) <= tau) {
                        ra = p.cell_start[row + xa];
                        rlen = p.cell_start[row + xb + 1] - ra;
                    }
                }
                int rincl = rlen;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t2 = __shfl_up_sync(FULL, rincl, o);
                    if (lane >= o) rincl += t2;
                }
                const int total = __shfl_sync(FULL, rincl, 31);
                for (int v0 = 0; v0 < total; v0 += 32) {
                    const int v = v0 + lane;
                    int r = 0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const int probe = __shfl_sync(FULL, rincl, r + o - 1);
                        if (probe <= v) r += o;
                    }
                    r = r > 31 ? 31 : r;
                    const int src = __shfl_sync(FULL, ra, r) + (v - (__shfl_sync(FULL, rincl, r) - __shfl_sync(FULL, rlen, r)));
                    bool ok = false;
                    float4 c4 = make_float4(0.f, 0.f, 0.f, 0.f);
                    float d2 = 0.f;
                    if (v < total) {
                        c4 = __ldg(p.spos + checked(src, p.n, CHECK_SLOT));
                        d2 = key_d2(qx, qy, qz, c4.x, c4.y, c4.z);
                        ok = d2 <= tau && __float_as_int(c4.w) != i;
                    }
                    const unsigned m = __ballot_sync(FULL, ok);
                    if (ok) list[cnt + __popc(m & lt_mask)] = make_float2(c4.w, d2);
                    cnt += __popc(m);
                    if (cnt > KNN_RING_CAP - 32) {
                        __syncwarp();
                        cut();
                    }
                }
            }
            // every point whose cell differs by more than s from the query's in some dimension is
            // farther than s cell edges away: k keys within that distance cannot be improved
            __syncwarp();
            if (cnt >= k) {
                cut();                                            // sorted: the k-th key is the largest kept
                const float g = (float)s * P.hmin;
                if (tau <= g * g) break;
            }
            if (cx - s <= 0 && cy - s <= 0 && cz - s <= 0 && cx + s >= nx - 1 && cy + s >= ny - 1 && cz + s >= nz - 1) break;
        }
        __syncwarp();
        emit_sorted(P, i, select_sorted(list, cnt, lane), cnt < k ? cnt : k, reinterpret_cast<int*>(list), lane);
        __syncwarp();
    }
}

// ------------------------------------------------------------------------------ host side
// search radius: a ball of radius h holds about 2k points at the input's mean density
static float knn_search_radius(long long n, int k, const tiga_box* box) {
    double vol = 1.0, lmax = 0.0;
    for (int d = 0; d < 3; ++d) {
        vol *= (double)box->len[d];
        lmax = (double)box->len[d] > lmax ? (double)box->len[d] : lmax;
    }
    if (n < 2) return (float)lmax;
    const double h = cbrt(KNN_BALL_FACTOR * (double)k * vol / ((double)n * 4.18879020478639));
    return (float)(h < lmax ? h : lmax);
}

static tiga_status knn_check(long long n, int k, const tiga_box* box) {
    if (!box || n < 0 || k < 1) return TIGA_ERR_INVALID_ARG;
    if (k > TIGA_KNN_MAX_K) return TIGA_ERR_UNSUPPORTED;
    for (int d = 0; d < 3; ++d) {
        if (!(box->len[d] > 0.f) || !isfinite(box->len[d])) return TIGA_ERR_INVALID_ARG;
        if (box->periodic[d]) return TIGA_ERR_UNSUPPORTED;
    }
    return TIGA_OK;
}

static size_t knn_carve(KnnParams* P, void* ws, int32_t** fill, RadiusLayout* lay) {
    *lay = carve_radius(&P->rp, ws, fill);
    Carver cv(ws);
    cv.off = lay->bytes;
    P->queue = cv.take<int32_t>((size_t)P->rp.n + 1);
    return cv.off;
}

}  // namespace tiga

using namespace tiga;

extern "C" size_t tiga_knn_workspace_bytes(int64_t n, int32_t k, const tiga_box* box) {
    if (knn_check(n, k, box) != TIGA_OK) return 0;
    KnnParams P{};
    if (fill_params(&P.rp, n, knn_search_radius(n, k, box), box) != TIGA_OK) return 0;
    int32_t* fill;
    RadiusLayout lay;
    return knn_carve(&P, nullptr, &fill, &lay) + 256;
}

extern "C" tiga_status tiga_apply_knn(const float* pos, const float* feat, int64_t n, int32_t F, int32_t k,
                                      const tiga_box* box, float* out, int32_t* nbr, float* nbr_d2,
                                      void* ws, size_t ws_bytes, void* stream) {
    tiga_status st = knn_check(n, k, box);
    if (st != TIGA_OK) return st;
    if (F < 1) return TIGA_ERR_INVALID_ARG;
    KnnParams P{};
    const float h = knn_search_radius(n, k, box);
    st = fill_params(&P.rp, n, h, box);
    if (st != TIGA_OK) return st;
    if (n == 0) return TIGA_OK;
    if (!pos || !feat || !out || !aligned16(pos)) return TIGA_ERR_INVALID_ARG;
    if (!ws || !aligned16(ws) || ws_bytes < tiga_knn_workspace_bytes(n, k, box)) return TIGA_ERR_WORKSPACE;
    int32_t* fill;
    RadiusLayout lay;
    knn_carve(&P, ws, &fill, &lay);
    P.rp.pos = pos; P.rp.feat = feat; P.rp.F = F;
    P.k = k;
    cut_cells(P.rp, 148 * 84);           // a query costs more here: finer slices
    P.h2 = h * h;
    P.prune2 = P.rp.r2_hi * 1.0001f;
    float hmin = P.rp.hcell[0];
    for (int d = 1; d < 3; ++d) hmin = P.rp.hcell[d] < hmin ? P.rp.hcell[d] : hmin;
    P.hmin = hmin * (1.f - 1.f / 1024.f);
    P.out = out; P.nbr = nbr; P.nbr_d2 = nbr_d2;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    st = run_binning(P.rp, fill, lay.nblocks, s);
    if (st != TIGA_OK) return st;
    constexpr int smem = KNN_PER_WARP * TRAV_WARPS;
    auto cells = k > 20 ? knn_cells_kernel<2> : knn_cells_kernel<4>;
    TIGA_CUDA_TRY(cudaFuncSetAttribute(cells, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    cells<<<counted(unit_blocks(P.rp)), TRAV_THREADS, smem, s>>>(P);
    knn_rings_kernel<<<counted(KNN_RING_BLOCKS), RING_THREADS, 0, s>>>(P);
    return launch_status();
}

namespace tiga { unsigned check_status_knn(bool reset) { return read_check_status(reset); } }
