// Edge neural network over the generated radius relation (paper Appendix A):
//     y_i = sum over j in N(i) of [ W2 ReLU( W1 [p_j - p_i ; x_j] + b1 ) + b2 ]
// fused with the cell-directory traversal, and its reverse mode with the membership frozen
// (Section 5), which recomputes the pre-activations per pair instead of storing them and gives
// gradients with respect to node features, positions and the four parameter arrays.
//
// Staging and candidate test are those of radius_test.cuh (a run of cells per warp, persistent grid); accepted pairs
// are compacted into one list of (displacement, staged slot) per query.  A pair is then evaluated by HID lanes, one
// hidden unit each, with the lane's row of W1 in registers and the pair's inputs broadcast from shared memory, so 32 / HID
// pairs advance together.  Everything behind the ReLU is linear, so it is applied once per query to sums over the pairs:
//     S[a] = sum relu(h_a)      c[a] = #(h_a > 0)      D[a] = sum (p_j - p_i) [h_a > 0]
//     out_i = W2 S + |N(i)| b2
// Backward, owner computes: with v = W2^T ybar, query k and its neighbours m,
//     G[a] = sum over m of v_m[a] [h_a of the pair (m <- k) > 0]
//     xbar_k = W1x^T G,   pbar_k = W1p^T (G - v_k c)          (no atomics, reproducible)
//     W1bar += [ v_k D ; G x_k ],   b1bar += v_k c,   W2bar += ybar_k S,   b2bar += |N(k)| ybar_k
// where every lane accumulates the parameter gradients of its hidden unit in registers over all its queries; at the end
// warps fold into the CTA's shared copy and the CTA adds that to global memory with one atomic per entry.
//
// Bound by instruction issue (57 % of the slots, 28 and 49 M warp instructions) and the tail of the work units.  35,947 surface
// points, 15.6 neighbours, 8 features, HID = 32: forward 121 -> 55 us, backward 512 -> 86 us against one lane per pair with
// the weights read from shared memory (the earlier form, some 600 shared-memory reads per 32 pairs); 300 k uniform points,
// 32 neighbours, HID = 16: 455 -> 383 and 1750 -> 603 us.  (Sums that keep their precision, below, add 5 % to the surface's two passes.)
//
// The displacement is formed from coordinates relative to the corner of the query's cell and the pre-activation as one chain
// of fused multiply-adds (bias, displacement, features): a ReLU switches on the last bit of that sum.
#include "radius_direct.cuh"
#include <float.h>

namespace tiga {

// Forward: one warp per CTA, a CTA per unit of points.  Backward: a persistent grid of one CTA per SM (the parameter gradients
// are folded once per CTA), which owns every 148th unit and whose 16 (FQ > 2: 12) warps draw from those through a counter in
// shared memory: balanced within the SM, and nothing of the caller's plan is written.  Against one counter for all CTAs
// in the workspace, which calls that share a plan would share too: 35,947 surface points 82.9 us with either, uniform points
// within 2 %, 8 k clustered points 318 -> 309 us with 8 features, 226 -> 283 us with 13.  Four-warp CTAs that own their units
// (4 of 16 warps balance each other): 83 -> 87 and 318 -> 380 us; clusters of eight such CTAs with one counter: 126 us.
template <int FQ> __host__ __device__ constexpr int mlp_warps(bool bwd) { return bwd ? (FQ <= 2 ? 16 : 12) : 1; }

template <int HID, int FQ, bool BWD> struct MlpSmem {
    static constexpr int NX = 4 * FQ;                                            // staged features per candidate (zero padded)
    static constexpr int STAGE_CAP = 144, LIST_CAP = 176;
    static_assert(LIST_CAP >= STAGE_CAP, "a query's whole chunk fits the list");
    static constexpr int STAGE_BYTES = TestStage<STAGE_CAP>::BYTES;
    static constexpr int X_BYTES = STAGE_CAP * NX * 4, G_BYTES = BWD ? STAGE_CAP * 16 : 0, LIST_BYTES = LIST_CAP * 16;
    static constexpr int PER_WARP = STAGE_BYTES + X_BYTES + G_BYTES + LIST_BYTES + ((2 * TEST_BATCH + QDENSE + 20) * 4 + 15) / 16 * 16;
    static constexpr int K_PAD = 3 + NX;
    static constexpr int GRAD_FLOATS = HID * (K_PAD + 1 + 4) + 4;                // W1, b1, W2, b2 of the CTA's gradient copy
    static constexpr int CTA_BYTES = BWD ? (GRAD_FLOATS * 4 + 4 + 15) / 16 * 16 : 0;      // and its unit counter
    static constexpr int WARPS = mlp_warps<FQ>(BWD), THREADS = 32 * WARPS, TOTAL = CTA_BYTES + WARPS * PER_WARP;
};

// resident warps per SM the kernel is compiled for (register budget)
template <int FQ, bool BWD> __host__ __device__ constexpr int mlp_warps_per_sm() { return BWD ? (FQ <= 2 ? 16 : 12) : (FQ <= 2 ? 20 : 16); }

// Sums v[0..NV) over the L lanes of an aligned group by a halving exchange; afterwards lane l holds, in v[0..NV / min(NV, L)),
// the totals of the entries from spread_first<NV, L>(l).
template <int NV, int L, typename T>
static __device__ __forceinline__ void spread_sum(T* v, const int l) {
#pragma unroll
    for (int j = 0; (1 << j) < L; ++j) {
        const int left = NV >> j;
        if (left > 1) {
            const bool up = (l >> j) & 1;
#pragma unroll
            for (int k = 0; k < left / 2; ++k) {
                const T send = up ? v[k] : v[k + left / 2], keep = up ? v[k + left / 2] : v[k];
                v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 1 << j);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1 << j);
        }
    }
}
template <int NV, int L>
static __device__ __forceinline__ int spread_first(const int l) {
    int first = 0;
#pragma unroll
    for (int j = 0; (1 << j) < L && (NV >> j) > 1; ++j) first += ((l >> j) & 1) * (NV >> (j + 1));
    return first;
}

template <int HID, int FQ, bool BWD, bool MI>
__global__ void __launch_bounds__(32 * mlp_warps<FQ>(BWD), (mlp_warps_per_sm<FQ, BWD>() / mlp_warps<FQ>(BWD))) radius_mlp_kernel(const __grid_constant__ RadiusParams p) {
    using SM = MlpSmem<HID, FQ, BWD>;
    constexpr int STAGE_CAP = SM::STAGE_CAP, LIST_CAP = SM::LIST_CAP, NX = SM::NX, KP = SM::K_PAD;
    constexpr int PS = 32 / HID;                       // pairs evaluated together
    constexpr unsigned FULL = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int a = lane % HID, ps = lane / HID;
    const int Fin = p.Fin, Fout = p.Fout, K = 3 + p.Fin;

    float* sG = reinterpret_cast<float*>(s_raw);       // BWD: W1 [HID][KP], b1 [HID], W2 [4][HID], b2 [4]
    unsigned* s_drawn = reinterpret_cast<unsigned*>(sG + SM::GRAD_FLOATS);       // BWD: units of the CTA taken so far
    if constexpr (BWD) {
        for (int e = threadIdx.x; e < SM::GRAD_FLOATS; e += SM::THREADS) sG[e] = 0.f;
        if (threadIdx.x == 0) *s_drawn = 0;
        __syncthreads();
    }
    unsigned char* base = s_raw + SM::CTA_BYTES + (size_t)wib * SM::PER_WARP;
    const TestStage<STAGE_CAP> stage(base);
    float* s_x = reinterpret_cast<float*>(base + SM::STAGE_BYTES);                       // [slot][NX]
    float4* s_g = reinterpret_cast<float4*>(base + SM::STAGE_BYTES + SM::X_BYTES);       // [slot] cotangents (BWD)
    float4* list = reinterpret_cast<float4*>(base + SM::STAGE_BYTES + SM::X_BYTES + SM::G_BYTES);
    int* s_off = reinterpret_cast<int*>(list + LIST_CAP);                                // list of every query of the batch: start,
    int* s_end = s_off + TEST_BATCH;                                                     // end
    int* s_self = s_end + TEST_BATCH;                                                    // staged slot of every query, or -1
    int* s_delta = s_self + QDENSE;

    // this lane's hidden unit
    float w[KP], w2[4], b1 = p.b1[a], b2 = lane < Fout ? p.b2[lane] : 0.f;
#pragma unroll
    for (int k = 0; k < KP; ++k) w[k] = k < K ? p.W1[a * K + k] : 0.f;
#pragma unroll
    for (int o = 0; o < 4; ++o) w2[o] = o < Fout ? p.W2[o * HID + a] : 0.f;
    float gW1[BWD ? KP : 1], gW2[4] = {0.f, 0.f, 0.f, 0.f}, gb1 = 0.f, gb2 = 0.f;
#pragma unroll
    for (int k = 0; k < (BWD ? KP : 1); ++k) gW1[k] = 0.f;

    const bool mi0 = MI && p.periodic[0] && p.nc[0] <= 3, mi1 = MI && p.periodic[1] && p.nc[1] <= 3, mi2 = MI && p.periodic[2] && p.nc[2] <= 3;
    auto delta = [&](const int d, const float q, const float c4) -> float {
        const bool mi = d == 0 ? mi0 : d == 1 ? mi1 : mi2;
        return (MI && mi) ? mi_delta(q, c4, p.len[d], 0.5f * p.len[d]) : q - c4;
    };
    const unsigned lt_mask = (1u << lane) - 1u;
    // compensated: W2 S + |N| b2 and W1^T G cancel where the messages do, and a sum of hundreds of terms must not lose more
    // there than adding the messages one by one would.  `lost` is added at the end, so the loop waits for one addition.
    auto add = [](float& sum, float& lost, const float term) {
        const float t = sum + term;
        lost += term - (t - sum);
        sum = t;
    };

    auto slice = [&](const int (&cell)[3], const int run, const int qs0, const int qe0) {
        const RunFrame frame(p, cell, run);
        const RunStencil sten(p, frame.c, run, s_delta);
        float blo[3] = {FAR_AWAY, FAR_AWAY, FAR_AWAY}, bhi[3] = {-FAR_AWAY, -FAR_AWAY, -FAR_AWAY};
        for (int q = qs0 + lane; q < qe0; q += 32) {
            float4 pq = p.spos[q];
            frame.shift(p, pq);
            const float l[3] = {pq.x, pq.y, pq.z};
#pragma unroll
            for (int d = 0; d < 3; ++d) { blo[d] = fminf(blo[d], l[d]); bhi[d] = fmaxf(bhi[d], l[d]); }
        }
#pragma unroll
        for (int d = 0; d < 3; ++d) { blo[d] = warp_min(blo[d]); bhi[d] = warp_max(bhi[d]); }
        if (mi0) { blo[0] = -FAR_AWAY; bhi[0] = FAR_AWAY; }   // a dimension folded by the explicit minimum image is not pruned
        if (mi1) { blo[1] = -FAR_AWAY; bhi[1] = FAR_AWAY; }
        if (mi2) { blo[2] = -FAR_AWAY; bhi[2] = FAR_AWAY; }
        for (int k = lane; k < qe0 - qs0; k += 32) s_self[k] = -1;
        __syncwarp();                        // staging sets the slot of a query from whichever lane holds its point

        auto process_chunk = [&](const int ns, const bool first_chunk) {
            stage.seal(ns);
            __syncwarp();
            const int all = qe0 - qs0;
            const int per = all <= TEST_BATCH ? all : all <= 2 * TEST_BATCH ? (all + 1) >> 1 : TEST_BATCH;
            for (int qb0 = qs0; qb0 < qe0; qb0 += per) {
                const int nq = (qe0 - qb0 < per) ? qe0 - qb0 : per;
                const LaneSplit split(nq);
                float4 qv = p.spos[qb0 + (split.active ? split.q : 0)];
                const int qid = checked(__float_as_int(qv.w), p.n, CHECK_POINT);
                // corner of the query's cell, in the frame (moved down with its points where a run touches an upper face)
                float ox = (float)(p.cell[qid] - (cell[2] * p.nc[1] + cell[1]) * p.nc[0]) * p.hcell[0];
                float oy = (float)cell[1] * p.hcell[1], oz = (float)cell[2] * p.hcell[2];
                if (frame.face) {
                    if (ox + 0.5f * p.hcell[0] > frame.thr[0]) ox -= p.len[0];
                    if (oy + 0.5f * p.hcell[1] > frame.thr[1]) oy -= p.len[1];
                    if (oz + 0.5f * p.hcell[2] > frame.thr[2]) oz -= p.len[2];
                }
                frame.shift(p, qv);
                unsigned mask[4];
                test_candidates<MI, STAGE_CAP>(p, stage, ns, split, qv.x, qv.y, qv.z, mask, delta);
                drop_candidate(mask, split, split.active ? s_self[qb0 - qs0 + split.q] : -1);

                const int mine = __popc(mask[0]) + __popc(mask[1]) + __popc(mask[2]) + __popc(mask[3]);
                int cnt = mine;                                    // exact decisions below may take some back
                int incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(FULL, incl, o);
                    if (lane >= o) incl += t;
                }
                for (int qa = 0; qa < nq;) {
                    // queries [qa, qb): as many as the list holds
                    const int e0 = __shfl_sync(FULL, incl - mine, qa * split.lpq);
                    const int qb = qa + __popc(__ballot_sync(FULL, split.active && split.q >= qa && split.sub == split.lpq - 1 && incl - e0 <= LIST_CAP));
                    const bool part = split.active && split.q >= qa && split.q < qb;
                    int at = incl - mine - e0;
                    if (part && split.sub == 0) s_off[split.q] = at;
                    if (part && split.sub == split.lpq - 1) s_end[split.q] = at + mine;
                    if (part) {
#pragma unroll
                        for (int wd = 0; wd < 4; ++wd) {
                            unsigned m = mask[wd];
                            while (m) {
                                const int k = __clz(m);
                                m ^= 0x80000000u >> k;
                                int slot = 2 * (split.sub + split.lpq * (TEST_GROUP * (wd >> 1) + k)) + (wd & 1);
                                const float *c4 = stage.x + slot;
                                constexpr int SL = TestStage<STAGE_CAP>::SLOTS;
                                const float jx = c4[0], jy = c4[SL], jz = c4[2 * SL];
                                const float ex = delta(0, qv.x, jx), ey = delta(1, qv.y, jy), ez = delta(2, qv.z, jz);
                                // within the fp32 error band of the cutoff: decided in fp64
                                if (fmaf(ez, ez, fmaf(ey, ey, ex * ex)) > p.r2_mid - p.r2_band && !exact_pair(p, qid, stage.id[slot])) { slot = -1; --cnt; }
                                // source minus destination
                                list[at++] = make_float4(mi0 ? -ex : (jx - ox) - (qv.x - ox), mi1 ? -ey : (jy - oy) - (qv.y - oy),
                                                         mi2 ? -ez : (jz - oz) - (qv.z - oz), __int_as_float(slot));
                            }
                        }
                    }
                    int nin = cnt;                                 // neighbours of the lane's query: sum over its lanes, in the first
#pragma unroll
                    for (int o = 1; o < TEST_LPQ; o <<= 1) {
                        if (o >= split.lpq) break;
                        const int other = __shfl_down_sync(FULL, nin, o);
                        if (split.sub + o < split.lpq) nin += other;
                    }
                    __syncwarp();
                    for (int q = qa; q < qb; ++q) {                // the warp evaluates one query at a time
                        const int oq = __shfl_sync(FULL, qid, q * split.lpq), nq_in = __shfl_sync(FULL, nin, q * split.lpq);
                        const int off = s_off[q], end = s_end[q];
                        if (nq_in == 0) {
                            // no neighbour in this chunk: nothing is formed from the weights, the cotangent or the features (0 times
                            // an infinite one would be NaN)
                            if (first_chunk) {
                                if (!BWD && lane < Fout) p.out[(size_t)oq * Fout + lane] = 0.f;
                                if (BWD && p.gpos && lane < 3) p.gpos[3 * (size_t)oq + lane] = 0.f;
                                if (BWD && p.gfeat && lane < Fin) p.gfeat[(size_t)oq * Fin + lane] = 0.f;
                            }
                            continue;
                        }
                        float S = 0.f, lost = 0.f, cpos = 0.f, D0 = 0.f, D1 = 0.f, D2 = 0.f, G = 0.f, v = 0.f;
                        float xq[BWD ? NX : 1], gq[4];
                        if constexpr (BWD) {
#pragma unroll
                            for (int f = 0; f < NX; ++f) xq[f] = f < Fin ? __ldg(p.feat + (size_t)oq * Fin + f) : 0.f;
#pragma unroll
                            for (int o = 0; o < 4; ++o) gq[o] = o < Fout ? __ldg(p.gy + (size_t)oq * Fout + o) : 0.f;
                        }
                        for (int t = off + ps; t < end; t += 2 * PS) {
                            // two pairs side by side (their chains are independent); an absent or refused one adds nothing
                            const bool two = t + PS < end;
                            const float4 e[2] = {list[t], list[two ? t + PS : t]};
                            const int slot[2] = {__float_as_int(e[0].w), __float_as_int(e[1].w)};
                            const bool in[2] = {slot[0] >= 0, two && slot[1] >= 0};
                            float h[2];
                            const float4* xr[2];
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                xr[u] = reinterpret_cast<const float4*>(s_x + (slot[u] < 0 ? 0 : slot[u]) * NX);
                                h[u] = fmaf(w[2], e[u].z, fmaf(w[1], e[u].y, fmaf(w[0], e[u].x, b1)));
                            }
#pragma unroll
                            for (int i = 0; i < FQ; ++i) {
#pragma unroll
                                for (int u = 0; u < 2; ++u) {
                                    const float4 x4 = xr[u][i];
                                    h[u] = fmaf(w[3 + 4 * i], x4.x, h[u]); h[u] = fmaf(w[4 + 4 * i], x4.y, h[u]);
                                    h[u] = fmaf(w[5 + 4 * i], x4.z, h[u]); h[u] = fmaf(w[6 + 4 * i], x4.w, h[u]);
                                }
                            }
                            if constexpr (BWD) {
                                // the pairs the other way round: the query as the source
                                float h2[2], vm[2];
#pragma unroll
                                for (int u = 0; u < 2; ++u) {
                                    h2[u] = fmaf(w[2], -e[u].z, fmaf(w[1], -e[u].y, fmaf(w[0], -e[u].x, b1)));
                                    const float4 g4 = s_g[slot[u] < 0 ? 0 : slot[u]];
                                    vm[u] = fmaf(w2[3], g4.w, fmaf(w2[2], g4.z, fmaf(w2[1], g4.y, w2[0] * g4.x)));
                                }
#pragma unroll
                                for (int f = 0; f < NX; ++f) {
#pragma unroll
                                    for (int u = 0; u < 2; ++u) h2[u] = fmaf(w[3 + f], xq[f], h2[u]);
                                }
#pragma unroll
                                for (int u = 0; u < 2; ++u) {
                                    if (in[u] && h[u] > 0.f) { S += h[u]; cpos += 1.f; D0 += e[u].x; D1 += e[u].y; D2 += e[u].z; }
                                    if (!(in[u] && h2[u] > 0.f)) vm[u] = 0.f;
                                }
                                add(G, lost, vm[0] + vm[1]);
                            } else {
                                add(S, lost, (in[0] ? fmaxf(h[0], 0.f) : 0.f) + (in[1] ? fmaxf(h[1], 0.f) : 0.f));
                            }
                        }
                        // sums over the groups of HID lanes
                        double total = BWD ? G : S;
                        if (fabsf(lost) <= FLT_MAX) total += lost;       // (not a number behind an infinite sum)
#pragma unroll
                        for (int o = HID; o < 32; o <<= 1) {
                            total += __shfl_xor_sync(FULL, total, o);
                            if constexpr (BWD) {
                                S += __shfl_xor_sync(FULL, S, o); cpos += __shfl_xor_sync(FULL, cpos, o);
                                D0 += __shfl_xor_sync(FULL, D0, o); D1 += __shfl_xor_sync(FULL, D1, o); D2 += __shfl_xor_sync(FULL, D2, o);
                            }
                        }
                        if constexpr (!BWD) {
                            double y[4];
#pragma unroll
                            for (int o = 0; o < 4; ++o) y[o] = (double)w2[o] * total;
                            spread_sum<4, HID>(y, a);
                            const int o = spread_first<4, HID>(a);
                            const float bias = __shfl_sync(FULL, b2, o);
                            if (lane < 4 && o < Fout) {
                                float* dst = p.out + (size_t)oq * Fout + o;
                                const float val = (float)fma((double)nq_in, (double)bias, y[0]);
                                *dst = first_chunk ? val : *dst + val;
                            }
                        } else {
                            G = (float)total;
                            v = cpos > 0.f ? fmaf(w2[3], gq[3], fmaf(w2[2], gq[2], fmaf(w2[1], gq[1], w2[0] * gq[0]))) : 0.f;
                            const float vc = v * cpos;
                            const double Y = total - (double)v * (double)cpos;
                            gW1[0] = fmaf(v, D0, gW1[0]); gW1[1] = fmaf(v, D1, gW1[1]); gW1[2] = fmaf(v, D2, gW1[2]);
#pragma unroll
                            for (int f = 0; f < NX; ++f) gW1[3 + f] = fmaf(G, xq[f], gW1[3 + f]);
                            gb1 += vc;
#pragma unroll
                            for (int o = 0; o < 4; ++o) gW2[o] = fmaf(gq[o], S, gW2[o]);
                            gb2 = fmaf((float)nq_in, lane == 0 ? gq[0] : lane == 1 ? gq[1] : lane == 2 ? gq[2] : gq[3], gb2);     // lanes 0..3
                            double pb[4];                          // the position gradient is the difference of the two sums
#pragma unroll
                            for (int k = 0; k < 4; ++k) pb[k] = k < 3 ? (double)w[k] * Y : 0.0;
                            spread_sum<4, HID>(pb, a);
                            const int cp = spread_first<4, HID>(a);
                            if (p.gpos && lane < 4 && cp < 3) {
                                float* dst = p.gpos + 3 * (size_t)oq + cp;
                                *dst = first_chunk ? (float)pb[0] : *dst + (float)pb[0];
                            }
                            constexpr int NV = NX <= 4 ? 4 : NX <= 8 ? 8 : 16;
                            float r[NV];
#pragma unroll
                            for (int k = 0; k < NV; ++k) r[k] = k < NX ? w[k < NX ? 3 + k : 0] * G : 0.f;
                            spread_sum<NV, HID>(r, a);
                            constexpr int LEFT = NV > HID ? NV / HID : 1;
                            const int first = spread_first<NV, HID>(a);
                            if (p.gfeat && lane < (NV < HID ? NV : HID)) {
#pragma unroll
                                for (int k = 0; k < LEFT; ++k) {
                                    if (first + k >= Fin) continue;
                                    float* dst = p.gfeat + (size_t)oq * Fin + first + k;
                                    *dst = first_chunk ? r[k] : *dst + r[k];
                                }
                            }
                        }
                    }
                    __syncwarp();
                    if (!BWD && p.count && part && split.sub == 0) p.count[qid] = first_chunk ? nin : p.count[qid] + nin;
                    qa = qb;
                }
            }
            __syncwarp();
        };

        // the stage fills with candidates that survive the pruning; a step that does not fit is taken again
        bool first_chunk = true, full = false;
        int nst = 0, before = -1;
        constexpr int SU = 4;
        static_assert(STAGE_CAP >= 32 * SU, "a step fits an empty stage");
        for (int k0 = 0;;) {
            const bool done = k0 >= sten.total;
            if (full || (done && (nst > 0 || first_chunk))) {
                process_chunk(nst, first_chunk);
                first_chunk = false;
                full = false;
                nst = 0;
                for (int k = lane; k < qe0 - qs0; k += 32) s_self[k] = -1;
                __syncwarp();
            }
            if (done) break;
            const int step = sten.total - k0 < 32 * SU ? sten.total - k0 : 32 * SU, before0 = before;
            float4 c4[SU];
            int src[SU];
            unsigned kept[SU];
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                c4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                src[u] = -1;
                if (32 * u >= step) continue;
                src[u] = sten.source(k0 + 32 * u, before, s_delta);
                if (k0 + 32 * u + lane < sten.total) c4[u] = __ldg(p.spos + checked(src[u], p.n, CHECK_SLOT));
            }
            int all = nst;
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                kept[u] = 0u;
                if (32 * u >= step) continue;
                frame.shift(p, c4[u]);
                const float ex = fmaxf(fmaxf(blo[0] - c4[u].x, c4[u].x - bhi[0]), 0.f);
                const float ey = fmaxf(fmaxf(blo[1] - c4[u].y, c4[u].y - bhi[1]), 0.f);
                const float ez = fmaxf(fmaxf(blo[2] - c4[u].z, c4[u].z - bhi[2]), 0.f);
                kept[u] = __ballot_sync(FULL, k0 + 32 * u + lane < sten.total && fmaf(ez, ez, fmaf(ey, ey, ex * ex)) <= p.r2_hi * 1.0001f);
                all += __popc(kept[u]);
            }
            if (all > STAGE_CAP) { full = true; before = before0; continue; }
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                if ((kept[u] >> lane) & 1u) {
                    const int slot = nst + __popc(kept[u] & lt_mask);
                    stage.put(slot, c4[u]);
                    if (src[u] >= qs0 && src[u] < qe0) s_self[src[u] - qs0] = slot;
                    const int id = checked(__float_as_int(c4[u].w), p.n, CHECK_POINT);
                    const float* xr = p.feat + (size_t)id * Fin;
                    float4* dst = reinterpret_cast<float4*>(s_x + slot * NX);
#pragma unroll
                    for (int i = 0; i < FQ; ++i)
                        dst[i] = (Fin & 3) == 0 ? __ldg(reinterpret_cast<const float4*>(xr) + i)
                                                : make_float4(4 * i < Fin ? __ldg(xr + 4 * i) : 0.f, 4 * i + 1 < Fin ? __ldg(xr + 4 * i + 1) : 0.f,
                                                              4 * i + 2 < Fin ? __ldg(xr + 4 * i + 2) : 0.f, 4 * i + 3 < Fin ? __ldg(xr + 4 * i + 3) : 0.f);
                    if constexpr (BWD) {
                        const float* gr = p.gy + (size_t)id * Fout;
                        s_g[slot] = make_float4(__ldg(gr), Fout > 1 ? __ldg(gr + 1) : 0.f, Fout > 2 ? __ldg(gr + 2) : 0.f, Fout > 3 ? __ldg(gr + 3) : 0.f);
                    }
                }
                nst += __popc(kept[u]);
            }
            k0 += 32 * SU;
        }
    };
    if constexpr (!BWD) {
        walk_unit(p, blockIdx.x, p.run, slice);
    } else {
        const unsigned units = ((unsigned)p.n + p.unit - 1) / p.unit;
        for (;;) {
            unsigned u = 0;
            if (lane == 0) u = blockIdx.x + gridDim.x * atomicAdd(s_drawn, 1u);
            u = __shfl_sync(FULL, u, 0);
            if (u >= units) break;
            walk_unit(p, (int)u, p.run, slice);
        }
    }

    if constexpr (BWD) {
        // warps -> CTA copy in shared memory -> one atomic per parameter entry and CTA
        float* gW1s = sG;
        float* gb1s = gW1s + HID * KP;
        float* gW2s = gb1s + HID;
        float* gb2s = gW2s + 4 * HID;
        if (ps == 0) {
#pragma unroll
            for (int k = 0; k < KP; ++k) atomicAdd(gW1s + a * KP + k, gW1[k]);
#pragma unroll
            for (int o = 0; o < 4; ++o) atomicAdd(gW2s + o * HID + a, gW2[o]);
            atomicAdd(gb1s + a, gb1);
        }
        if (lane < 4) atomicAdd(gb2s + lane, gb2);
        __syncthreads();
        for (int e = threadIdx.x; e < HID * KP; e += SM::THREADS) {
            const int i = e / KP, k = e % KP;
            if (k < K && p.gW1) atomicAdd(p.gW1 + i * K + k, gW1s[e]);
        }
        for (int e = threadIdx.x; e < HID; e += SM::THREADS) if (p.gb1) atomicAdd(p.gb1 + e, gb1s[e]);
        for (int e = threadIdx.x; e < Fout * HID; e += SM::THREADS) if (p.gW2) atomicAdd(p.gW2 + e, gW2s[e]);
        if (threadIdx.x < Fout && p.gb2) atomicAdd(p.gb2 + threadIdx.x, gb2s[threadIdx.x]);
    }
}

// parameter gradients start from zero (one launch)
__global__ void mlp_zero_kernel(float* a, int na, float* b, int nb, float* c, int nc, float* d, int nd) {
    for (int k = threadIdx.x; k < na; k += blockDim.x) a[k] = 0.f;
    for (int k = threadIdx.x; k < nb; k += blockDim.x) b[k] = 0.f;
    for (int k = threadIdx.x; k < nc; k += blockDim.x) c[k] = 0.f;
    for (int k = threadIdx.x; k < nd; k += blockDim.x) d[k] = 0.f;
}

template <int HID, int FQ, bool BWD, bool MI>
static tiga_status launch_mlp_t(const RadiusParams& p, cudaStream_t s) {
    using SM = MlpSmem<HID, FQ, BWD>;
    auto kern = radius_mlp_kernel<HID, FQ, BWD, MI>;
    if (SM::TOTAL > 48 * 1024) TIGA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SM::TOTAL));
    static_assert(SM::TOTAL <= 227 * 1024, "one CTA per SM");
    const unsigned need = unit_count(p), cap = 148u * mlp_warps_per_sm<FQ, BWD>() / SM::WARPS;
    kern<<<counted(BWD && need > cap ? cap : need), SM::THREADS, SM::TOTAL, s>>>(p);
    return launch_status();
}

template <int HID, bool BWD, bool MI>
static tiga_status launch_mlp_k(const RadiusParams& p, cudaStream_t s) {
    switch ((p.Fin + 3) / 4) {
        case 1: return launch_mlp_t<HID, 1, BWD, MI>(p, s);
        case 2: return launch_mlp_t<HID, 2, BWD, MI>(p, s);
        case 3: return launch_mlp_t<HID, 3, BWD, MI>(p, s);
        default: return launch_mlp_t<HID, 4, BWD, MI>(p, s);
    }
}

template <bool BWD>
static tiga_status launch_mlp(const RadiusParams& p, int hidden, cudaStream_t s) {
    bool mi = false;
    for (int d = 0; d < 3; ++d) mi = mi || (p.periodic[d] && p.nc[d] <= 3);
    if (hidden == 8) return mi ? launch_mlp_k<8, BWD, true>(p, s) : launch_mlp_k<8, BWD, false>(p, s);
    if (hidden == 16) return mi ? launch_mlp_k<16, BWD, true>(p, s) : launch_mlp_k<16, BWD, false>(p, s);
    return mi ? launch_mlp_k<32, BWD, true>(p, s) : launch_mlp_k<32, BWD, false>(p, s);
}

static tiga_status mlp_common(RadiusParams* p, const float* pos, const float* feat, int64_t n, float r, const tiga_box* box,
                              const tiga_edge_mlp* mlp, void* ws, size_t ws_bytes, int32_t** fill, RadiusLayout* lay) {
    if (!mlp) return TIGA_ERR_INVALID_ARG;
    if (mlp->f_in < 1 || mlp->f_out < 1 || mlp->hidden < 1) return TIGA_ERR_INVALID_ARG;
    if (mlp->f_in > 13 || mlp->f_out > 4 || (mlp->hidden != 8 && mlp->hidden != 16 && mlp->hidden != 32)) return TIGA_ERR_UNSUPPORTED;
    if (!mlp->W1 || !mlp->b1 || !mlp->W2 || !mlp->b2) return TIGA_ERR_INVALID_ARG;
    tiga_status st = fill_params(p, n, r, box);
    if (st != TIGA_OK) return st;
    if (n > 0 && (!pos || !aligned16(pos) || !feat || !aligned16(feat))) return TIGA_ERR_INVALID_ARG;
    if (!ws || !aligned16(ws) || ws_bytes < tiga_radius_workspace_bytes(n, mlp->f_in, r, box, 0)) return TIGA_ERR_WORKSPACE;
    cut_cells(*p, 148 * 84);             // a query costs more here: finer slices
    *lay = carve_radius(p, ws, fill);
    p->pos = pos; p->feat = feat; p->F = mlp->f_in; p->Fin = mlp->f_in; p->Fout = mlp->f_out;
    p->W1 = mlp->W1; p->b1 = mlp->b1; p->W2 = mlp->W2; p->b2 = mlp->b2;
    return TIGA_OK;
}

}  // namespace tiga

using namespace tiga;

extern "C" tiga_status tiga_apply_radius_mlp(const float* pos, const float* feat, int64_t n, float r, const tiga_box* box,
                                             const tiga_edge_mlp* mlp, float* out, int32_t* count,
                                             void* ws, size_t ws_bytes, void* stream) {
    RadiusParams p{};
    int32_t* fill;
    RadiusLayout lay;
    tiga_status st = mlp_common(&p, pos, feat, n, r, box, mlp, ws, ws_bytes, &fill, &lay);
    if (st != TIGA_OK) return st;
    if (n == 0) return TIGA_OK;
    if (!out || !aligned16(out)) return TIGA_ERR_INVALID_ARG;
    p.out = out; p.count = count;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    st = run_binning(p, fill, lay.nblocks, s);
    if (st != TIGA_OK) return st;
    return launch_mlp<false>(p, mlp->hidden, s);
}

extern "C" tiga_status tiga_apply_radius_mlp_backward(const float* pos, const float* feat, int64_t n, float r, const tiga_box* box,
                                                      const tiga_edge_mlp* mlp, const float* grad_out,
                                                      float* grad_feat, float* grad_pos,
                                                      float* grad_W1, float* grad_b1, float* grad_W2, float* grad_b2,
                                                      void* ws, size_t ws_bytes, int reuse_plan, void* stream) {
    RadiusParams p{};
    int32_t* fill;
    RadiusLayout lay;
    tiga_status st = mlp_common(&p, pos, feat, n, r, box, mlp, ws, ws_bytes, &fill, &lay);
    if (st != TIGA_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int K = 3 + mlp->f_in;
    mlp_zero_kernel<<<counted(1), 256, 0, s>>>(grad_W1, grad_W1 ? mlp->hidden * K : 0, grad_b1, grad_b1 ? mlp->hidden : 0,
                                               grad_W2, grad_W2 ? mlp->f_out * mlp->hidden : 0, grad_b2, grad_b2 ? mlp->f_out : 0);
    if (launch_status() != TIGA_OK) return TIGA_ERR_CUDA;
    if (n == 0) return TIGA_OK;
    if (!grad_out || !aligned16(grad_out)) return TIGA_ERR_INVALID_ARG;
    p.gy = grad_out; p.gfeat = grad_feat; p.gpos = grad_pos;
    p.gW1 = grad_W1; p.gb1 = grad_b1; p.gW2 = grad_W2; p.gb2 = grad_b2;
    if (!reuse_plan) {
        st = run_binning(p, fill, lay.nblocks, s);
        if (st != TIGA_OK) return st;
    }
    return launch_mlp<true>(p, mlp->hidden, s);
}

namespace tiga { unsigned check_status_radius_mlp(bool reset) { return read_check_status(reset); } }
