// Traversal that consumes a pair where it is accepted (test: radius_test.cuh): every query has its own lanes, and a
// lane adds the messages of its accepted candidates in registers.  No lists, no gathers, no atomics.
//
// Msg supplies the message:
//   CAP, WARPS      candidates the stage holds, and warps per SM
//   STAGED          features per point that are staged with the candidates
//   OUT             sums per query
//   OUTSIDE         squared distance given to a half that adds nothing (an absent or refused candidate); its features read as
//                   zero, and the message of that distance times zero must be zero (no decay with the distance is assumed:
//                   a Gaussian as wide as fp32 allows gives every distance the weight one)
//   Msg(p)          constants
//   pair<STRIDE>(...)  adds the messages of two accepted candidates to acc[OUT], one per half; STRIDE between staged features
//   scale(f, v)     the stored value of sum f
#pragma once
#include "radius_test.cuh"

namespace tiga {

template <typename Msg> struct DirectSmem {
    static constexpr int STAGE_CAP = Msg::CAP, STAGED = Msg::STAGED;
    static constexpr int STAGE_BYTES = TestStage<STAGE_CAP>::BYTES;
    static constexpr int FEAT_STRIDE = STAGE_CAP + 4;                       // the entry behind the stage stays zero
    static constexpr int FEAT_BYTES = STAGED * FEAT_STRIDE * 4;
    static constexpr int PER_WARP = (STAGE_BYTES + FEAT_BYTES + (QDENSE + 20) * 4 + 15) / 16 * 16;
};

// MI: some periodic dimension has three cells or fewer and uses the explicit minimum image.
template <typename Msg, bool MI>
__device__ __forceinline__ void direct_slice(const RadiusParams& p, const int (&cell)[3], const int run, const int qs0, const int qe0, unsigned char* s_raw) {
    using SM = DirectSmem<Msg>;
    constexpr int STAGE_CAP = SM::STAGE_CAP, OUT = Msg::OUT, NF = Msg::STAGED;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    unsigned char* base = s_raw + (size_t)(threadIdx.x >> 5) * SM::PER_WARP;
    const TestStage<STAGE_CAP> stage(base);
    float* s_feat = reinterpret_cast<float*>(base + SM::STAGE_BYTES);                   // [NF][FEAT_STRIDE]
    int* s_self = reinterpret_cast<int*>(base + SM::STAGE_BYTES + SM::FEAT_BYTES);      // staged slot of every query, or -1
    int* s_delta = s_self + QDENSE;

    const Msg msg(p);
    const bool mi0 = MI && p.periodic[0] && p.nc[0] <= 3, mi1 = MI && p.periodic[1] && p.nc[1] <= 3, mi2 = MI && p.periodic[2] && p.nc[2] <= 3;
    auto delta = [&](const int d, const float q, const float c4) -> float {
        const bool mi = d == 0 ? mi0 : d == 1 ? mi1 : mi2;
        return (MI && mi) ? mi_delta(q, c4, p.len[d], 0.5f * p.len[d]) : q - c4;
    };
    const unsigned lt_mask = (1u << lane) - 1u;
    const RunFrame frame(p, cell, run);
    const RunStencil sten(p, frame.c, run, s_delta);

    // bounding box of the queries: a candidate farther than the cutoff from it is not staged
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
    if (lane < NF) s_feat[lane * SM::FEAT_STRIDE + STAGE_CAP] = 0.f;
    __syncwarp();                            // staging sets the slot of a query from whichever lane holds its point

    auto process_chunk = [&](const int ns, const bool first_chunk) {
        stage.seal(ns);
        __syncwarp();
        // batches of one size, at most TEST_BATCH: a short last one would idle as many lanes as a full one keeps busy
        const int all = qe0 - qs0;
        const int per = all <= TEST_BATCH ? all : all <= 2 * TEST_BATCH ? (all + 1) >> 1 : TEST_BATCH;
        for (int qb0 = qs0; qb0 < qe0; qb0 += per) {
            const int nq = (qe0 - qb0 < per) ? qe0 - qb0 : per;
            const LaneSplit split(nq);
            float4 qv = p.spos[qb0 + (split.active ? split.q : 0)];
            frame.shift(p, qv);
            const int qid = checked(__float_as_int(qv.w), p.n, CHECK_POINT);
            unsigned mask[4];
            test_candidates<MI, STAGE_CAP>(p, stage, ns, split, qv.x, qv.y, qv.z, mask, delta);
            drop_candidate(mask, split, split.active ? s_self[qb0 - qs0 + split.q] : -1);
            f32x2 acc2[OUT];
            int cnt = 0;
#pragma unroll
            for (int f = 0; f < OUT; ++f) acc2[f] = 0ull;
            if (p.count) cnt = __popc(mask[0]) + __popc(mask[1]) + __popc(mask[2]) + __popc(mask[3]);
            // the lane's accepted candidates, two at a time; a lane moves on to its next word by itself, so the
            // warp makes as many trips as its busiest lane needs
            const f32x2 qx2 = dup2(qv.x), qy2 = dup2(qv.y), qz2 = dup2(qv.z);
            unsigned m = mask[0], m1 = mask[1], m2 = mask[2], m3 = mask[3];
            int word = 2 * split.sub, next = 1;                         // stage slot of bit 31 of the current word, step to the next
            while (m | m1 | m2 | m3) {
                if (m == 0u) { m = m1; m1 = m2; m2 = m3; m3 = 0u; word += next; next = 2 * TEST_GROUP * split.lpq - next; }
                if (m == 0u) continue;
                const int ka = __clz(m);
                m ^= 0x80000000u >> ka;
                const bool two = m != 0u;
                const int kb = two ? __clz(m) : ka;
                m &= 0x7fffffffu >> kb;
                const int sa = word + 2 * split.lpq * ka, sb = word + 2 * split.lpq * kb;
                const float *ca = stage.x + sa, *cb = stage.x + sb;
                constexpr int SL = TestStage<STAGE_CAP>::SLOTS;
                f32x2 dx, dy, dz;
                if constexpr (!MI) {
                    dx = sub2(qx2, pack2(ca[0], cb[0]));
                    dy = sub2(qy2, pack2(ca[SL], cb[SL]));
                    dz = sub2(qz2, pack2(ca[2 * SL], cb[2 * SL]));
                } else {
                    dx = pack2(delta(0, qv.x, ca[0]), delta(0, qv.x, cb[0]));
                    dy = pack2(delta(1, qv.y, ca[SL]), delta(1, qv.y, cb[SL]));
                    dz = pack2(delta(2, qv.z, ca[2 * SL]), delta(2, qv.z, cb[2 * SL]));
                }
                float da, db;
                unpack2(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), da, db);
                int fa = sa, fb = two ? sb : STAGE_CAP;              // where the halves read their features
                if (fmaxf(da, db) > p.r2_mid - p.r2_band) {        // within the fp32 error band of the cutoff: decided in fp64
                    if (da > p.r2_mid - p.r2_band && !exact_pair(p, qid, stage.id[sa])) { da = Msg::OUTSIDE; fa = STAGE_CAP; --cnt; }
                    if (two && db > p.r2_mid - p.r2_band && !exact_pair(p, qid, stage.id[sb])) { db = Msg::OUTSIDE; fb = STAGE_CAP; --cnt; }
                }
                if (!two) db = Msg::OUTSIDE;
                msg.template pair<SM::FEAT_STRIDE>(acc2, da, db, dx, dy, dz, s_feat + fa, s_feat + fb);
            }
            float acc[OUT];
#pragma unroll
            for (int f = 0; f < OUT; ++f) { float lo, hi; unpack2(acc2[f], lo, hi); acc[f] = lo + hi; }
            // sum over the lanes of a query, result in its lane with sub = 0
            auto query_sum = [&](auto v) {
#pragma unroll
                for (int o = 1; o < TEST_LPQ; o <<= 1) {
                    if (o >= split.lpq) break;
                    const auto other = __shfl_down_sync(FULL, v, o);
                    if (split.sub + o < split.lpq) v += other;
                }
                return v;
            };
#pragma unroll
            for (int f = 0; f < OUT; ++f) acc[f] = msg.scale(f, query_sum(acc[f]));
            if (p.count) cnt = query_sum(cnt);
            if (split.active && split.sub == 0) {
                float* o = p.out + (size_t)qid * OUT;
                if constexpr (OUT == 4) {
                    float4 v = make_float4(acc[0], acc[1], acc[2], acc[3]);
                    if (!first_chunk) { const float4 old = *reinterpret_cast<float4*>(o); v.x += old.x; v.y += old.y; v.z += old.z; v.w += old.w; }
                    *reinterpret_cast<float4*>(o) = v;
                } else {
#pragma unroll
                    for (int f = 0; f < OUT; ++f) o[f] = first_chunk ? acc[f] : o[f] + acc[f];
                }
                if (p.count) p.count[qid] = first_chunk ? cnt : p.count[qid] + cnt;
            }
        }
        __syncwarp();
    };

    // The stage fills with candidates that survive the pruning and is processed when the next step's survivors do
    // not fit (that step is then taken again), so the chunks are as full as the pruning allows: one chunk for all but
    // dense cells.
    bool first_chunk = true, full = false;
    int nst = 0;                                                             // candidates staged (warp uniform)
    int before = -1;                                                         // ranges that began before the step, minus one
    constexpr int SU = 4;                                                    // staging groups in flight
    static_assert(STAGE_CAP >= 32 * SU, "a step fits an empty stage");
    for (int k0 = 0;;) {
        const bool done = k0 >= sten.total;
        if (full || (done && (nst > 0 || first_chunk))) {                    // the one place a chunk is processed
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
        for (int u = 0; u < SU; ++u) {                                       // all loads of the step first
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
        float xf[SU][NF > 0 ? NF : 1];
        if constexpr (NF > 0) {
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                if (!((kept[u] >> lane) & 1u)) continue;
                const float* xr = p.feat + (size_t)(unsigned)checked(__float_as_int(c4[u].w), p.n, CHECK_POINT) * NF;
                if constexpr (NF == 4) {
                    const float4 v = __ldg(reinterpret_cast<const float4*>(xr));
                    xf[u][0] = v.x; xf[u][1] = v.y; xf[u][2] = v.z; xf[u][3] = v.w;
                } else {
#pragma unroll
                    for (int f = 0; f < NF; ++f) xf[u][f] = __ldg(xr + f);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < SU; ++u) {
            if ((kept[u] >> lane) & 1u) {
                const int slot = nst + __popc(kept[u] & lt_mask);
                stage.put(slot, c4[u]);
                if (src[u] >= qs0 && src[u] < qe0) s_self[src[u] - qs0] = slot;
#pragma unroll
                for (int f = 0; f < NF; ++f) s_feat[f * SM::FEAT_STRIDE + slot] = xf[u][f];
            }
            nst += __popc(kept[u]);
        }
        k0 += 32 * SU;
    }
}

template <typename Msg, bool MI>
__global__ void __launch_bounds__(TRAV_THREADS, Msg::WARPS / TRAV_WARPS) radius_direct_kernel(const __grid_constant__ RadiusParams p) {
    extern __shared__ __align__(16) unsigned char s_raw[];
    auto work = [&](const int (&cell)[3], const int run, const int qs, const int qe) { direct_slice<Msg, MI>(p, cell, run, qs, qe, s_raw); };
    walk_unit(p, blockIdx.x * TRAV_WARPS + (threadIdx.x >> 5), p.run, work);
}

template <typename Msg, bool MI>
static tiga_status launch_direct_slices(const RadiusParams& p, cudaStream_t s) {
    constexpr int smem = DirectSmem<Msg>::PER_WARP * TRAV_WARPS;
    auto kern = radius_direct_kernel<Msg, MI>;
    if (smem > 48 * 1024) TIGA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    kern<<<counted(unit_blocks(p)), TRAV_THREADS, smem, s>>>(p);
    return launch_status();
}

}  // namespace tiga
