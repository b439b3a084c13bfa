// Traversal that consumes a pair where it is accepted, by groups of queries (radius_group.cuh): the lanes of a query add the
// messages of its accepted candidates in registers.  Nothing is gathered, no atomics.  The messages are those of
// radius_direct.cuh, with GROUP_CAP and GROUP_WARPS in the places of CAP and WARPS where cells hold several points.
#pragma once
#include "radius_direct.cuh"
#include "radius_group.cuh"
#include <type_traits>

namespace tiga {

template <typename Msg, bool SPARSE> struct GroupDirectSmem {
    using Stage = std::conditional_t<SPARSE, GroupStage<256, 560>, GroupStage<Msg::GROUP_CAP, 1088>>;
    static constexpr int WARPS = SPARSE ? 24 : Msg::GROUP_WARPS;
    static constexpr int STAGED = Msg::STAGED, STAGE_BYTES = Stage::BYTES;
    static constexpr int FEAT_STRIDE = Stage::SLOTS;                        // the entry of the far slot stays zero
    static constexpr int PER_WARP = STAGE_BYTES + STAGED * FEAT_STRIDE * 4;
    static_assert(PER_WARP % 16 == 0, "the stage is accessed as 16-byte vectors");
    static_assert(DirectSmem<Msg>::PER_WARP <= PER_WARP, "crowded cells take the cells' form");
};

// COUNT: the numbers of neighbours are wanted.
template <typename Msg, bool SPARSE, bool COUNT>
__device__ __forceinline__ bool direct_group(const RadiusParams& p, typename GroupDirectSmem<Msg, SPARSE>::Stage& st, float* s_feat, const int (&cell)[3], const int run, const int qs, const int nq) {
    using SM = GroupDirectSmem<Msg, SPARSE>;
    constexpr int OUT = Msg::OUT, NF = Msg::STAGED;
    constexpr unsigned FULL = 0xffffffffu;
    using Stage = typename SM::Stage;
    const int lane = threadIdx.x & 31;
    const Msg msg(p);
    Group<Stage> grp(p, st, cell, run, qs, nq);

    // the lane's query and its sums
    const int q = lane >> grp.lsh, lpq = 1 << grp.lsh, sub = lane & (lpq - 1);
    const float4 qv = grp.query(q < nq ? q : 0);
    const f32x2 qx2 = dup2(qv.x), qy2 = dup2(qv.y), qz2 = dup2(qv.z);
    f32x2 acc2[OUT];
    int cnt = 0;
#pragma unroll
    for (int f = 0; f < OUT; ++f) acc2[f] = 0ull;
    // A list's terms are added up by themselves, and so are the sums of eight lists: however long the stencil, no partial sum runs
    // long (rms error over 24 k positive terms 0.6e-7 of their magnitude; 5.7e-7 with one running sum per lane and half, 1.4e-7 in cells).
    // Most groups have one list per query; the others keep these sums in local memory, as registers are short, and add them up behind a list (4.1 M
    // Lennard-Jones particles 1232 us with and without; in front of it 1239; in registers, which spills in the loop below, 1307).
    volatile f32x2 sum8[OUT], sums[OUT];
    int folds = 0;
    auto fold = [&]() {
#pragma unroll
        for (int f = 0; f < OUT; ++f) {
            f32x2 s = acc2[f];
            if (folds & 7) s = add2(sum8[f], s);
            if ((folds & 7) < 7) sum8[f] = s;
            else sums[f] = folds > 7 ? add2(sums[f], s) : s;
            acc2[f] = 0ull;
        }
        ++folds;
    };

    for (int k0 = 0; k0 < grp.sten.total; k0 += Stage::CAPACITY) {
        const int ns = grp.stage(k0);
        if (ns == 0) return false;
        if constexpr (NF > 0) {
            for (int b = lane; b - lane < ns; b += 128) {          // four rows in flight
                float x[4][NF];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int id = b + 32 * u < ns ? __float_as_int(grp.st.c[b + 32 * u].w) : -1;
#pragma unroll
                    for (int f = 0; f < NF; ++f) x[u][f] = 0.f;
                    if (id < 0) continue;
                    const float* xr = p.feat + (size_t)(unsigned)checked(id, p.n, CHECK_POINT) * NF;
                    if constexpr (NF == 4) {
                        const float4 x4 = __ldg(reinterpret_cast<const float4*>(xr));
                        x[u][0] = x4.x; x[u][1] = x4.y; x[u][2] = x4.z; x[u][3] = x4.w;
                    } else {
#pragma unroll
                        for (int f = 0; f < NF; ++f) x[u][f] = __ldg(xr + f);
                    }
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (b + 32 * u >= ns) continue;
#pragma unroll
                    for (int f = 0; f < NF; ++f) s_feat[f * SM::FEAT_STRIDE + b + 32 * u] = x[u][f];
                }
            }
        }
        GroupMask<Stage::WORDS> mask;
        grp.test(ns, k0, mask);
        grp.lists(ns, mask, [&](const int first, const int end) {
            for (int j = first + 2 * sub; j < end; j += 2 * lpq) {
                const unsigned two = *reinterpret_cast<const unsigned*>(grp.st.list + j);
                unsigned sa = two & 0xffffu, sb = two >> 16;
                const float4 ca = *reinterpret_cast<const float4*>(reinterpret_cast<const unsigned char*>(st.c) + sa);
                const float4 cb = *reinterpret_cast<const float4*>(reinterpret_cast<const unsigned char*>(st.c) + sb);
                const f32x2 dx = sub2(qx2, pack2(ca.x, cb.x)), dy = sub2(qy2, pack2(ca.y, cb.y)), dz = sub2(qz2, pack2(ca.z, cb.z));
                float da, db;
                unpack2(fma2(dz, dz, fma2(dy, dy, mul2(dx, dx))), da, db);
                bool in_a = da <= p.r2_mid, in_b = db <= p.r2_mid;
                const float ea = fabsf(da - p.r2_mid), eb = fabsf(db - p.r2_mid);
                if (fminf(ea, eb) <= p.r2_band) {                  // within the fp32 error band around the cutoff: decided in fp64
                    if (ea <= p.r2_band) in_a = exact_pair(p, __float_as_int(qv.w), __float_as_int(ca.w));
                    if (eb <= p.r2_band) in_b = exact_pair(p, __float_as_int(qv.w), __float_as_int(cb.w));
                }
                if (!in_a) { da = Msg::OUTSIDE; sa = 16 * Stage::FAR; }
                if (!in_b) { db = Msg::OUTSIDE; sb = 16 * Stage::FAR; }
                if (COUNT) cnt += (int)in_a + (int)in_b;
                msg.template pair<SM::FEAT_STRIDE>(acc2, da, db, dx, dy, dz, reinterpret_cast<const float*>(reinterpret_cast<const unsigned char*>(s_feat) + (sa >> 2)),
                         reinterpret_cast<const float*>(reinterpret_cast<const unsigned char*>(s_feat) + (sb >> 2)));
            }
        }, fold);
        if (grp.sten.total - k0 > Stage::CAPACITY + 128) fold();   // (a short last stage adds little: to the piece before)
    }
#pragma unroll
    for (int f = 0; f < OUT; ++f) {
        if (folds & 7) acc2[f] = add2(sum8[f], acc2[f]);
        if (folds > 7) acc2[f] = add2(sums[f], acc2[f]);
    }
    float acc[OUT];
#pragma unroll
    for (int f = 0; f < OUT; ++f) { float lo, hi; unpack2(acc2[f], lo, hi); acc[f] = lo + hi; }
    for (int o = 1; o < lpq; o <<= 1) {
#pragma unroll
        for (int f = 0; f < OUT; ++f) acc[f] += __shfl_xor_sync(FULL, acc[f], o);
        if (COUNT) cnt += __shfl_xor_sync(FULL, cnt, o);
    }
    if (q < nq && sub == 0) {
        const int qid = checked(__float_as_int(qv.w), p.n, CHECK_POINT);
#pragma unroll
        for (int f = 0; f < OUT; ++f) acc[f] = msg.scale(f, acc[f]);
        float* o = p.out + (size_t)qid * OUT;
        if constexpr (OUT == 4) {
            *reinterpret_cast<float4*>(o) = make_float4(acc[0], acc[1], acc[2], acc[3]);
        } else {
#pragma unroll
            for (int f = 0; f < OUT; ++f) o[f] = acc[f];
        }
        if (COUNT) p.count[qid] = cnt;
    }
    return true;
}

// What a kernel of groups does with clustered inputs.  Slices sort candidates out beforehand, and short ones spread over more warps than units of
// groups do; but of these kernels fewer warps run at once than of the one for slices alone.  (us, cells / groups, full units as slices where sparse /
// this rule, F = 1: 40 k clustered points, one per cell on average 256 / 431 / 260, eight 418 / 518 / 446.  200 k, one 1861 / 1738, eight 3144 / 3540;
// as cells and slices in this kernel 1843 and 3780.  A surface of 50 k points, 32 a cell, 82 / 102.)
enum class Clustered {
    Groups,        // nothing: many dense units, whose groups keep the machine busy, lose less than slices at this occupancy
    Units,         // many sparse units: those with a full cell as slices
    Cells,         // fewer units than two rounds of the machine: the whole input as cells and slices, by units of that form, when more than a quarter of
                   // the points lie in cells that stand out (RadiusParams::full; a sixteenth: a slab of 40 points a cell, 20 k points, 70 -> 87 us)
};

template <typename Msg, bool SPARSE, Clustered MODE, bool COUNT>
__global__ void __launch_bounds__(32, (GroupDirectSmem<Msg, SPARSE>::WARPS)) radius_group_kernel(const __grid_constant__ RadiusParams p, const int unit) {
    using SM = GroupDirectSmem<Msg, SPARSE>;
    extern __shared__ __align__(16) unsigned char s_raw[];
    if constexpr (MODE == Clustered::Cells) {
        if (*p.crowded > p.n >> 2) {
            auto slice = [&](const int (&cell)[3], const int run, const int qs, const int qe) { direct_slice<Msg, false>(p, cell, run, qs, qe, s_raw); };
            if (blockIdx.x * (long long)p.unit < p.n) walk_unit(p, blockIdx.x, p.run, slice);
            return;
        }
        if (blockIdx.x * (long long)unit >= p.n) return;
    }
    const GroupUnit work(p, blockIdx.x, unit);
    if constexpr (MODE == Clustered::Units) {
        if (work.full(p)) {
            work.walk(p, [&](const int (&cell)[3], const int run, const int qs, const int nq) {
                direct_slice<Msg, false>(p, cell, run, qs, qs + nq, s_raw);
                return true;
            });
            return;
        }
    }
    float* s_feat = reinterpret_cast<float*>(s_raw + SM::STAGE_BYTES);                   // [STAGED][FEAT_STRIDE]
    if (threadIdx.x < SM::STAGED) s_feat[threadIdx.x * SM::FEAT_STRIDE + SM::Stage::FAR] = 0.f;
    typename SM::Stage st(s_raw);
    const int end = p.n - work.begin < unit ? p.n : work.begin + unit;
    work.walk(p, [&](const int (&cell)[3], const int run, const int qs, const int nq) {
        if (direct_group<Msg, SPARSE, COUNT>(p, st, s_feat, cell, run, qs, nq)) return true;
        st.wait(COPY_TRIES);                                       // no copy outlives the warp, unless another limit is over
        give_up(p, Msg::OUT, qs, end);
        return false;
    });
}

template <typename Msg, bool SPARSE, Clustered MODE>
static tiga_status launch_direct_group(const RadiusParams& p, cudaStream_t s) {
    constexpr int smem = GroupDirectSmem<Msg, SPARSE>::PER_WARP;
    static_assert(smem <= 48 * 1024, "no attribute needed");
    auto kern = p.count ? radius_group_kernel<Msg, SPARSE, MODE, true> : radius_group_kernel<Msg, SPARSE, MODE, false>;
    const int unit = group_unit(p.n);
    RadiusParams q = p;
    // (half of the groups' unit at least: warps without work cost 30 k uniform points a microsecond)
    if (MODE == Clustered::Cells) q.unit = p.unit < unit / 2 ? unit / 2 : p.unit < unit ? p.unit : unit;
    else q.unit = unit;
    kern<<<counted(unit_count(q)), 32, smem, s>>>(q, unit);
    return launch_status();
}

// Groups or cells and slices (radius_direct.cuh).  Groups need points that fill them: where cells hold less than 0.7 points on average
// the input is a surface or clustered, and cells win (us, cells / groups: 100 k surface points, 16 neighbours 73 / 77; 40 k clustered
// points 231 / 272).  Uniform points: 1 M, 32 neighbours, F = 1 392 / 367, F = 4 458 / 378; 4 neighbours, F = 1 288 / 239; 300 k,
// 8 neighbours, F = 3 151 / 121; 30 k, 45 neighbours, F = 3 63 / 47.  Inputs that leave the machine half empty either way: 4 k, 16
// neighbours, F = 1 24.3 / 25.2, but dense ones gain (Lennard-Jones, 1728 particles 24.9 / 23.7).
// Inputs with the explicit minimum image take cells: their tests are scalar either way, and groups sort no candidate out first (1 k points in three
// cells a side, F = 1 78 / 162, Lennard-Jones 80 / 158; 8 k 695 / 1319; only 24 k points in one cell gained, 4287 / 3628).
template <typename Msg, bool MI>
static tiga_status launch_direct_t(const RadiusParams& p, cudaStream_t s) {
    if constexpr (!MI) {
        if (group_lengths(p) && 10LL * p.n >= 7LL * p.ncells && (p.n >= 8192 || p.n >= 8LL * p.ncells)) {
            if (p.n <= 2LL * GROUP_PLACES * GROUP)
                return group_sparse(p) ? launch_direct_group<Msg, true, Clustered::Cells>(p, s) : launch_direct_group<Msg, false, Clustered::Cells>(p, s);
            return group_sparse(p) ? launch_direct_group<Msg, true, Clustered::Units>(p, s) : launch_direct_group<Msg, false, Clustered::Groups>(p, s);
        }
    }
    return launch_direct_slices<Msg, MI>(p, s);
}

}  // namespace tiga
