// Lennard-Jones over the generated radius relation (paper Section 4.9): fused cell-list traversal, pair force and
// energy, sum reducer (radius_group_direct.cuh).
//
// Every row walks its full neighbourhood, which forms each unordered pair twice but needs no atomics, no memset and no
// list in memory, and is reproducible.  Bound by instruction issue (two thirds of the slots): per group of 15.7 particles about 880 warp
// instructions find and stage 470 candidates, 720 test them, 670 gather the accepted ones into lists, 830 form the forces.
// 4.1 M particles with binning 1456 -> 1238 us against cells of 12.6 particles tested with packed fp32 instructions (300 instead of 200
// warp instructions per particle); 20 warps per SM (what the stage allows) measured faster than 24 with 80 registers (1272 us),
// units of 32 points faster than 16 (1262 us).
#include "radius_group_direct.cuh"

namespace tiga {

struct LjMsg {
    static constexpr int CAP = 256, STAGED = 0, OUT = 4, WARPS = 28, GROUP_CAP = 512, GROUP_WARPS = 20;
    static constexpr float OUTSIDE = INFINITY;             // reciprocal 0: no force, no energy
    float s2, force, energy;
    __device__ __forceinline__ explicit LjMsg(const RadiusParams& p) : s2(p.p1 * p.p1), force(24.f * p.p0), energy(2.f * p.p0) {}
    template <int>
    __device__ __forceinline__ void pair(f32x2 (&acc)[4], const float da, const float db, const f32x2 dx, const f32x2 dy, const f32x2 dz,
                                         const float*, const float*) const {
        const f32x2 inv = pack2(fast_rcp(da), fast_rcp(db));
        const f32x2 qq = mul2(dup2(s2), inv);
        const f32x2 q3 = mul2(mul2(qq, qq), qq);             // (s / d)^6
        const f32x2 en = fma2(q3, q3, mul2(q3, dup2(-1.f)));  // q3^2 - q3
        const f32x2 fs = mul2(fma2(q3, q3, en), inv);        // (2 q3^2 - q3) / d^2
        acc[0] = fma2(fs, dx, acc[0]); acc[1] = fma2(fs, dy, acc[1]); acc[2] = fma2(fs, dz, acc[2]);
        acc[3] = add2(acc[3], en);
    }
    __device__ __forceinline__ float scale(const int f, const float v) const { return (f < 3 ? force : energy) * v; }
};

tiga_status launch_lj(const RadiusParams& p, cudaStream_t s) {
    bool mi = false;
    for (int d = 0; d < 3; ++d) mi = mi || (p.periodic[d] && p.nc[d] <= 3);
    return mi ? launch_direct_t<LjMsg, true>(p, s) : launch_direct_t<LjMsg, false>(p, s);
}

}  // namespace tiga

namespace tiga { unsigned check_status_radius_lj(bool reset) { return read_check_status(reset); } }
