// Candidate test of the traversals that consume a pair where it is accepted: the frame of a run of cells, its
// stencil as candidate ranges, the stage and the test.
//
// The stage holds the candidates' coordinates by component, so that a test reads two candidates with one 64-bit load
// per component and forms both squared distances with packed instructions.  Every query of the run gets
// LPQ = 32 / queries lanes.  A lane keeps its query in registers, walks the candidate pairs sub, sub + LPQ, ... and
// shifts one sign bit per candidate into a mask, which costs about seven instructions per 32 tests; only accepted
// candidates (one in four at the usual density) are looked at again, two at a time per lane.
#pragma once
#include "radius_shared.cuh"

namespace tiga {

constexpr int TEST_BATCH = 16;         // queries tested together: at least two lanes each
constexpr int TEST_LPQ = 8;            // most lanes per query
constexpr int TEST_PAD = 40;           // sentinels behind the staged candidates (a test reads up to 4 TEST_LPQ + 1 further)

// Frame of a run of cells along x (one cell; several where cells hold a point or two): in a dimension whose stencil
// wraps around a face, every coordinate above the threshold moves down by the box length (the wrapped cell at
// the top when the run touches the lower face; the run and its lower neighbour when it touches the upper face).
// Both shifts are exact in fp32.
struct RunFrame {
    int c[3];
    bool face;
    float thr[3];
    __device__ __forceinline__ RunFrame(const RadiusParams& p, const int (&cell)[3], const int run) {
        c[0] = cell[0]; c[1] = cell[1]; c[2] = cell[2];
        face = false;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            thr[d] = INFINITY;
            const int last = d == 0 ? c[0] + run - 1 : c[d];
            if (p.periodic[d] && p.nc[d] >= 4) {
                if (c[d] == 0) { thr[d] = ((float)(last - c[d]) + 2.5f) * p.hcell[d]; face = true; }
                else if (last == p.nc[d] - 1) { thr[d] = 1.5f * p.hcell[d]; face = true; }
            }
        }
    }
    __device__ __forceinline__ void shift(const RadiusParams& p, float4& v) const {
        if (face) {
            if (v.x > thr[0]) v.x -= p.len[0];
            if (v.y > thr[1]) v.y -= p.len[1];
            if (v.z > thr[2]) v.z -= p.len[2];
        }
    }
};

// The run's stencil: lanes 0..8 hold the (y, z) rows over the run's x range, lanes 9..17 the cell that row
// reaches around a periodic x face.  begin: flattened position of the lane's range.  Returns the source of its first position.
// divide: how the row is found.  Without a division is shorter, but the compiler then shares the 72 registers of the list kernels out in another way
// (see there).
static __device__ __forceinline__ int stencil_range(const RadiusParams& p, const int (&c)[3], const int run, const bool divide, int& begin, int& len, int& total) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int row = lane < 9 ? lane : lane - 9;
    const int oz = divide ? row / 3 - 1 : row >= 6 ? 1 : row >= 3 ? 0 : -1, oy = divide ? row % 3 - 1 : row - 3 * oz - 4;
    int y = c[1] + oy, z = c[2] + oz, cs = 0;
    bool ok = lane < 18;
    if (p.nc[1] == 1) { ok = ok && oy == 0; y = 0; }
    else if (y < 0) { if (p.periodic[1]) y += p.nc[1]; else ok = false; }
    else if (y >= p.nc[1]) { if (p.periodic[1]) y -= p.nc[1]; else ok = false; }
    if (p.nc[2] == 1) { ok = ok && oz == 0; z = 0; }
    else if (z < 0) { if (p.periodic[2]) z += p.nc[2]; else ok = false; }
    else if (z >= p.nc[2]) { if (p.periodic[2]) z -= p.nc[2]; else ok = false; }
    const int lo = c[0] - 1, hi = c[0] + run, top = p.nc[0] - 1;
    int xa = lo > 0 ? lo : 0, xb = hi < top ? hi : top;
    if (lane >= 9) {
        xa = xb = lo < 0 ? top : 0;
        ok = ok && p.periodic[0] && top > 0 && (lo < 0 || hi > top);
    }
    len = 0;
    if (ok) {
        const int id = (z * p.nc[1] + y) * p.nc[0];
        cs = p.cell_start[id + xa];
        len = p.cell_start[id + xb + 1] - cs;
    }
    begin = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULL, begin, o);
        if (lane >= o) begin += t;
    }
    total = __shfl_sync(FULL, begin, 31);
    begin -= len;
    return cs;
}

// The stencil by position: s_delta maps a flattened position to its source.
struct RunStencil {
    int begin, len, total;
    __device__ __forceinline__ RunStencil(const RadiusParams& p, const int (&c)[3], const int run, int* s_delta, const bool divide = false) {
        const int lane = threadIdx.x & 31;
        const int cs = stencil_range(p, c, run, divide, begin, len, total);
        const unsigned some = __ballot_sync(0xffffffffu, len > 0);
        if (len > 0) s_delta[__popc(some & ((1u << lane) - 1u))] = cs - begin;
        __syncwarp();
    }
    // source of flattened position k0 + lane; `before` counts the ranges that began before k0 (start with -1).  The
    // ranges that begin in this window of 32 positions set one bit each: the bits at and below a lane count up to
    // the lane's range.
    __device__ __forceinline__ int source(const int k0, int& before, const int* s_delta) const {
        const int lane = threadIdx.x & 31;
        const int w0 = begin - k0;
        const unsigned starts = __reduce_or_sync(0xffffffffu, len > 0 && w0 >= 0 && w0 < 32 ? 1u << w0 : 0u);
        const int r = before + __popc(starts & (0xffffffffu >> (31 - lane)));
        before += __popc(starts);
        return s_delta[r] + k0 + lane;
    }
};

// Candidates by component; pairs of neighbouring slots are read as one f32x2.
template <int CAP>
struct TestStage {
    static constexpr int SLOTS = CAP + TEST_PAD;
    static constexpr int BYTES = SLOTS * 16;
    float *x, *y, *z;
    int* id;
    __device__ __forceinline__ explicit TestStage(unsigned char* base) {
        x = reinterpret_cast<float*>(base);
        y = x + SLOTS;
        z = y + SLOTS;
        id = reinterpret_cast<int*>(z + SLOTS);
    }
    __device__ __forceinline__ void put(const int slot, const float4& v) const {
        float* s = x + slot;
        s[0] = v.x; s[SLOTS] = v.y; s[2 * SLOTS] = v.z; s[3 * SLOTS] = v.w;
    }
    __device__ __forceinline__ void seal(const int ns) const {
        for (int k = threadIdx.x & 31; k < TEST_PAD; k += 32) { x[ns + k] = -FAR_AWAY; y[ns + k] = -FAR_AWAY; z[ns + k] = -FAR_AWAY; id[ns + k] = -1; }
    }
};

// How the lanes of the warp are shared out to a batch of nq <= TEST_BATCH queries: lane -> (query q, sub), LPQ lanes per
// query.
struct LaneSplit {
    int lpq, q, sub;
    unsigned inv;                  // ceil(65536 / lpq): x * inv >> 16 is x / lpq for every x that occurs
    bool active;
    __device__ __forceinline__ explicit LaneSplit(const int nq) {
        const int lane = threadIdx.x & 31;
        lpq = nq <= 4 ? 8 : nq == 5 ? 6 : nq == 6 ? 5 : nq <= 8 ? 4 : nq <= 10 ? 3 : 2;      // 32 / nq, at most TEST_LPQ
        inv = lpq == 8 ? 8192u : lpq == 6 ? 10923u : lpq == 5 ? 13108u : lpq == 4 ? 16384u : lpq == 3 ? 21846u : 32768u;
        q = (int)(lane * inv >> 16);
        sub = lane - q * lpq;
        active = q < nq;
    }
};

// Mask words of a lane: word 2 g + b holds the tests of candidates 2 (sub + lpq (32 g + k)) + b, k = 0..31 from the top bit
// down, so a set bit is a candidate slot with one multiply-add.  Two groups cover 64 pairs a lane: the whole stage of
// 256 at two lanes per query.
constexpr int TEST_GROUP = 32;

// Tests query (qx, qy, qz) of every lane against the ns staged candidates: a bit is set when the candidate lies within
// the cutoff or in the fp32 error band around it.
// delta(component, query coordinate, candidate coordinate) is the scalar displacement of the explicit-minimum-image form.
template <bool MI, int CAP, typename Delta>
__device__ __forceinline__ void test_candidates(const RadiusParams& p, const TestStage<CAP>& st, const int ns, const LaneSplit& split,
                                                const float qx, const float qy, const float qz, unsigned (&mask)[4], Delta delta) {
    static_assert(CAP <= 4 * 2 * TEST_GROUP, "two groups of tests cover the stage");
    constexpr int NEXT = TestStage<CAP>::SLOTS / 2;                              // next component, in pairs
    static_assert(TestStage<CAP>::SLOTS % 2 == 0, "pairs");
    const int steps = ((int)((((ns + 1) >> 1) + split.lpq - 1) * split.inv >> 16) + 1) & ~1;      // even
    const f32x2 qx2 = dup2(qx), qy2 = dup2(qy), qz2 = dup2(qz), neg = dup2(-p.r2_hi);
    const f32x2* pc = reinterpret_cast<const f32x2*>(st.x) + split.sub;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
        const int here = steps - TEST_GROUP * g < TEST_GROUP ? steps - TEST_GROUP * g : TEST_GROUP;
        unsigned m0 = 0u, m1 = 0u;
        if (here > 0) {
            for (int s = 0; s < here; s += 2) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    float t0, t1;
                    const f32x2 cx = pc[0], cy = pc[NEXT], cz = pc[2 * NEXT];
                    pc += split.lpq;
                    if constexpr (!MI) {
                        const f32x2 dx = sub2(qx2, cx), dy = sub2(qy2, cy), dz = sub2(qz2, cz);
                        unpack2(fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, neg))), t0, t1);
                    } else {
                        float x0, x1, y0, y1, z0, z1;
                        unpack2(cx, x0, x1); unpack2(cy, y0, y1); unpack2(cz, z0, z1);
                        const float ax = delta(0, qx, x0), ay = delta(1, qy, y0), az = delta(2, qz, z0);
                        const float bx = delta(0, qx, x1), by = delta(1, qy, y1), bz = delta(2, qz, z1);
                        t0 = fmaf(az, az, fmaf(ay, ay, fmaf(ax, ax, -p.r2_hi)));
                        t1 = fmaf(bz, bz, fmaf(by, by, fmaf(bx, bx, -p.r2_hi)));
                    }
                    m0 = __funnelshift_l(__float_as_uint(t0), m0, 1);
                    m1 = __funnelshift_l(__float_as_uint(t1), m1, 1);
                }
            }
            m0 = split.active ? m0 << (TEST_GROUP - here) : 0u;
            m1 = split.active ? m1 << (TEST_GROUP - here) : 0u;
        }
        mask[2 * g] = m0;
        mask[2 * g + 1] = m1;
    }
}

// clears the bit of staged slot `slot` (the query itself) where this lane tested it
static __device__ __forceinline__ void drop_candidate(unsigned (&mask)[4], const LaneSplit& split, const int slot) {
    const int pair = slot >> 1;
    const int step = (int)((unsigned)pair * split.inv >> 16);               // pair / lpq
    if (slot < 0 || pair - step * split.lpq != split.sub) return;
    const unsigned bit = 0x80000000u >> (step & 31);
    const int w = (step >> 5) * 2 + (slot & 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) if (k == w) mask[k] &= ~bit;
}

}  // namespace tiga
