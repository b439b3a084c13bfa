// Pieces of the generated-radius path shared by radius.cu (binning, Gaussian / distance /
// Lennard-Jones traversals) and radius_mlp.cu (edge-network message).
#pragma once
#include "common.cuh"
#include <math.h>

namespace tiga {

// one warp per CTA: units differ in work (0 to 3 cells), and a CTA holds its place until its last warp is done (four
// warps: forward of 1 M points, 32 neighbours, 725 instead of 557 us)
constexpr int TRAV_WARPS = 1;
constexpr int TRAV_THREADS = TRAV_WARPS * 32;
constexpr int STAGE_PAD = 32;           // sentinels behind the staged candidates: no bounds checks
constexpr int QB = 8;                   // queries per batch (kernels that run faster with four define their own width)
constexpr float FAR_AWAY = 1.0e18f;
constexpr int QSLICE = 16;              // most queries of a slice of a dense cell (cut_cells)
constexpr int QDENSE = QSLICE + QSLICE / 2;   // most queries of one piece of work
constexpr int UNIT_MAX = 32;            // most points per unit of work (at most 32: a lane each)
constexpr int RUN_CELLS = 8;            // longest run of cells along x that one warp covers
constexpr int GROUP_RUN = 16;           // most cells along x a group of queries spans
constexpr int RUN_QUERIES = 16;         // points a warp joins cells for
constexpr int COPY_TRIES = 1 << 20;     // looks at a staged copy, up to a microsecond each, before a traversal gives up
constexpr int SORT_DENSE = 256;         // a cell with more points than this is ordered by a sorting network, not by rank counting

struct RadiusParams {
    const float* pos;
    const float* feat;
    const float* gy;
    float* out;
    int32_t* count;
    float* gfeat;
    float* gpos;
    int n;
    int F;
    float r;
    float r2_lo, r2_hi;       // fp32 filter band around r^2
    float r2_mid, r2_band;    // its centre and half width
    double r2_exact;          // (double)r * (double)r
    float len[3];
    int periodic[3];
    int nc[3];
    float invh[3];
    float hcell[3];           // cell edge, len / nc
    int ncells;
    float p0, p1;             // message parameters
    // edge network (radius_mlp.cu): device pointers to W1 [H, 3+Fin], b1 [H], W2 [Fout, H], b2 [Fout]
    const float *W1, *b1, *W2, *b2;
    float *gW1, *gb1, *gW2, *gb2;
    int Fin, Fout;
    // plan (workspace)
    int32_t* cell;
    int32_t* cnt;
    int32_t* cell_start;
    int32_t* order_tmp;
    int32_t* order;
    float4* spos;             // positions in cell order, .w = original point id (bit pattern)
    int32_t* blocksum;
    int run;                  // cells along x that a warp joins at most
    int unit;                 // points per warp (walk_unit)
    int group_run;            // cells along x that a group of queries spans at most (walk_groups)
    int dense, slice;         // a cell with more than `dense` points is cut into slices of `slice` queries
    int* queue_n;             // length of the kNN queue (zeroed with the counts)
    int full;                 // a cell with more points than this stands out from the mean (full_cell)
    int* crowded;             // points in such cells (zeroed with the counts)
    int32_t* b_items;         // cells with more than SORT_DENSE points (queued by the scan), and how many
    int* b_count;
    // optional user copies of the plan
    int32_t* u_cell;
    int32_t* u_cell_start;
    int32_t* u_order;
#ifdef TIGA_CHECKED
    int copy_tries;           // in the place of COPY_TRIES
#endif
};

#ifdef TIGA_CHECKED
static __device__ __forceinline__ int copy_tries(const RadiusParams& p) { return p.copy_tries; }
#else
static __device__ __forceinline__ int copy_tries(const RadiusParams&) { return COPY_TRIES; }
#endif

struct RadiusLayout {
    size_t bytes;
    int nblocks;
};

// host side, defined in radius.cu
tiga_status fill_params(RadiusParams* p, long long n, float r, const tiga_box* box);
RadiusLayout carve_radius(RadiusParams* p, void* ws, int32_t** fill);
tiga_status run_binning(RadiusParams& p, int32_t* fill, int nblocks, cudaStream_t s);
// host side, defined in radius_lj.cu
tiga_status launch_lj(const RadiusParams& p, cudaStream_t s);

// cell coordinate of a point coordinate: one rounded product, clamped to the grid
static __device__ __forceinline__ int cell_coordinate(const RadiusParams& p, const float v, const int d) {
    const int k = (int)floorf(__fmul_rn(v, p.invh[d]));
    return k > p.nc[d] - 1 ? p.nc[d] - 1 : k < 0 ? 0 : k;
}

// The defining predicate in double precision (same operations as the plain definition).
static __device__ __noinline__ bool exact_within(const RadiusParams& p, const float4 a, const float4 b) {
    const float pa[3] = {a.x, a.y, a.z}, pb[3] = {b.x, b.y, b.z};
    double d2 = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        double t = __dsub_rn((double)pa[d], (double)pb[d]);
        if (p.periodic[d]) {
            const double L = (double)p.len[d];
            t = __dsub_rn(t, __dmul_rn(L, rint(__ddiv_rn(t, L))));
        }
        const double sq = __dmul_rn(t, t);
        d2 = (d == 0) ? sq : __dadd_rn(d2, sq);
    }
    return d2 <= p.r2_exact;
}

// The traversals share the points out by their place in cell order: unit u, one warp's work, is the cells whose first
// point lies in [u p.unit, (u + 1) p.unit), and of a cell with more than p.dense points the slices of p.slice queries that
// begin there.  So every warp has about p.unit queries whatever the density, empty cells cost nothing and a dense cell
// spreads over many warps, without a list of work items.  (Short slices: a dense cell's queries meet thousands of
// candidates each.)  Neighbouring cells along x are joined to runs of at most `run` cells and RUN_QUERIES points.
// work(first cell of the run, cells, first query, end)
template <typename Work>
static __device__ __forceinline__ void walk_unit(const RadiusParams& p, const int u, const int run, Work& work) {
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int i = u * p.unit + lane;
    const bool valid = lane < p.unit && i < p.n;
    int at = 0, qe = 0;                                         // cell of the lane's point, ten bits per coordinate; end of its queries
    bool dense = false, head = false;
    if (valid) {
        const float4 v = p.spos[i];
        const int x = cell_coordinate(p, v.x, 0), y = cell_coordinate(p, v.y, 1), z = cell_coordinate(p, v.z, 2);
        at = x | y << 10 | z << 20;
        const int id = (z * p.nc[1] + y) * p.nc[0] + x;
        const int cs = p.cell_start[id], ce = p.cell_start[id + 1];
        dense = ce - cs > p.dense;
        head = dense ? (i - cs) % p.slice == 0 : i == cs;
        qe = dense && i + p.slice < ce ? i + p.slice : ce;
    }
    unsigned left = __ballot_sync(FULL, head);                  // cells and slices of the unit not done yet
    qe |= dense ? 0x80000000 : 0;
    while (left) {
        const int a = __ffs(left) - 1;
        left &= left - 1u;
        const int first = __shfl_sync(FULL, at, a), qs = u * p.unit + a;
        int end = __shfl_sync(FULL, qe, a), last = first;
        if (end >= 0) {                                         // not a slice: join what follows in the row
            while (left) {
                const int b = __ffs(left) - 1;
                const int next = __shfl_sync(FULL, at, b), more = __shfl_sync(FULL, qe, b);
                if (((next ^ first) >> 10) != 0 || next - first >= run || more - qs > RUN_QUERIES || more < 0) break;
                end = more; last = next;
                left &= left - 1u;
            }
        }
        const int cell[3] = {first & 1023, (first >> 10) & 1023, first >> 20};
        work(cell, last - first + 1, qs, end & 0x7fffffff);
        __syncwarp();
    }
}

// Slices of four to QSLICE queries, so that there are about `warps` of them before a slice grows; a cell is cut when that
// gives at least two.
static inline void cut_cells(RadiusParams& p, long long warps) {
    const long long want = (p.n / warps + 3) / 4 * 4;
    p.slice = (int)(want < 4 ? 4 : want < QSLICE ? want : QSLICE);
    p.dense = p.slice + p.slice / 2;
}

static inline unsigned unit_count(const RadiusParams& p) { return (unsigned)(((long long)p.n + p.unit - 1) / p.unit); }
// CTAs with one warp per unit
static inline unsigned unit_blocks(const RadiusParams& p) { return (unit_count(p) + TRAV_WARPS - 1) / TRAV_WARPS; }

static __device__ __forceinline__ float fast_exp2(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

static __device__ __forceinline__ float fast_rcp(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// minimum / maximum over the warp in one instruction (sm_100a has the fp32 form), the result in every lane
static __device__ __forceinline__ float warp_min(float v) {
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
static __device__ __forceinline__ float warp_max(float v) {
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Minimum-image displacement of two coordinates of a periodic dimension that is not split into enough
// cells for a frame shift: the subtraction that can lose bits (x near 0 against x near len) is replaced
// by an exact shift of the coordinate next to the upper face.
static __device__ __forceinline__ float mi_delta(float a, float b, float len, float half) {
    float t = a - b;
    if (t > half) t = (a - len) - b;
    else if (t < -half) t = a - (b - len);
    return t;
}

// exact predicate for the pair of original point ids (a, b)
static __device__ __noinline__ bool exact_pair(const RadiusParams& p, int a, int b) {
    const float4 pa = make_float4(p.pos[3 * (size_t)a], p.pos[3 * (size_t)a + 1], p.pos[3 * (size_t)a + 2], 0.f);
    const float4 pb = make_float4(p.pos[3 * (size_t)b], p.pos[3 * (size_t)b + 1], p.pos[3 * (size_t)b + 2], 0.f);
    return exact_within(p, pa, pb);
}

}  // namespace tiga
