// A warp's group of queries against the candidates of its stencil, tested on the tensor cores.
//
// A group is up to GROUP = 16 points that follow each other in cell order within one row of cells, whatever the cells hold:
// 15 to 16 queries a group at every density, where cells taken one at a time (7.6 or 12.6 points) leave a quarter to a half of
// the lanes without a query and stage 340 candidates for 12.6 queries instead of 470 for 16.
//
// The whole stencil is staged, one float4 per candidate as it lies in memory (coordinates, point id).  With q and c relative to
// the middle of the group's cells
//     |q - c|^2 - T = (|q|^2 - T) + (-2 q, 0, 1, 1, 1, 0) . (c, -, c^2, -),
// so one mma of 16 queries by 8 candidates with K = 8 forms 128 tests, whose signs are the answer: 40 instructions per
// 512 tests against 96 with packed fp32 instructions (and the tests are cheap enough not to sort out the candidates that are far
// from all queries, which cost more).  The operands have TF32 precision, so this is a filter: T lies above the squared cutoff by
// the bound of the product's error, 2^-8 |q| (|q| + r) with |q| up to half the length of the group: 2 % more pairs pass than are
// neighbours at 8 points per cell, 7 % at 3, a third at one, where 16 points span 14 cells.  Every pair that passes is decided in fp32
// from the coordinates and, near the cutoff, in fp64.  (mma.sync and not tcgen05: a warp's 16 x 8 results are looked at by the lanes
// that hold them, one instruction later; a tcgen05 tile has 64 rows or more and its results go through tensor memory.)
//
// The accepted slots are gathered into one list per query, so that the lanes share every query's neighbours evenly.
#pragma once
#include "radius_test.cuh"

namespace tiga {

constexpr int GROUP_PLACES = 148 * 20;     // warps of groups that run at once, about
constexpr int GROUP = 16;                  // queries of a group: rows of the mma
constexpr float FILTER_PRODUCT = 3.95e-3f; // margin of the test (Group): of the products, in |q| |c|;
constexpr float FILTER_REACH = 1.001f;     // |c| of a neighbour exceeds |q| by this many cutoffs at most;
constexpr float FILTER_SUMS = 4e-6f;       // of the sums, in |c|^2

// A unit of a large sparse input with a point in a cell of more than this many is done as slices of cells: the input is clustered there, and what the
// slices sort out beforehand is worth more than cheap tests (us, cells / groups / either by unit above 20; 200 k clustered points, one point per
// cell on average, F = 1 1131 / 1265 / 1003, F = 4 1298 / 1580 / 1191, Lennard-Jones 1255 / 1353 / 1076).  Above 20 / 40 points (200 k): clustered,
// two per cell on average, F = 4 2377 / 2464; a slab of 20 points a cell 266 / 234 (cells 209).  The look costs uniform points 0 to 2 % (1 M, 4
// neighbours, F = 1 222 / 226).
constexpr int FULL_CELL = 40;
// Unit u: points [u unit, (u + 1) unit) in cell order, a lane each.
struct GroupUnit {
    int begin, at;                         // first point; cell of the lane's point, ten bits per coordinate
    bool valid;
    __device__ __forceinline__ GroupUnit(const RadiusParams& p, const int u, const int unit) : begin(u * unit), at(0) {
        const int lane = threadIdx.x & 31, i = begin + lane;
        valid = lane < unit && (unsigned)i < (unsigned)p.n;
        if (valid) {
            const float4 v = p.spos[i];
            at = cell_coordinate(p, v.x, 0) | cell_coordinate(p, v.y, 1) << 10 | cell_coordinate(p, v.z, 2) << 20;
        }
    }
    // whether a point lies in a cell of more than FULL_CELL points
    __device__ __forceinline__ bool full(const RadiusParams& p) const {
        int count = 0;
        if (valid) {
            const int* start = p.cell_start + ((at >> 20) * p.nc[1] + ((at >> 10) & 1023)) * p.nc[0] + (at & 1023);
            count = start[1] - start[0];
        }
        return __any_sync(0xffffffffu, count > FULL_CELL);
    }
    // The points, cut into groups where the row of cells changes, at GROUP queries and at p.group_run cells.
    // work(first cell, cells, first query, queries) returns whether to go on
    template <typename Work>
    __device__ __forceinline__ void walk(const RadiusParams& p, Work work) const {
        constexpr unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        unsigned left = __ballot_sync(FULL, valid);
        while (left) {
            const int a = __ffs(left) - 1;
            const int first = __shfl_sync(FULL, at, a);
            const unsigned in = __ballot_sync(FULL, (left >> lane) & 1u && ((at ^ first) >> 10) == 0 && at - first < p.group_run && lane - a < GROUP);
            const int last = __shfl_sync(FULL, at, 31 - __clz(in));
            left &= ~in;
            const int cell[3] = {first & 1023, (first >> 10) & 1023, first >> 20};
            if (!work(cell, last - first + 1, begin + a, __popc(in))) return;
            __syncwarp();
        }
    }
};

// Points per warp.
static inline int group_unit(const long long n) {
    const long long places = GROUP_PLACES;
    return n >= 3 * 32 * places ? 32 : n >= 8 * places ? 16 : n >= 4 * places ? 8 : 4;
}

// The groups fill their stage up with the far slot: it has to lie outside the box and beyond every cutoff.  (At the small end nothing is lost:
// squares are cut downwards, which lets more pairs through, and the tensor cores keep products below the normal numbers.)
static inline bool group_lengths(const RadiusParams& p) {
    return fmaxf(fmaxf(p.len[0], p.len[1]), p.len[2]) < 0.25f * FAR_AWAY && p.r < FAR_AWAY;
}

// Few points per cell: the stencil of 16 queries has fewer than 256 candidates, and a smaller stage lets more warps share an SM.
static inline bool group_sparse(const RadiusParams& p) { return (long long)p.n < 3LL * p.ncells; }

// Shared memory of a warp: the stage and the lists of accepted slots (times 16: byte offsets into the stage), one after the other; a list
// is filled up to whole steps of its query's lanes with the far slot.  CAP: slots of the stage; LIST: entries of all lists.
template <int CAP, int LIST> struct GroupStage {
    // bits of a mask word (eight candidates each) taken together when the accepted slots exceed the lists
    static constexpr int WINDOW = LIST >= GROUP * (8 * 8 + 3) ? 8 : 4;
    static_assert(LIST % 8 == 0 && LIST >= GROUP * (8 * WINDOW + 3), "a window accepted by all queries fits, filled up");
    static_assert(CAP % 32 == 0 && CAP <= 512, "whole steps; two mask words for either column of a lane");
    static constexpr int WORDS = (CAP + 255) / 256;            // mask words per query and column
    static constexpr int CAPACITY = CAP, ENTRIES = LIST;
    static constexpr int FAR = CAP;                            // slot behind the stage, far from everything
    static constexpr int SLOTS = CAP + 4;
    static constexpr int STAGE_BYTES = SLOTS * 16, LIST_BYTES = LIST * 2;
    static constexpr int BYTES = STAGE_BYTES + LIST_BYTES + 16;
    static_assert(BYTES % 16 == 0, "several warps' stages follow each other");
    float4* c;
    unsigned short* list;
    unsigned arrived;                                          // shared address of the mbarrier that counts the staged bytes
    unsigned phase;
    __device__ __forceinline__ explicit GroupStage(unsigned char* base)
        : c(reinterpret_cast<float4*>(base)), list(reinterpret_cast<unsigned short*>(base + STAGE_BYTES)),
          arrived((unsigned)__cvta_generic_to_shared(base + STAGE_BYTES + LIST_BYTES)), phase(0u) {
        if ((threadIdx.x & 31) == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(arrived) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            c[FAR] = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, __int_as_float(-1));
        }
        __syncwarp();
    }
    // whether all bytes of the phase have arrived, the same for all lanes; false if they have not after `tries` looks of up to a
    // microsecond each.  The phase is over only when every lane has seen it: another wait after a failed one waits for the same bytes
    __device__ __forceinline__ bool wait(const int tries) {
        unsigned done = 0u;
        for (int k = 0; k < tries && !done; ++k)
            asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(done) : "r"(arrived), "r"(phase), "r"(1000u) : "memory");
        if (__any_sync(0xffffffffu, !done)) return false;
        phase ^= 1u;
        return true;
    }
};

// d = a b + c, one warp: a 16 x 8 (lane 4 g + t holds rows g and g + 8 of column t, then of column t + 4), b 8 x 8 (column g of rows t
// and t + 4), c and d 16 x 8 (columns 2 t and 2 t + 1 of row g, then of row g + 8)
static __device__ __forceinline__ void mma_16x8x8(float (&d)[4], const unsigned (&a)[4], const unsigned b0, const unsigned b1, const float c0, const float c1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %11, %11};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
}
// Accepted candidates of the lane's two queries, rows g (a) and g + 8 (b) of the group: bit k from the top of word WORDS h + w is slot
// 256 w + 8 k + 2 t + h.
template <int WORDS> struct GroupMask {
    unsigned a[2 * WORDS], b[2 * WORDS];
};

// The stencil by lane: cs is the source of the lane's first position.
struct GroupStencil {
    int begin, len, total, cs;
    __device__ __forceinline__ GroupStencil(const RadiusParams& p, const int (&c)[3], const int run) { cs = stencil_range(p, c, run, false, begin, len, total); }
};

// The group: frame, stencil, the lane's operands of the test.
template <typename Stage>
struct Group {
    const RadiusParams& p;
    Stage& st;
    const int qs, nq;
    const RunFrame frame;
    const GroupStencil sten;
    float4 origin;
    float ot;                              // the lane's component of the origin
    unsigned mask;                         // TF32 bits of the lane's component, nothing of the fourth
    unsigned a[4];
    float c0, c1;
    int lsh;                               // lanes per query: 2^lsh

    __device__ __forceinline__ Group(const RadiusParams& p_, Stage& st_, const int (&cell)[3], const int run, const int qs_, const int nq_)
        : p(p_), st(st_), qs(qs_), nq(nq_), frame(p_, cell, run), sten(p_, cell, run) {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        lsh = nq <= 4 ? 3 : nq <= 8 ? 2 : 1;
        // origin: the middle of the group's cells, not a point (one coordinate that is not finite would take the others' tests with it)
        origin = make_float4((cell[0] + 0.5f * run) * p.hcell[0], (cell[1] + 0.5f) * p.hcell[1], (cell[2] + 0.5f) * p.hcell[2], 0.f);
        frame.shift(p, origin);
        const float4 qa = query(g < nq ? g : 0), qb = query(g + 8 < nq ? g + 8 : 0);
        const float na = norm(qa), nb = norm(qb);
        ot = t == 0 ? origin.x : t == 1 ? origin.y : origin.z;
        mask = t == 3 ? 0u : 0xffffe000u;
        const float va = t == 0 ? qa.x : t == 1 ? qa.y : qa.z, vb = t == 0 ? qb.x : t == 1 ? qb.y : qb.z;
        a[0] = __float_as_uint(-2.f * (va - ot)) & mask;
        a[1] = __float_as_uint(-2.f * (vb - ot)) & mask;
        a[2] = a[3] = t == 3 ? 0u : __float_as_uint(1.f);
        // |q . c - (q . c of the operands)| <= |q| |c| (2^-10 + 2^-10 + 2^-20), |c| <= |q| + r for a neighbour; the squares are rounded
        // down; the rounding of the fp32 sums stays below 2^-18 of their largest term
        const float far = sqrtf(warp_max(fmaxf(na, nb))), reach = far + FILTER_REACH * p.r;
        const float thr = p.r2_hi + FILTER_PRODUCT * far * reach + FILTER_SUMS * reach * reach;
        c0 = g < nq ? na - thr : INFINITY;
        c1 = g + 8 < nq ? nb - thr : INFINITY;
    }
    // query k in the frame, .w = point id
    __device__ __forceinline__ float4 query(const int k) const {
        float4 v = p.spos[qs + k];
        frame.shift(p, v);
        return v;
    }
    __device__ __forceinline__ float norm(const float4& v) const {
        const float x = v.x - origin.x, y = v.y - origin.y, z = v.z - origin.z;
        return fmaf(z, z, fmaf(y, y, x * x));
    }

    // Stages positions [k0, k0 + CAPACITY) of the flattened stencil, the last step of 32 filled up with far candidates; returns the slots
    // staged, or 0 when the copies did not arrive.  Every range of the stencil is one bulk copy, issued by the lane that holds it (a lane
    // per candidate, its range looked up: 526 instead of 90 instructions per group).
    __device__ __forceinline__ int stage(const int k0) {
        const int lane = threadIdx.x & 31;
        const int n = sten.total - k0 < Stage::CAPACITY ? sten.total - k0 : Stage::CAPACITY;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // what was read and written here before
        __syncwarp();
        const int from = sten.begin > k0 ? sten.begin : k0, end = sten.begin + sten.len < k0 + n ? sten.begin + sten.len : k0 + n;
        const int src = sten.cs + from - sten.begin;
        const bool whole = checked_range(src, end - from, p.n, CHECK_SLOT);
        int copied = n;
#ifdef TIGA_CHECKED
        if (!whole) for (int k = 0; k < end - from; ++k) st.c[from - k0 + k] = p.spos[checked(src + k, p.n, CHECK_SLOT)];
        copied -= __reduce_add_sync(0xffffffffu, whole ? 0 : end - from);
#endif
        if (lane == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(st.arrived), "r"(16 * copied) : "memory");
        if (from < end && whole) {
            asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                         ::"r"((unsigned)__cvta_generic_to_shared(st.c + (from - k0))), "l"(p.spos + src), "r"(16 * (end - from)), "r"(st.arrived) : "memory");
        }
        const int ns = (n + 31) & ~31;
        if (n + lane < ns) st.c[n + lane] = make_float4(FAR_AWAY, FAR_AWAY, FAR_AWAY, __int_as_float(-1));
        if (!st.wait(copy_tries(p))) return 0;
        __syncwarp();
        if (frame.face) {                                      // warp uniform
            for (int k = lane; k < n; k += 32) frame.shift(p, st.c[k]);
            __syncwarp();
        }
        return ns;
    }

    // tests all queries against the ns staged candidates from stencil position k0
    __device__ __forceinline__ void test(const int ns, const int k0, GroupMask<Stage::WORDS>& m) const {
        const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
        const float* s = reinterpret_cast<const float*>(st.c) + lane;      // component t of slot g
#pragma unroll
        for (int w = 0; w < Stage::WORDS; ++w) {
            const int eights = ns - 256 * w >= 256 ? 32 : ns > 256 * w ? (ns - 256 * w) >> 3 : 0;      // multiple of four
            unsigned m0 = 0u, m1 = 0u, m2 = 0u, m3 = 0u;
            for (int k = 0; k < eights; k += 4) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float d[4];
                    const float v = s[32 * j] - ot;
                    mma_16x8x8(d, a, __float_as_uint(v) & mask, __float_as_uint(v * v) & mask, c0, c1);
                    m0 = __funnelshift_l(__float_as_uint(d[0]), m0, 1);
                    m1 = __funnelshift_l(__float_as_uint(d[1]), m1, 1);
                    m2 = __funnelshift_l(__float_as_uint(d[2]), m2, 1);
                    m3 = __funnelshift_l(__float_as_uint(d[3]), m3, 1);
                }
                s += 128;
            }
            const int up = 32 - eights;                        // 32: the words are zero
            m.a[w] = m0 << (up & 31); m.a[Stage::WORDS + w] = m1 << (up & 31);
            m.b[w] = m2 << (up & 31); m.b[Stage::WORDS + w] = m3 << (up & 31);
        }
        // the queries themselves: position qs + row of the range that holds the group's cells (lane 4)
        const int self = qs + __shfl_sync(0xffffffffu, sten.begin - sten.cs, 4) - k0;
        drop(m.a, self + g, t);
        drop(m.b, self + g + 8, t);
    }
    // takes arrival k out
    static __device__ __forceinline__ void drop(unsigned (&m)[2 * Stage::WORDS], const int at, const int t) {
        if (at < 0 || at >= Stage::CAPACITY || ((at >> 1) & 3) != t) return;
        const unsigned bit = 0x80000000u >> ((at >> 3) & 31);
        const int word = (at >> 8) + (at & 1) * Stage::WORDS;
#pragma unroll
        for (int k = 0; k < 2 * Stage::WORDS; ++k) if (k == word) m[k] &= ~bit;
    }

    // Writes the slots of the set bits of two words, base + 128 k (bytes) for bit k from the top, to the shared addresses la and lb.
    static __device__ __forceinline__ void put_slots(unsigned ma, unsigned mb, const int base, unsigned& la, unsigned& lb) {
        while (ma | mb) {
            asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 k, j, s;\n\t"
                         "setp.ne.u32 p, %0, 0;\n\tsetp.ne.u32 q, %1, 0;\n\t"
                         "clz.b32 k, %0;\n\tclz.b32 j, %1;\n\t"
                         "shr.u32 s, 0x80000000, k;\n\txor.b32 s, s, -1;\n\tand.b32 %0, %0, s;\n\t"
                         "shr.u32 s, 0x80000000, j;\n\txor.b32 s, s, -1;\n\tand.b32 %1, %1, s;\n\t"
                         "mad.lo.u32 k, k, 128, %4;\n\tmad.lo.u32 j, j, 128, %4;\n\t"
                         "@p st.shared.u16 [%2], k;\n\t@q st.shared.u16 [%3], j;\n\t"
                         "@p add.u32 %2, %2, 2;\n\t@q add.u32 %3, %3, 2;\n\t}"
                         : "+r"(ma), "+r"(mb), "+r"(la), "+r"(lb) : "r"(base) : "memory");
        }
    }

    // Calls consume(first, end) with the list of the lane's query (lane >> lsh), st.list[first, end), in whole steps of two entries per
    // lane; several times, with between() after all but the last, when the accepted slots do not fit.
    template <typename Consume, typename Between>
    __device__ __forceinline__ void lists(const int ns, const GroupMask<Stage::WORDS>& m, Consume consume, Between between) const {
        constexpr unsigned FULL = 0xffffffffu;
        constexpr int WORDS = Stage::WORDS, NW = 2 * WORDS, WINDOW = Stage::WINDOW;
        const int lane = threadIdx.x & 31, t = lane & 3;
        const int up = (2 << lsh) - 1;                         // lists are whole multiples of this plus one
        const int q = lane >> lsh, from = (q & 7) * 4;
        const unsigned list0 = (unsigned)__cvta_generic_to_shared(st.list);
        bool whole = true;
        for (int win = 0;;) {
            unsigned a[NW], b[NW];
#pragma unroll
            for (int k = 0; k < NW; ++k) {
                const unsigned take = whole ? FULL : win / (32 / WINDOW) == k % WORDS ? ~(~0u >> WINDOW) >> win % (32 / WINDOW) * WINDOW : 0u;
                a[k] = m.a[k] & take; b[k] = m.b[k] & take;
            }
            int na = 0, nb = 0;
#pragma unroll
            for (int k = 0; k < NW; ++k) { na += __popc(a[k]); nb += __popc(b[k]); }
            const int own = na | nb << 16;                     // both counts in one word: all lists together hold at most 16 (CAP + 16) < 2^16
            // The lane's place among the four of its row.  Row g's list begins with lane g mod 4: at any moment neighbouring queries read
            // slots of different lanes, which lie in different banks.
            int ex = 0, all = own;
#pragma unroll
            for (int o = 1; o < 4; ++o) {
                const int other = __shfl_sync(FULL, own, (lane & ~3) | ((t - o) & 3));
                if (((t - (lane >> 2)) & 3) >= o) ex += other;
                all += other;
            }
            const int filled = (all + (up | up << 16)) & ~(up | up << 16);
            int start = filled;                                // inclusive over the rows
#pragma unroll
            for (int o = 4; o < 32; o <<= 1) {
                const int other = __shfl_up_sync(FULL, start, o);
                if (lane >= o) start += other;
            }
            const int sum = __shfl_sync(FULL, start, 31);
            start -= filled;
            start += (sum & 0xffff) << 16;                     // rows 8 to 15 follow rows 0 to 7
            if (whole && (sum & 0xffff) + (sum >> 16) > Stage::ENTRIES) { whole = false; continue; }
            unsigned short* fa = st.list + (start & 0xffff);
            unsigned short* fb = st.list + (start >> 16);
            for (int k = (all & 0xffff) + t; k < (filled & 0xffff); k += 4) fa[k] = (unsigned short)(16 * Stage::FAR);
            for (int k = (all >> 16) + t; k < (filled >> 16); k += 4) fb[k] = (unsigned short)(16 * Stage::FAR);
            unsigned la = list0 + 2 * ((start + ex) & 0xffff), lb = list0 + 2 * ((start + ex) >> 16);
#pragma unroll
            for (int k = 0; k < NW; ++k) put_slots(a[k], b[k], 16 * (2 * t + 256 * (k % WORDS) + k / WORDS), la, lb);
            __syncwarp();
            const int s0 = __shfl_sync(FULL, start, from), f0 = __shfl_sync(FULL, filled, from);
            const int first = q < 8 ? s0 & 0xffff : s0 >> 16;
            consume(first, q < nq ? first + (q < 8 ? f0 & 0xffff : f0 >> 16) : first);
            __syncwarp();
            if (whole || 8 * WINDOW * ++win >= ns) break;
            between();
        }
    }
};

// Copies that did not arrive in time: points [from, end) in cell order, which the warp leaves undone, get sums that are not a number and counts
// of -1.  (Never seen; a caller who looks at the results cannot take them for sums.)
static __device__ __noinline__ void give_up(const RadiusParams& p, const int sums, const int from, const int end) {
    for (int i = from + (int)(threadIdx.x & 31); i < end; i += 32) {
        const int id = checked(__float_as_int(p.spos[i].w), p.n, CHECK_POINT);
        for (int f = 0; f < sums; ++f) p.out[(size_t)id * sums + f] = __int_as_float(0x7fffffff);
        if (p.count) p.count[id] = -1;
    }
}

}  // namespace tiga
