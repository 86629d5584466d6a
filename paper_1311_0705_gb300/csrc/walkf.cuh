// The walk of walk.cuh on grids whose bounds are all single-precision
// numbers (LeafRecF): the same cells, times, lengths and sums bit for bit,
// with most decisions of a crossing made in single precision and every load of
// a warp in flight at once.
//
// GB300 issues one FP64 warp instruction per 19 cycles and SM, and the walk
// of walk.cuh spends ten of them per crossing: six on the three wall times,
// two on the exit point, one on the length, one on the sum.  Only the time
// of the wall that is crossed, the length and the sum are results (four); the
// others only serve comparisons, which here are made on single-precision
// values with rigorous error bounds:
//
//   u = 2^-24; o, k the ray's origin and direction, i = 1/k per axis; o32 = o
//   (1 + u), i32 = i (1 + u), k32 = k (1 + 2.1u); w a wall, exact.
//   t32 = (w - o32) i32 differs from the contract's wall time t by at most
//   3.1 u |t32| + 1.1 u |o| |i32|, so t lies between
//     tl = t32 (1 - 5u) - E and tu = t32 (1 + 6u) + E,  E = 1.25 u |o32| |i32|.
//   Exit wall: with m the smallest tu, the axis of the contract's smallest
//   time is certain when exactly one axis has tl <= m.  (A wall time that
//   comes out slightly negative has |t32| <= E, which the slack in E covers.)
//   The exit time is that axis's t unless the walk is already past it
//   (contract: exit times never fall below the current time); m no smaller
//   than the upper bound of the current time makes sure that this moves
//   it by no more than the bounds' width.
//   Exit point: p32 = o32 + k32 tm, tm the middle of [tl, m]; it differs from
//   the contract's point (rounded, and clamped to the leaf) by at most
//     eps = 4.5 u (max |o| + max |domain|) + max |k| (m - tl) / 2,
//   since |k t| <= |o| + |domain| on a path inside the domain and the clamp
//   moves the point by no more than the 2^-48 or so by which double
//   rounding can place it outside the leaf it leaves.  A neighbor whose
//   bounds p32 clears by more than eps on both axes holds the point.
//
// Whatever these bounds leave open (a few crossings in a thousand) is
// decided by the contract's own FP64 arithmetic, as are all crossings of rays
// whose direction components leave [2^-30, 2^30] or whose origin is far out
// or, next to a wall at zero, has a component below 2^-60 (o32 = o (1 + u)
// and a normal E would not hold down to the smallest numbers; a component
// that is zero is exact) (SG_EXACT): E and eps are infinite there and every
// comparison fails.  A NaN
// fails every comparison too.  An axis with a zero direction gets i32 = 2^100
// and E = 2^100 (bound of the position error): its wall counts as out of
// reach unless the ray runs within that bound of it.
//
// Against walls that are single-precision numbers a double p compares as its
// directed image does: f = the largest float <= p, the next one down when p is a
// float and the point belongs to the lower side of a wall it lies on.  Then p
// is on the upper side of wall w exactly when f >= w, and in a leaf when lo
// <= f < hi, ties included (dir_float).
//
// The next leaf comes from the record's wall slot: the neighbor itself when one
// leaf covers the face; where two or four equal leaves with ids in arithmetic
// progression do (siblings, which the builders number consecutively), the first of
// them and the steps between them, the exit point picking the one; otherwise the
// face's rope node, below which the point is located.  On the disk octree (3.35e6
// leaves) 99.1 % of crossings need nothing but that slot; the list search of
// walk.cuh tested 1.105 records per crossing there.
//
// Latency: a lane that must wait for memory only changes its state (start
// record, leaf record or tree node under way) and issues its load; its warp goes on
// to the other lanes, and one wait per round serves all of them.  Lanes wait until
// kRefill of a warp are idle and are refilled together from queue items taken 32
// at a time.
//
// Measured, 1e6 rays on the disk octree, FP64 optical depth: walk 969 us with walk.cuh, 527 us here; calls 1248 -> 697 us, and
// 18.6 -> 11.4 ms for 1e7 rays through the torus (FP32K).  The records and decisions alone, inside the loop of walk.cuh, gained
// nothing (960 us): every round of a warp waited there for its lanes' chains of dependent refill loads (queue atomic,
// order, start record, first leaf) and list searches, which the lane states put under way together.  The four FP64
// operations per crossing bound the walk at 235 us; what it lives on is instructions, so they are few: the steps to equal
// neighbors in the spare bits of the wall slot, one comparison of the high words for "later than now, before the end" (the rest in
// the branch not taken), the two parts of eps in shared memory, and no register spills in the optical-depth walk (20 bytes
// of them cost it 12 %).
#pragma once

#include "walk.cuh"

namespace hg {

constexpr uint32_t SG_EXACT = 1u << 16;  // (RayStartF.sg) the ray's crossings are decided in FP64 throughout

// Double equal to a single-precision wall (0 or a normal number).
__device__ __forceinline__ double widen(float w) {
    const int b = __float_as_int(w);
    const int hi = ((b >> 3) & (int)0x8fffffff) + 0x38000000;
    return (b << 1) == 0 ? 0.0 : __hiloint2double(hi, b << 29);
}
// A non-negative double's single-precision lower bound, less than 2^-23 below (zero below 2^-126).
__device__ __forceinline__ float floor_float(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    if (hi < 0x38100000u) return 0.0f;
    return hi < 0x47f00000u ? __uint_as_float(__funnelshift_l(lo, hi - 0x38000000u, 3)) : CUDART_INF_F;
}
// Directed image of a point coordinate: compares with single-precision walls as p does (f >= w: upper side);
// down: a point on a wall belongs to its lower side.
__device__ __forceinline__ float dir_float(double p, bool down) {
    const uint32_t hi = (uint32_t)__double2hiint(p), lo = (uint32_t)__double2loint(p);
    const uint32_t mag = hi & 0x7fffffffu, neg = hi >> 31;
    if (mag < 0x38100000u) {  // between the walls next to zero, or zero
        const bool zero = (mag | lo) == 0u;
        return (zero ? down : neg != 0u) ? -CUDART_MIN_DENORM_F : 0.0f;
    }
    uint32_t f = __funnelshift_l(lo, mag - 0x38000000u, 3);
    const bool inexact = (lo & 0x1fffffffu) != 0u;
    if (neg)
        f += (inexact || down) ? 1u : 0u;
    else
        f -= (!inexact && down) ? 1u : 0u;
    return __uint_as_float((neg << 31) | f);
}

// Does a point on axis a with direction signs sg belong to the lower side of a wall it lies on?  (With a
// zero direction only on the domain's upper face, which is closed.)
__device__ __forceinline__ bool lower_side(const DevGrid &G, uint32_t sg, int a, double p) {
    return dneg(sg, a) || (!dpos(sg, a) && okey(p) == G.khi[a]);
}

// Top-down descent on directed images (descend, walk.cuh).  The first n_smem nodes come from shared memory.
// KIND: HG_OCTREE, HG_KDTREE, or 2 = read from G.kind.
template <int KIND>
__device__ __forceinline__ int32_t descend_f(const DevGrid &G, const unsigned char *snodes, int n_smem, float p0,
                                             float p1, float p2) {
    const bool kd = (KIND == 2) ? (G.kind == HG_KDTREE) : (KIND == HG_KDTREE);
    int32_t nd = 0;
    for (int it = 0; it <= G.max_depth; it++) {
        if (kd) {
            const uint2 v = nd < n_smem ? reinterpret_cast<const uint2 *>(snodes)[nd]
                                        : __ldg(reinterpret_cast<const uint2 *>(G.nodes) + nd);
            const int ax = (int)(v.y & 3u);
            if (ax == 3) return (int32_t)(v.y >> 2);
            nd = (int32_t)(v.y >> 2) + (sel3(ax, p0, p1, p2) >= __uint_as_float(v.x) ? 1 : 0);
        } else {
            const float4 v = nd < n_smem ? reinterpret_cast<const float4 *>(snodes)[nd]
                                         : __ldg(reinterpret_cast<const float4 *>(G.nodes) + nd);
            const int32_t link = __float_as_int(v.w);
            if (link < 0) return -1 - link;
            nd = link + (p0 >= v.x ? 1 : 0) + (p1 >= v.y ? 2 : 0) + (p2 >= v.z ? 4 : 0);
        }
    }
    return -1;
}

// Start state of a ray (RayStart for these grids) or of a path segment (records n + s), two 32-byte sectors.
struct alignas(32) RayStartF {
    double ik[3];       // 1/d per axis (0 where d_a == 0)
    long long ktstart;  // key of the entry time
    double o[3];        // origin (a signed zero as +0)
    int32_t cur;        // first leaf, or -1 when the ray does not walk
    uint32_t sg;        // direction sign bits | SG_SKIP_FIRST | SG_SPLIT | status bits << 8 | SG_EXACT
};
static_assert(sizeof(RayStartF) == 64, "the walks read start records like leaf records");

// Start record of a ray set up as R (R.work and R.t1 are kept apart).
__device__ __forceinline__ RayStartF start_f(const RayStart &R, const double *__restrict__ o,
                                             const double *__restrict__ d, int64_t r) {
    RayStartF S;
    S.ik[0] = R.ik0;
    S.ik[1] = R.ik1;
    S.ik[2] = R.ik2;
    S.ktstart = R.ktstart;
    S.cur = R.cur;
    bool exact = false;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const double x = o[3 * r + a], k = d[3 * r + a];
        S.o[a] = dzero(x) ? 0.0 : x;
        // zero, or of magnitude [2^-60, 2^20) (origin), [2^-30, 2^30) (direction), on the exponents
        const uint32_t mx = ((uint32_t)__double2hiint(x) & 0x7fffffffu) - 0x3c300000u;
        const uint32_t mk = ((uint32_t)__double2hiint(k) & 0x7fffffffu) - 0x3e100000u;
        exact = exact || !(dzero(x) || mx < 0x05000000u) || !(dzero(k) || mk < 0x03c00000u);
    }
    S.sg = R.sg | (exact ? SG_EXACT : 0u);
    return S;
}

// Location of a point given by its keys (ray_setup).
template <int KIND>
__device__ __forceinline__ int32_t locate_key_f(const DevGrid &G, const unsigned char *snodes, int n_smem,
                                                long long p0, long long p1, long long p2, uint32_t sg) {
    const double q0 = kdouble(p0), q1 = kdouble(p1), q2 = kdouble(p2);
    return descend_f<KIND>(G, snodes, n_smem, dir_float(q0, lower_side(G, sg, 0, q0)),
                           dir_float(q1, lower_side(G, sg, 1, q1)), dir_float(q2, lower_side(G, sg, 2, q2)));
}

// A leaf record, start record or tree node on its way or arrived: 64 bytes in registers.
struct RawRec {
    uint32_t v[16];
    __device__ __forceinline__ void load(const void *p) {
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                     : "l"(p));
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                       "=r"(v[15])
                     : "l"(static_cast<const char *>(p) + 32));
    }
    __device__ __forceinline__ void load_node(const DevGrid &G, int32_t nd) {
        if (G.kind == HG_KDTREE)
            asm volatile("ld.global.nc.v2.b32 {%0, %1}, [%2];"
                         : "=r"(v[0]), "=r"(v[1])
                         : "l"(static_cast<const KdNodeF *>(G.nodes) + nd));
        else
            asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                         : "l"(static_cast<const OctNodeF *>(G.nodes) + nd));
    }
    __device__ __forceinline__ double d(int j) const { return __hiloint2double((int)v[j + 1], (int)v[j]); }
    // leaf records
    __device__ __forceinline__ float lo(int a) const { return __uint_as_float(v[a]); }
    __device__ __forceinline__ float hi(int a) const { return __uint_as_float(v[3 + a]); }
    __device__ __forceinline__ double rho() const { return d(6); }
    __device__ __forceinline__ int32_t first(int w) const { return (int32_t)v[8 + w]; }
    __device__ __forceinline__ float rho32() const { return __uint_as_float(v[14]); }
};

// Per-ray walking state.  Shared memory holds, per thread, {o32, i32, E, k32} of each axis and the origin
// and 1/d in FP64, and the two parts of eps (104 bytes; slots strided by the block so that a warp's accesses
// fall on consecutive words): with them in registers four 256-thread blocks would not fit on an SM.
constexpr int kGeoBytesF = 104;
struct RayStateF {
    float4 *a;  // this thread's first axis slot
    double *g;  // its first FP64 slot
    float2 *e;  // {slope, constant} of eps in the width of the exit time's bounds
    int gs;     // slot stride
    long long ktcur;   // key of the current time
    long long klim;    // smaller of the keys of the path's end and of the time a path segment stops after;
                       // -1 while the segment's first leaf, which the segment before records, is walked
    float tp;          // upper bound of the current time
    uint32_t sg;
    int32_t cur, steps;  // current leaf; steps left
    __device__ __forceinline__ void bind(unsigned char *geo) {
        gs = (int)blockDim.x;
        a = reinterpret_cast<float4 *>(geo) + threadIdx.x;
        g = reinterpret_cast<double *>(geo + (size_t)gs * 3 * sizeof(float4)) + threadIdx.x;
        e = reinterpret_cast<float2 *>(geo + (size_t)gs * (3 * sizeof(float4) + 6 * sizeof(double))) + threadIdx.x;
    }
    __device__ __forceinline__ double o(int x) const { return g[x * gs]; }
    __device__ __forceinline__ double ik(int x) const { return g[(3 + x) * gs]; }
};

// Geometry of a ray from its start record (SG_EXACT rays: E and base infinite, the rest of no account).
__device__ __forceinline__ void start_geometry(const RawRec &V, float fdom, RayStateF &S) {
    const bool exact = (V.v[15] & SG_EXACT) != 0;
    float o32[3], scale = 0.0f, kmax = 0.0f;
#pragma unroll
    for (int x = 0; x < 3; x++) {
        o32[x] = near_float(V.d(8 + 2 * x));
        scale = fmaxf(scale, fabsf(o32[x]));
    }
    const float base = exact ? CUDART_INF_F : 4.5f * 0x1p-24f * (scale + fdom);
#pragma unroll
    for (int x = 0; x < 3; x++) {
        const double ik = V.d(2 * x);
        float i32 = near_float(ik), k32;
        float e = 1.25f * 0x1p-24f * fabsf(o32[x]) * fabsf(i32);
        asm("rcp.approx.f32 %0, %1;" : "=f"(k32) : "f"(i32));
        k32 = __fmaf_rn(k32, __fmaf_rn(-i32, k32, 1.0f), k32);
        if (i32 == 0.0f) {
            i32 = 0x1p100f;
            k32 = 0.0f;
            e = 0x1p100f * base;
        }
        kmax = fmaxf(kmax, fabsf(k32));
        S.a[x * S.gs] = make_float4(o32[x], i32, exact ? CUDART_INF_F : e, k32);
        S.g[x * S.gs] = V.d(8 + 2 * x);
        S.g[(3 + x) * S.gs] = ik;
    }
    S.e[0] = make_float2(0.501f * kmax, base);
}

// The exit wall by the contract's FP64 arithmetic: smallest time, ties to the lower axis (-1: no wall in finite time).
__device__ __forceinline__ int exit_exact(const RayStateF &S, const RawRec &L, long long *kt_out) {
    const uint32_t sg = S.sg;
    long long kt = KEY_INF;
    int ax = -1;
#pragma unroll
    for (int x = 0; x < 3; x++) {
        if (!(dpos(sg, x) || dneg(sg, x))) continue;
        const long long ct = okey((widen(dneg(sg, x) ? L.lo(x) : L.hi(x)) - S.o(x)) * S.ik(x));
        if (ct < kt) {
            kt = ct;
            ax = x;
        }
    }
    *kt_out = kt;
    return ax;
}

// The exit point and the leaf it is looked for in.
struct CandF {
    int32_t id;     // record (or, while it is located, tree node) to look at
    int32_t ax;     // exit axis; | CAND_EXACT: p1, p2 are directed images, eps infinite
    int32_t left;   // while it is located: nodes left to visit, | CAND_ROOT: from the root
    float wall;     // its coordinate on the exit axis
    float p1, p2;   // on the two other axes (b1 < b2), known to within eps
    float eps;      // minus infinity: the record is known to hold the point
    // A leaf known to hold the point is next.
    __device__ __forceinline__ void enter(int32_t leaf) {
        id = leaf;
        ax = 0;
        p1 = p2 = 0.0f;
        eps = -CUDART_INF_F;
    }
};
constexpr int32_t CAND_EXACT = 4, CAND_ROOT = 1 << 30;

// Directed images of the contract's exit point: o + d t rounded, clamped to the leaf being left.
__device__ __forceinline__ void exit_point_exact(const DevGrid &G, const WalkIO &io, int64_t r, const RayStateF &S,
                                                 CandF &C) {
    const double t = kdouble(S.ktcur);
    const LeafRecF *P = G.recf + S.cur;
#pragma unroll
    for (int j = 0; j < 2; j++) {
        const int b = j == 0 ? (C.ax == 0 ? 1 : 0) : (C.ax == 2 ? 1 : 2);
        double p = __fma_rn(io.d[3 * r + b], t, S.o(b));
        const double lo = widen(__ldg(&P->lo[b])), hi = widen(__ldg(&P->hi[b]));
        if (okey(p) < okey(lo)) p = lo;
        if (okey(p) > okey(hi)) p = hi;
        const float f = dir_float(p, lower_side(G, S.sg, b, p));
        if (j == 0)
            C.p1 = f;
        else
            C.p2 = f;
    }
    C.ax |= CAND_EXACT;
    C.eps = CUDART_INF_F;
}

// One step of the top-down location of the exit point from the node in V: true when C.id is the leaf, false
// when it is the next node.  Where the bounds leave the side open the point is taken exactly and the search
// starts anew at the root.
__device__ __forceinline__ bool locate_step(const DevGrid &G, const WalkIO &io, int64_t r, const RayStateF &S,
                                            const RawRec &V, CandF &C) {
    const int ax = C.ax & 3;
    const float e = (C.ax & CAND_EXACT) ? -1.0f : C.eps;
    // a point on the wall belongs to the side the ray goes to
    const bool neg = dneg(S.sg, ax);
    auto upper = [&](int x, float p, float s) { return x != ax ? p >= s : (neg ? C.wall > s : C.wall >= s); };
    bool open;
    int32_t next;
    if (G.kind == HG_KDTREE) {
        const uint32_t link = V.v[1];
        const int x = (int)(link & 3u);
        next = (int32_t)(link >> 2);
        if (x == 3) {
            C.id = next;
            return true;
        }
        const float s = __uint_as_float(V.v[0]);
        const float p = x == (ax == 0 ? 1 : 0) ? C.p1 : C.p2;
        open = x != ax && !(fabsf(p - s) > e);
        next += upper(x, p, s) ? 1 : 0;
    } else {
        const int32_t link = (int32_t)V.v[3];
        if (link < 0) {
            C.id = -1 - link;
            return true;
        }
        const float s0 = __uint_as_float(V.v[0]), s1 = __uint_as_float(V.v[1]), s2 = __uint_as_float(V.v[2]);
        const float p0 = C.p1, p1 = ax == 0 ? C.p1 : C.p2, p2 = C.p2;
        open = !((ax == 0 || fabsf(p0 - s0) > e) && (ax == 1 || fabsf(p1 - s1) > e) && (ax == 2 || fabsf(p2 - s2) > e));
        next = link + (upper(0, p0, s0) ? 1 : 0) + (upper(1, p1, s1) ? 2 : 0) + (upper(2, p2, s2) ? 4 : 0);
    }
    if (open) {
        exit_point_exact(G, io, r, S, C);
        C.left = (G.max_depth + 2) | CAND_ROOT;  // one more than visits: the caller counts this step
        next = 0;
    }
    C.id = next;
    return false;
}

// What a lane's loads on their way are; DONE: its item has ended (the outputs not yet written), EXIT: the
// queue is empty.
enum { LANE_WALK = 0, LANE_START = 1, LANE_NODE = 2, LANE_DONE = 3, LANE_EXIT = 4 };
// Idle lanes of a warp that are refilled together: a refill is ~100 instructions whatever the number of
// lanes taking part, an idle lane costs its share of a round.  2, 4, 5, 6, 8 lanes: disk octree (1e6 rays) 741, 715, 708, 703,
// 693 us, torus (1e7) 11.57, 11.32, 11.37, 11.47, 11.66 ms per call.
constexpr int kRefill = 5;
struct PoolItem {
    int64_t item;  // queue item: a ray, or n_rays + s for path segment s
    int64_t of;    // the ray it is, or is part of (batches: its grid)
};

// The walking loop (walk_loop, walk.cuh) on single-precision records, of either tree and navigation.
// Src hands a warp up to 32 queue items at a time: int grab(PoolItem *pool, const WalkIO &io), called by all lanes,
// and what an item's walk needs: void item(const PoolItem &, const DevGrid *&, int32_t &max_steps).
// geo: shared memory, kGeoBytesF per thread of the block, 16-byte aligned; pool: 32 items per warp.
template <int MODE, int PREC, class Src>
__device__ __forceinline__ void walk_loop_f(Src &src, const WalkIO &io, unsigned char *geo, PoolItem *pool) {
    constexpr bool SEGS = Src::kSegments;
    using TallyT = Tally<MODE, PREC, SEGS>;
    constexpr bool USE32 = TallyT::TAU && TallyT::TPREC == HG_FP32K;
    const DevGrid *Gp = nullptr;
    const LeafRecF *rec = nullptr;
    RayStateF S;
    S.bind(geo);
    RawRec V;
    CandF C;
    TallyT T(io);
    T.ray = -1;
    int state = LANE_DONE;
    int have = 0, used = 0;  // items in the warp's pool, and of those taken
    bool drained = false;
    pool += (threadIdx.x >> 5) * 32;
    // the grid and its records: launch constants of a single-grid walk, looked up per ray in a batch
    auto grid = [&]() -> const DevGrid & {
        if constexpr (SEGS)
            return *src.G;
        else
            return *Gp;
    };
    auto records = [&]() -> const LeafRecF * {
        if constexpr (SEGS)
            return src.G->recf;
        else
            return rec;
    };
    auto ray_of = [&]() -> int64_t {
        return (SEGS && T.ray >= io.n_rays) ? io.segs[T.ray - io.n_rays].ray : T.ray;
    };
    for (;;) {
        // ---- idle lanes: outputs of the finished items, new items
        const unsigned need = __ballot_sync(0xffffffffu, state == LANE_DONE);
        const unsigned busy = __ballot_sync(0xffffffffu, state < LANE_DONE);
        if ((need | busy) == 0u) break;
        if (__popc(need) >= kRefill || busy == 0u) {
            if (used == have && !drained) {
                __syncwarp();
                have = src.grab(pool, io);
                used = 0;
                drained = have == 0;
                __syncwarp();
            }
            const int rank = __popc(need & ((1u << (threadIdx.x & 31)) - 1u));
            const int left = have - used;
            if (state == LANE_DONE) {
                if (T.ray >= 0) T.finish(io, S.cur, S.ktcur);
                T.ray = -1;
                if (drained) {
                    state = LANE_EXIT;
                } else if (rank < left) {
                    const PoolItem P = pool[used + rank];
                    src.item(P, Gp, S.steps);
                    if (!SEGS) rec = Gp->recf;
                    T.ray = P.item;
                    T.reset();
                    V.load(static_cast<const RayStartF *>(io.starts) + P.item);
                    S.klim = KEY_INF;
                    if (SEGS && P.item >= io.n_rays) S.klim = io.segs[P.item - io.n_rays].ktstop;
                    S.ktcur = KEY_INF;
                    if (io.smax) S.ktcur = __double_as_longlong(__ldg(io.smax + (SEGS ? P.of : P.item)));
                    T.fetch(io, SEGS ? P.of : P.item);
                    state = LANE_START;
                }
            }
            const int taken = __popc(need);
            used += taken < left ? taken : left;
        }
        if (state == LANE_WALK) {
            const DevGrid &G = grid();
            const uint32_t sg = S.sg;
            {
                const bool x0 = (C.ax & 3) == 0, x2 = (C.ax & 3) == 2;
                const float l1 = x0 ? V.lo(1) : V.lo(0), h1 = x0 ? V.hi(1) : V.hi(0);
                const float l2 = x2 ? V.lo(1) : V.lo(2), h2 = x2 ? V.hi(1) : V.hi(2);
                const float q = fminf(fminf(C.p1 - l1, h1 - C.p1), fminf(C.p2 - l2, h2 - C.p2));
                if (!(q > C.eps)) {  // not certainly inside
                    if (!(C.ax & CAND_EXACT)) exit_point_exact(G, io, ray_of(), S, C);
                    if (!(l1 <= C.p1 && C.p1 < h1 && l2 <= C.p2 && C.p2 < h2)) {
                        // an exit point on the domain surface with the direction pointing out ends the path;
                        // else it is on an edge or corner: located from the root
                        const float gl1 = x0 ? G.flo[1] : G.flo[0], gh1 = x0 ? G.fhi[1] : G.fhi[0];
                        const float gl2 = x2 ? G.flo[1] : G.flo[2], gh2 = x2 ? G.fhi[1] : G.fhi[2];
                        if (!(gl1 <= C.p1 && C.p1 < gh1 && gl2 <= C.p2 && C.p2 < gh2)) {
                            state = LANE_DONE;
                        } else {
                            C.left = (G.max_depth + 1) | CAND_ROOT;
                            C.id = 0;
                            V.load_node(G, 0);
                            state = LANE_NODE;
                        }
                        goto next_round;
                    }
                }
            }
            S.cur = C.id;
            // exit wall
            const float4 A0 = S.a[0], A1 = S.a[S.gs], A2 = S.a[2 * S.gs];  // {o32, i32, E, k32}
            const float2 ep = S.e[0];
            const float w0 = dneg(sg, 0) ? V.lo(0) : V.hi(0);
            const float w1 = dneg(sg, 1) ? V.lo(1) : V.hi(1);
            const float w2 = dneg(sg, 2) ? V.lo(2) : V.hi(2);
            const float t0 = (w0 - A0.x) * A0.y, t1 = (w1 - A1.x) * A1.y, t2 = (w2 - A2.x) * A2.y;
            constexpr float cl = 1.0f - 5.0f * 0x1p-24f, cu = 1.0f + 6.0f * 0x1p-24f;
            const float tl0 = __fmaf_rn(t0, cl, -A0.z), tu0 = __fmaf_rn(t0, cu, A0.z);
            const float tl1 = __fmaf_rn(t1, cl, -A1.z), tu1 = __fmaf_rn(t1, cu, A1.z);
            const float tl2 = __fmaf_rn(t2, cl, -A2.z), tu2 = __fmaf_rn(t2, cu, A2.z);
            float m = fminf(fminf(tu0, tu1), tu2);
            float ml = fminf(fminf(tl0, tl1), tl2);
            const bool q0 = !(tl0 > m), q1 = !(tl1 > m), q2 = !(tl2 > m);
            const bool sure = ((q0 != q1) != q2) && !(q0 && q1) && m >= S.tp;  // exactly one
            int ax = q0 ? 0 : (q1 ? 1 : 2);
            bool nowall = false;
            if (!sure) {
                long long kt;
                ax = exit_exact(S, V, &kt);
                nowall = ax < 0;
                ml = floor_float(kdouble(kt < S.ktcur ? S.ktcur : kt));
                m = __fmaf_rn(ml, 1.0f + 0x1p-21f, 0x1p-126f);
            }
            const bool x0 = ax == 0, x1 = ax == 1;
            C.wall = x0 ? w0 : (x1 ? w1 : w2);
            const int32_t g0 = dneg(sg, 0) ? V.first(0) : V.first(1);
            const int32_t g1 = dneg(sg, 1) ? V.first(2) : V.first(3);
            const int32_t g2 = dneg(sg, 2) ? V.first(4) : V.first(5);
            int32_t f = x0 ? g0 : (x1 ? g1 : g2);
            // exit point
            const float wid = m - ml;
            const float tm = __fmaf_rn(-0.5f, wid, m);
            C.eps = __fmaf_rn(ep.x, wid, ep.y);
            const float p0 = __fmaf_rn(A0.w, tm, A0.x), p1 = __fmaf_rn(A1.w, tm, A1.x), p2 = __fmaf_rn(A2.w, tm, A2.x);
            C.p1 = x0 ? p1 : p0;
            C.p2 = (x0 || x1) ? p2 : p1;
            C.ax = ax;
            S.tp = m;
            if (f >= 1 << kStepShift) {  // which of two or four equal neighbors
                const uint32_t steps = (uint32_t)f >> kStepShift;
                const bool x2 = ax == 2;
                const float m1 = 0.5f * (x0 ? V.lo(1) + V.hi(1) : V.lo(0) + V.hi(0));
                const float m2 = 0.5f * (x2 ? V.lo(1) + V.hi(1) : V.lo(2) + V.hi(2));
                f &= (1 << kStepShift) - 1;
                f += C.p1 >= m1 ? (1 << (steps & 3u)) >> 1 : 0;
                f += C.p2 >= m2 ? (1 << (steps >> 2)) >> 1 : 0;
            }
            const double rho = V.rho();
            const float rho32 = USE32 ? V.rho32() : 0.0f;
            if (nowall) f = -1;
            if (f >= 0) {
                C.id = f;
                V.load(records() + f);
            } else if (f < -1) {  // locate the exit point below the rope node
                C.id = -2 - f;
                C.left = G.max_depth + 1;
                V.load_node(G, C.id);
                state = LANE_NODE;
            }
            // the exit time, the segment and its sums, while the next record is under way
            long long kt = KEY_INF;
            if (!nowall) kt = __double_as_longlong((widen(C.wall) - S.o(ax)) * S.ik(ax));
            bool end = f == -1, put = true;
            const long long kin = S.ktcur;
            const int hi = (int)(kt >> 32);
            S.steps--;
            if (!(hi > (int)(kin >> 32) && hi < (int)(S.klim >> 32) && S.steps >= 0)) {
                // no later than the current time, or near or past the end of the path, its segment or its steps
                const bool seg = SEGS && T.ray >= io.n_rays;
                const long long ktend = io.smax ? okey(io.smax[ray_of()]) : KEY_INF;
                const long long ktstop = seg ? io.segs[T.ray - io.n_rays].ktstop : KEY_INF;
                const bool skip = SEGS && S.klim < 0;  // the segment before records this leaf
                S.klim = ktend < ktstop ? ktend : ktstop;
                if (ktend < kt) {
                    kt = ktend;
                    end = true;
                }
                if (kt < kin) kt = kin;
                end = end || (SEGS && kt > ktstop);
                put = kt != kin && !skip;
                if (S.steps < 0) {
                    T.st = HG_RAY_STEPLIMIT;
                    kt = kin;
                    end = true;
                    put = false;
                }
            }
            S.ktcur = kt;
            if (put) {
                const double tex = __longlong_as_double(kt);
                if (T.put(io, S.cur, tex - __longlong_as_double(kin), rho, rho32, kin, tex)) end = true;
            }
            if (end) state = LANE_DONE;
        } else if (state == LANE_START) {
            const bool seg = SEGS && T.ray >= io.n_rays;
            const uint32_t sg = V.v[15];
            S.cur = (int32_t)V.v[14];
            T.st = (sg >> 8) & 0xffu;
            int rs = S.cur < 0 ? WALK_END : WALK_GO;
            rs = T.start(io, rs);
            state = LANE_DONE;
            if (SEGS && !seg && (sg & SG_SPLIT) && S.cur >= 0) {
                T.ray = -1;  // its segments do the work
            } else if (rs == WALK_GO) {
                const long long ktend = okey(__longlong_as_double(S.ktcur));
                if (ktend < S.klim) S.klim = ktend;
                if (SEGS && (sg & SG_SKIP_FIRST)) S.klim = -1;
                start_geometry(V, grid().fdom, S);
                S.sg = sg & 0x3fu;
                S.ktcur = (long long)(((unsigned long long)V.v[7] << 32) | V.v[6]);
                S.tp = __fmaf_rn(floor_float(__longlong_as_double(S.ktcur)), 1.0f + 0x1p-21f, 0x1p-126f);
                if (S.ktcur == 0) S.tp = 0.0f;
                C.enter(S.cur);
                V.load(records() + C.id);
                state = LANE_WALK;
            }
        } else if (state == LANE_NODE) {
            const DevGrid &G = grid();
            if (locate_step(G, io, ray_of(), S, V, C)) {
                if (C.left & CAND_ROOT) C.enter(C.id);
                V.load(records() + C.id);
                state = LANE_WALK;
            } else if ((--C.left & ~CAND_ROOT) > 0) {
                V.load_node(G, C.id);
            } else {
                T.st = HG_RAY_LOST;
                state = LANE_DONE;
            }
        }
    next_round:;
    }
}

}  // namespace hg
