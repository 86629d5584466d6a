// Arguments and ray queue of the single-grid walking kernels.
#pragma once

#include <cooperative_groups.h>

#include "walkf.cuh"

namespace cg = cooperative_groups;

namespace hg {

struct TraceArgs {
    DevGrid G;
    int64_t n;
    const double *o;
    const double *d;
    const double *smax;
    double kappa;
    void *tau;
    int32_t *ncross;
    uint8_t *status;
    const int64_t *seg_off;
    int32_t *seg_cell;
    void *seg_ds;
    int64_t seg_cap;
    const float *w;
    void *grad;
    uint32_t gmul, gmask;   // gradient slot of leaf c: (c * gmul) & gmask; gmul 0: slot c
    const double *rho_ext;  // densities replacing the grid's own (MODE_TAU), or NULL
    int64_t max_steps;
    unsigned long long *counter;
    const void *starts;  // RayStart or RayStartF
    const int64_t *order;  // queue position -> ray (most work first), or NULL
    int n_smem;
    int dyn;
    // path segments of split rays (queue positions before the rays), or NULL
    const unsigned long long *n_seg;
    int64_t n_seg_cap;
    const SegStart *segs;
    double *part_acc;
    int32_t *part_nc;
    int32_t *part_last;
    uint8_t *part_st;
    const int64_t *seg_base;  // emission offset of each path segment (fill walks)
    // emission staging (MODE_*_STAGE)
    void *stg_ent;
    uint32_t *stg_next;
    uint32_t stg_nchunks;
    unsigned long long *stg_ctr;
    uint32_t *stg_start_ray;
    uint32_t *stg_start_seg;
    uint32_t *stg_overflow;
    const uint32_t *run_if;  // when non-NULL, the walk runs only if *run_if != 0
    // interaction points (MODE_INTERACT)
    const double *tau_int;
    int32_t *int_cell;
    double *int_t;
};

// Stage the first n nodes of the (breadth-first) node list in shared memory.  Whole 16-byte words: the
// node array is padded to one.
__device__ __forceinline__ void stage_nodes(const void *nodes, int bytes, unsigned char *smem) {
    const int4 *src = reinterpret_cast<const int4 *>(nodes);
    int4 *dst = reinterpret_cast<int4 *>(smem);
    for (int i = threadIdx.x; i < (bytes + 15) / 16; i += blockDim.x) dst[i] = __ldg(src + i);
    __syncthreads();
}

// Rays of one grid for the walking loop: a static stride, or a
// warp-aggregated atomic on a global counter.
struct GridRays {
    static constexpr bool kSegments = true;
    const DevGrid *G;
    int64_t n;
    int32_t turn;  // (next, static schedule: rays this thread has taken; grab: turns of this warp)
    unsigned long long *counter;
    const int64_t *order;
    int64_t n_seg;  // queue positions 0 .. n_seg-1 are path segments (items n + s)
    int32_t max_steps;
    bool dyn;
    __device__ __forceinline__ explicit GridRays(const TraceArgs &A) {
        G = &A.G;
        n = A.n;
        turn = 0;
        counter = A.counter;
        order = A.order;
        max_steps = (int32_t)(A.max_steps < 0x7fffffff ? A.max_steps : 0x7fffffff);
        dyn = A.dyn != 0;
        n_seg = 0;
        if (A.n_seg && dyn) {
            const unsigned long long c = *A.n_seg;
            n_seg = (int64_t)(c < (unsigned long long)A.n_seg_cap ? c : (unsigned long long)A.n_seg_cap);
        }
    }
    __device__ __forceinline__ bool next(int64_t &ray, const DevGrid *&g, int32_t &ms) {
        g = G;
        ms = max_steps;
        if (dyn) {
            cg::coalesced_group grp = cg::coalesced_threads();
            unsigned long long base = 0;
            if (grp.thread_rank() == 0) base = atomicAdd(counter, (unsigned long long)grp.size());
            base = grp.shfl(base, 0);
            int64_t pos = (int64_t)(base + grp.thread_rank());
            if (pos < n_seg) {
                ray = n + pos;
                return true;
            }
            pos -= n_seg;
            ray = (pos < n && order) ? order[pos] : pos;
            return pos < n;
        }
        ray = ((int64_t)turn * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
        turn++;
        return ray < n;
    }
    // Up to 32 queue items for the calling warp (all lanes); 0: none left.  The first turn hands every warp
    // an equal share of the head of the queue, at the stride of the warps so that each gets heavy and
    // light ones; further items come from the counter, a quarter of a warp's share of the rest at a time.
    // The static schedule goes on at the stride of the threads.
    __device__ __forceinline__ int grab(PoolItem *pool, const WalkIO &io) {
        const int lane = threadIdx.x & 31;
        const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
        const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
        const int64_t total = n_seg + n;
        int64_t pos;
        if (!dyn) {
            pos = (turn * warps + warp) * 32 + lane;
        } else {
            const int64_t even = (total + warps - 1) / warps;
            const int64_t share = even < 32 ? even : 32;
            if (turn == 0) {
                pos = lane < share ? warp + lane * warps : total;
            } else {
                const int64_t rest = (total - share * warps) / (4 * warps);
                const int64_t chunk = rest < 4 ? 4 : (rest < 32 ? rest : 32);
                unsigned long long base = 0;
                if (lane == 0) base = atomicAdd(counter, (unsigned long long)chunk);
                base = __shfl_sync(0xffffffffu, base, 0);
                pos = lane < chunk ? share * warps + (int64_t)base + lane : total;
            }
        }
        turn++;
        const bool ok = pos < total;
        if (ok) {
            PoolItem P;
            if (pos < n_seg) {
                P.item = n + pos;
                P.of = io.segs[pos].ray;
            } else {
                P.item = order ? order[pos - n_seg] : pos - n_seg;
                P.of = P.item;
            }
            pool[lane] = P;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const char *>(io.starts) + P.item * 64));
        }
        return __popc(__ballot_sync(0xffffffffu, ok));
    }
    __device__ __forceinline__ void item(const PoolItem &, const DevGrid *&g, int32_t &ms) const {
        g = G;
        ms = max_steps;
    }
};

// Dynamic shared memory of a walking launch: the top tree nodes, then the
// threads' geometry slots (RayState) at a 16-byte boundary.
constexpr int kGeoBytes = 9 * (int)sizeof(double);
__host__ __device__ __forceinline__ size_t geo_offset(size_t node_bytes) { return (node_bytes + 15) / 16 * 16; }
__host__ __device__ __forceinline__ size_t walk_smem(size_t node_bytes, int block) {
    return geo_offset(node_bytes) + (size_t)block * kGeoBytes;
}
// The same on single-precision records: geometry slots (RayStateF), then each warp's queue items.
__host__ __device__ __forceinline__ size_t walk_smem_f(int block) {
    return (size_t)block * (kGeoBytesF + sizeof(PoolItem));
}

__device__ __forceinline__ void walk_io(const TraceArgs &A, WalkIO &io) {
    io.o = A.o;
    io.d = A.d;
    io.smax = A.smax;
    io.starts = A.starts;
    io.kappa = A.kappa;
    io.tau = A.tau;
    io.ncross = A.ncross;
    io.status = A.status;
    io.seg_off = A.seg_off;
    io.seg_cell = A.seg_cell;
    io.seg_ds = A.seg_ds;
    io.seg_cap = A.seg_cap;
    io.w = A.w;
    io.grad = A.grad;
    if (A.gmul) {
        io.gmul = A.gmul;
        io.gmask = A.gmask;
    }
    io.rho_ext = A.rho_ext;
    io.n_rays = A.n;
    io.segs = A.segs;
    io.part_acc = A.part_acc;
    io.part_nc = A.part_nc;
    io.part_last = A.part_last;
    io.part_st = A.part_st;
    io.seg_base = A.seg_base;
    io.stg_ent = A.stg_ent;
    io.stg_next = A.stg_next;
    io.stg_nchunks = A.stg_nchunks;
    io.stg_ctr = A.stg_ctr;
    io.stg_start_ray = A.stg_start_ray;
    io.stg_start_seg = A.stg_start_seg;
    io.stg_overflow = A.stg_overflow;
    io.tau_int = A.tau_int;
    io.int_cell = A.int_cell;
    io.int_t = A.int_t;
}

constexpr int kWalkNodes = 64;  // top tree nodes that the walks of 96-byte records stage by default (trace.cu)

typedef void (*KernelFn)(const TraceArgs);
KernelFn pick_kernel_f(int mode, int prec);  // single-precision records (tracef.cu)

}  // namespace hg
