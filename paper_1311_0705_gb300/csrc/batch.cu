// Batched launch over many grids and the launch-shape autotuner.
//
// The rays of all grids form one queue, ordered so that the grids with the
// most rays come first; persistent threads take queue positions through a
// warp-aggregated atomic counter, map a position to (grid, ray) with a
// binary search over the per-grid queue offsets held in shared memory, and
// walk it with the same per-crossing loop as the single-grid kernel.  One
// launch covers the whole batch, so it can be captured in a CUDA graph.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <numeric>
#include <vector>

#include "hg_internal.h"
#include "scratch.h"
#include "trace_args.cuh"
#include "walkf.cuh"

namespace cg = cooperative_groups;

namespace hg {
hg_status cuda_err(cudaError_t e, const char *what);
int sm_count();

constexpr int kMaxBatch = 1024;

struct BatchEntry {
    DevGrid G;
    int64_t ray0;
    int64_t max_steps;
};

struct BatchArgs {
    const BatchEntry *E;
    const int64_t *qbeg;  // [n_grids+1] queue offsets in processing order
    const int32_t *perm;  // [n_grids] grid at each queue slot
    int n_grids;
    int64_t total;
    const double *o;
    const double *d;
    const double *smax;
    double kappa;
    void *tau;
    int32_t *ncross;
    uint8_t *status;
    int64_t max_steps;  // 0: per grid 4 n_leaves + 64
    unsigned long long *counter;
    void *starts;       // [total] start records (RayStart or RayStartF), indexed by ray
};

// Queue position -> slot (grid in processing order) by binary search.
__device__ __forceinline__ int queue_slot(const int64_t *s_qbeg, int n_grids, int64_t q) {
    int lo = 0, hi = n_grids - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_qbeg[mid] <= q)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Setup pass over the whole batch (checks, 1/d, clip, first leaf).  F: the grids hold single-precision
// records.
template <bool F>
__global__ void __launch_bounds__(256) batch_setup_kernel(const BatchArgs A) {
    __shared__ int64_t s_qbeg[kMaxBatch + 1];
    __shared__ int32_t s_perm[kMaxBatch];
    for (int i = threadIdx.x; i <= A.n_grids; i += blockDim.x) s_qbeg[i] = A.qbeg[i];
    for (int i = threadIdx.x; i < A.n_grids; i += blockDim.x) s_perm[i] = A.perm[i];
    __syncthreads();
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < A.total; q += (int64_t)gridDim.x * blockDim.x) {
        const int slot = queue_slot(s_qbeg, A.n_grids, q);
        const BatchEntry *E = A.E + s_perm[slot];
        const int64_t ray = E->ray0 + (q - s_qbeg[slot]);
        const DevGrid &G = E->G;
        const RayStart R = ray_setup(
            G,
            [&](long long p0, long long p1, long long p2, uint32_t sg) {
                return F ? locate_key_f<2>(G, nullptr, 0, p0, p1, p2, sg) : descend<2>(G, nullptr, 0, p0, p1, p2, sg);
            },
            A.o, A.d, A.smax, ray);
        if (F)
            static_cast<RayStartF *>(A.starts)[ray] = start_f(R, A.o, A.d, ray);
        else
            static_cast<RayStart *>(A.starts)[ray] = R;
    }
}

// Rays of the whole batch: queue positions from a warp-aggregated atomic
// counter, mapped to (grid, ray) through the queue offsets in shared memory.
struct BatchRays {
    static constexpr bool kSegments = false;
    const BatchArgs *A;
    const int64_t *s_qbeg;
    const int32_t *s_perm;
    __device__ __forceinline__ bool next(int64_t &ray, const DevGrid *&g, int32_t &ms) {
        cg::coalesced_group grp = cg::coalesced_threads();
        unsigned long long base = 0;
        if (grp.thread_rank() == 0) base = atomicAdd(A->counter, (unsigned long long)grp.size());
        base = grp.shfl(base, 0);
        const int64_t q = (int64_t)(base + grp.thread_rank());
        if (q >= A->total) return false;
        const int slot = queue_slot(s_qbeg, A->n_grids, q);
        const BatchEntry *E = A->E + s_perm[slot];
        ray = E->ray0 + (q - s_qbeg[slot]);
        g = &E->G;
        const int64_t m = A->max_steps > 0 ? A->max_steps : E->max_steps;
        ms = (int32_t)(m < 0x7fffffff ? m : 0x7fffffff);
        return true;
    }
    // Up to 32 items for the calling warp (GridRays::grab); with each item's grid.
    __device__ __forceinline__ int grab(PoolItem *pool, const WalkIO &) const {
        const int lane = threadIdx.x & 31;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(A->counter, 32ULL);
        base = __shfl_sync(0xffffffffu, base, 0);
        const int64_t q = (int64_t)base + lane;
        const bool ok = q < A->total;
        if (ok) {
            const int slot = queue_slot(s_qbeg, A->n_grids, q);
            const int32_t g = s_perm[slot];
            PoolItem P;
            P.item = A->E[g].ray0 + (q - s_qbeg[slot]);
            P.of = g;
            pool[lane] = P;
            asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const RayStartF *>(A->starts) + P.item));
        }
        return __popc(__ballot_sync(0xffffffffu, ok));
    }
    __device__ __forceinline__ void item(const PoolItem &P, const DevGrid *&g, int32_t &ms) const {
        const BatchEntry *E = A->E + P.of;
        g = &E->G;
        const int64_t m = A->max_steps > 0 ? A->max_steps : E->max_steps;
        ms = (int32_t)(m < 0x7fffffff ? m : 0x7fffffff);
    }
};

// NAV: 0 every grid holds neighbor lists, 1 every grid ropes, 2 a mix (read per grid); 3 the grids hold
// single-precision records with either.
template <int PREC, int NAV>
__global__ void __launch_bounds__(256, NAV == 3 ? 4 : 1) batch_kernel(const BatchArgs A) {
    __shared__ int64_t s_qbeg[kMaxBatch + 1];
    __shared__ int32_t s_perm[kMaxBatch];
    // the walking threads' ray geometry (blocks of at most 256)
    __shared__ __align__(16) unsigned char s_geo[256 * (NAV == 3 ? kGeoBytesF : kGeoBytes)];
    for (int i = threadIdx.x; i <= A.n_grids; i += blockDim.x) s_qbeg[i] = A.qbeg[i];
    for (int i = threadIdx.x; i < A.n_grids; i += blockDim.x) s_perm[i] = A.perm[i];
    __syncthreads();
    BatchRays src{&A, s_qbeg, s_perm};
    WalkIO io{};
    io.o = A.o;
    io.d = A.d;
    io.smax = A.smax;
    io.starts = A.starts;
    io.kappa = A.kappa;
    io.tau = A.tau;
    io.ncross = A.ncross;
    io.status = A.status;
    if constexpr (NAV == 3) {
        __shared__ PoolItem s_pool[256];
        walk_loop_f<MODE_TAU, PREC>(src, io, s_geo, s_pool);
    } else
        walk_loop<2, MODE_TAU, PREC, NAV>(src, io, nullptr, 0, reinterpret_cast<double *>(s_geo));
}

}  // namespace hg

// The grids of a batch in one or two queues, one launch each: those with double-precision records and those
// with single-precision ones.
struct hg_batch {
    struct Queue {
        int n_grids = 0;
        int64_t total = 0;
        int64_t *d_qbeg = nullptr;
        int32_t *d_perm = nullptr;
        unsigned long long *d_counter = nullptr;
        int nav = 0;  // as batch_kernel's NAV
    } q[2];
    int n_grids = 0;
    int64_t total = 0;  // rays of the whole batch
    hg::BatchEntry *d_entries = nullptr;
    int device = 0;
};

using namespace hg;

extern "C" hg_status hg_batch_create(int32_t n_grids, const hg_grid *const *grids, const int64_t *ray_begin,
                                     int32_t chunk, hg_batch **out) {
    (void)chunk;
    if (!out || !grids || !ray_begin || n_grids < 1 || n_grids > kMaxBatch) {
        set_error("hg_batch_create: need 1..%d grids, grid pointers and ray offsets", kMaxBatch);
        return HG_EINVAL;
    }
    *out = nullptr;
    if (ray_begin[0] != 0) {
        set_error("hg_batch_create: ray_begin[0] must be 0");
        return HG_EINVAL;
    }
    std::vector<BatchEntry> ent((size_t)n_grids);
    std::vector<int64_t> cnt((size_t)n_grids);
    for (int i = 0; i < n_grids; i++) {
        if (!grids[i] || ray_begin[i + 1] < ray_begin[i]) {
            set_error("hg_batch_create: bad grid %d or ray range", i);
            return HG_EINVAL;
        }
        ent[i].G = grids[i]->d;
        ent[i].ray0 = ray_begin[i];
        ent[i].max_steps = 4 * grids[i]->d.n_leaves + 64;
        cnt[i] = ray_begin[i + 1] - ray_begin[i];
    }
    hg_batch *b = new hg_batch();
    b->n_grids = n_grids;
    b->total = ray_begin[n_grids];
    cudaGetDevice(&b->device);
    cudaError_t e = device_malloc((void **)&b->d_entries, ent.size() * sizeof(BatchEntry));
    if (e == cudaSuccess) e = cudaMemcpy(b->d_entries, ent.data(), ent.size() * sizeof(BatchEntry), cudaMemcpyHostToDevice);
    for (int f = 0; f < 2 && e == cudaSuccess; f++) {
        hg_batch::Queue &Q = b->q[f];
        std::vector<int32_t> perm;
        int n_ropes = 0;
        for (int i = 0; i < n_grids; i++)
            if ((grids[i]->d.recf != nullptr) == (f == 1)) {
                perm.push_back(i);
                n_ropes += grids[i]->d.nav == HG_NAV_ROPES ? 1 : 0;
            }
        if (perm.empty()) continue;
        // largest ray counts first, so that the long queues start early
        std::stable_sort(perm.begin(), perm.end(), [&](int32_t x, int32_t y) { return cnt[x] > cnt[y]; });
        std::vector<int64_t> qbeg(perm.size() + 1, 0);
        for (size_t s = 0; s < perm.size(); s++) qbeg[s + 1] = qbeg[s] + cnt[perm[s]];
        Q.n_grids = (int)perm.size();
        Q.nav = f == 1 ? 3 : (n_ropes == 0 ? 0 : (n_ropes == Q.n_grids ? 1 : 2));
        Q.total = qbeg.back();
        e = device_malloc((void **)&Q.d_qbeg, qbeg.size() * sizeof(int64_t));
        if (e == cudaSuccess) e = device_malloc((void **)&Q.d_perm, perm.size() * sizeof(int32_t));
        if (e == cudaSuccess) e = device_malloc((void **)&Q.d_counter, sizeof(unsigned long long));
        if (e == cudaSuccess) e = cudaMemcpy(Q.d_qbeg, qbeg.data(), qbeg.size() * sizeof(int64_t), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(Q.d_perm, perm.data(), perm.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    }
    if (e != cudaSuccess) {
        hg_batch_free(b);
        return cuda_err(e, "hg_batch_create");
    }
    *out = b;
    return HG_OK;
}

extern "C" void hg_batch_free(hg_batch *b) {
    if (!b) return;
    cudaFree(b->d_entries);
    for (auto &Q : b->q) {
        cudaFree(Q.d_qbeg);
        cudaFree(Q.d_perm);
        cudaFree(Q.d_counter);
    }
    delete b;
}

extern "C" hg_status hg_batch_trace(hg_batch *b, const double *o, const double *d, const double *s_max,
                                    double kappa, const hg_trace_opts *opts, void *tau, int32_t *ncross,
                                    uint8_t *ray_status, hg_stream stream) {
    if (!b || (b->total > 0 && (!o || !d || !tau || !ncross))) {
        set_error("hg_batch_trace: bad arguments");
        return HG_EINVAL;
    }
    const int prec = opts ? opts->precision : HG_FP64;
    if (prec != HG_FP64 && prec != HG_FP32K) {
        set_error("hg_batch_trace: bad precision");
        return HG_EINVAL;
    }
    if (b->total == 0) return HG_OK;
    cudaStream_t s = (cudaStream_t)stream;
    BatchArgs A{};
    A.E = b->d_entries;
    A.o = o;
    A.d = d;
    A.smax = s_max;
    A.kappa = kappa;
    A.tau = tau;
    A.ncross = ncross;
    A.status = ray_status;
    A.max_steps = opts ? opts->max_steps : 0;
    const int block = (opts && opts->block > 0) ? opts->block : 256;
    if (block < 32 || block > 256 || block % 32) {
        set_error("hg_batch_trace: block must be a multiple of 32 in 32..256");
        return HG_EINVAL;
    }
    using BatchFn = void (*)(const BatchArgs);
    static const BatchFn kernels[2][4] = {{&batch_kernel<HG_FP64, 0>, &batch_kernel<HG_FP64, 1>, &batch_kernel<HG_FP64, 2>,
                                           &batch_kernel<HG_FP64, 3>},
                                          {&batch_kernel<HG_FP32K, 0>, &batch_kernel<HG_FP32K, 1>,
                                           &batch_kernel<HG_FP32K, 2>, &batch_kernel<HG_FP32K, 3>}};
    // start records of either kind, indexed by ray: two queues never share a record's bytes
    const size_t rec = b->q[1].total > 0 ? sizeof(RayStartF) : sizeof(RayStart);
    const size_t both = b->q[0].total > 0 && b->q[1].total > 0 ? (size_t)b->total * sizeof(RayStart) : 0;
    Scratch scratch;
    cudaError_t e = scratch_get(scratch, (size_t)b->total * rec + both, s);
    if (e != cudaSuccess) return cuda_err(e, "batch start scratch");
    unsigned char *starts = static_cast<unsigned char *>(scratch.p);
    for (int f = 0; f < 2 && e == cudaSuccess; f++) {
        const hg_batch::Queue &Q = b->q[f];
        if (Q.total == 0) continue;
        A.qbeg = Q.d_qbeg;
        A.perm = Q.d_perm;
        A.n_grids = Q.n_grids;
        A.total = Q.total;
        A.counter = Q.d_counter;
        A.starts = f == 0 && both ? starts + (size_t)b->total * rec : starts;
        const BatchFn kern = kernels[prec == HG_FP64 ? 0 : 1][Q.nav];
        int per_sm = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, block, 0);
        if (e != cudaSuccess) break;
        int64_t blocks = (int64_t)std::max(1, per_sm) * sm_count();
        blocks = std::min<int64_t>(blocks, (Q.total + block - 1) / block);
        e = cudaMemsetAsync(Q.d_counter, 0, sizeof(unsigned long long), s);
        if (e != cudaSuccess) break;
        const int64_t sblocks = std::min<int64_t>((Q.total + 255) / 256, (int64_t)sm_count() * 8);
        if (f == 1)
            batch_setup_kernel<true><<<(unsigned)sblocks, 256, 0, s>>>(A);
        else
            batch_setup_kernel<false><<<(unsigned)sblocks, 256, 0, s>>>(A);
        kern<<<(unsigned)blocks, block, 0, s>>>(A);
        note_launches(2);
        e = cudaGetLastError();
    }
    scratch_put(scratch, s);
    return e == cudaSuccess ? HG_OK : cuda_err(e, "batch launch");
}

// ------------------------------------------------------------------ autotuner

extern "C" hg_status hg_autotune(hg_grid *g, int64_t n, const double *o, const double *d, int32_t precision,
                                 hg_trace_opts *best, float *best_ms, hg_stream stream) {
    if (!g || n <= 0 || !o || !d || (precision != HG_FP64 && precision != HG_FP32K)) {
        set_error("hg_autotune: bad arguments");
        return HG_EINVAL;
    }
    cudaStream_t s = (cudaStream_t)stream;
    Scratch scratch;
    cudaError_t e = scratch_get(scratch, (size_t)n * 12, s);
    if (e != cudaSuccess) return cuda_err(e, "hg_autotune scratch");
    void *tau = scratch.p;
    int32_t *nc = reinterpret_cast<int32_t *>(static_cast<unsigned char *>(scratch.p) + (size_t)n * 8);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    const int node_bytes = node_bytes_of(g->d);
    const int blocks[] = {128, 256};
    // walks of 64-byte records stage no nodes and have one form each: neither choice makes a difference there, and
    // the defaults stand for both
    const bool one_form = g->d.recf != nullptr;
    const int nodes_at[] = {one_form ? kWalkNodes : 0, 8 * 1024 / node_bytes, 32 * 1024 / node_bytes, 64 * 1024 / node_bytes};
    const int n_nodes_at = one_form ? 1 : 4;
    hg_trace_opts win{};
    float win_ms = 1e30f;
    hg_status st = HG_OK;
    for (int sched = 1; sched <= 3 && st == HG_OK; sched++)
        for (int occ = one_form ? 4 : 3; occ <= 4; occ++)
            for (int bl : blocks)
                for (int j = 0; j < n_nodes_at; j++) {
                    hg_trace_opts op{};
                    op.precision = precision;
                    op.block = bl;
                    op.smem_nodes = (int)std::min<int64_t>(g->d.n_nodes, nodes_at[j]);
                    op.schedule = sched;
                    op.min_blocks = occ;
                    st = hg_trace_rays(g, n, o, d, nullptr, 1.0, &op, tau, nc, nullptr, stream);
                    if (st == HG_EINVAL) {  // shape does not fit: skip it
                        st = HG_OK;
                        continue;
                    }
                    if (st != HG_OK) break;
                    float best_here = 1e30f;
                    for (int rep = 0; rep < 3; rep++) {
                        cudaEventRecord(e0, s);
                        st = hg_trace_rays(g, n, o, d, nullptr, 1.0, &op, tau, nc, nullptr, stream);
                        cudaEventRecord(e1, s);
                        cudaEventSynchronize(e1);
                        float ms = 0.f;
                        cudaEventElapsedTime(&ms, e0, e1);
                        best_here = std::min(best_here, ms);
                    }
                    if (best_here < win_ms) {
                        win_ms = best_here;
                        win = op;
                    }
                }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    scratch_put(scratch, s);
    cudaStreamSynchronize(s);
    if (st != HG_OK) return st;
    TuneEntry &T = g->tuned[precision];
    T.valid = 1;
    T.block = win.block;
    T.smem_nodes = win.smem_nodes;
    T.schedule = win.schedule;
    T.min_blocks = win.min_blocks;
    if (best) *best = win;
    if (best_ms) *best_ms = win_ms;
    return HG_OK;
}
