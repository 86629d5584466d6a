// Walking kernels of the grids with single-precision records (walkf.cuh).
#include <cuda_runtime.h>

#include "hg_internal.h"
#include "trace_args.cuh"
#include "walkf.cuh"

namespace hg {

// As trace_kernel (trace.cu), either tree and navigation.  Four blocks of 256 threads per SM at 64 registers;
// the interaction search, which carries the drawn depth and its own state, spills 72 bytes there and runs
// with three blocks at 80 (1e6 packets, disk octree: call 747 -> 687 us).
template <int MODE, int PREC>
__global__ void __launch_bounds__(256, MODE == MODE_INTERACT ? 3 : 4) trace_kernel_f(const __grid_constant__ TraceArgs A) {
    extern __shared__ __align__(16) unsigned char smem[];
    if (A.run_if && *A.run_if == 0u) return;  // a fallback walk with nothing to do
    GridRays src(A);
    WalkIO io;
    walk_io(A, io);
    walk_loop_f<MODE, PREC>(src, io, smem, reinterpret_cast<PoolItem *>(smem + blockDim.x * kGeoBytesF));
}

KernelFn pick_kernel_f(int mode, int prec) {
    static const KernelFn table[7][4] = {
        {&trace_kernel_f<MODE_TAU, 0>, &trace_kernel_f<MODE_TAU, 1>, nullptr, nullptr},
        {&trace_kernel_f<MODE_FILL, 0>, &trace_kernel_f<MODE_FILL, 1>, nullptr, nullptr},
        {&trace_kernel_f<MODE_ADJ, 0>, &trace_kernel_f<MODE_ADJ, 1>, nullptr, nullptr},
        {&trace_kernel_f<MODE_TAUADJ, 0>, &trace_kernel_f<MODE_TAUADJ, 1>, &trace_kernel_f<MODE_TAUADJ, 2>,
         &trace_kernel_f<MODE_TAUADJ, 3>},
        {&trace_kernel_f<MODE_TAU_STAGE, 0>, &trace_kernel_f<MODE_TAU_STAGE, 1>, nullptr, nullptr},
        {&trace_kernel_f<MODE_TAUADJ_STAGE, 0>, &trace_kernel_f<MODE_TAUADJ_STAGE, 1>,
         &trace_kernel_f<MODE_TAUADJ_STAGE, 2>, &trace_kernel_f<MODE_TAUADJ_STAGE, 3>},
        {&trace_kernel_f<MODE_INTERACT, 0>, nullptr, nullptr, nullptr}};
    return table[mode][prec];
}

}  // namespace hg
