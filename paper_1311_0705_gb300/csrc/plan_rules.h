// Rules of the work estimate and of the path-segment planner as plain functions, for the kernels and for host
// programs.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define HG_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define HG_HOST_DEVICE inline
#endif

namespace hg {

// Cell of a lattice of 16 along one axis.  A coordinate x of 0 .. 16 enters as p = x kLatticeScale - kLatticeShift: less 1/2,
// and drawn in towards the middle by 2^-13 of a cell, so that the domain's faces, and points past them by rounding,
// count for the cells they touch.  The cell is read off the low mantissa bits of p + 1.5 * 2^23, a sum of numbers of spacing
// 1 whichever sign p has (next to 2^23 itself, half of it below: the lower quarter of cell 0 counted for cell 15).  A
// coordinate within 2^-13 of another cell may count for that one.
constexpr float kLatticeScale = 1.0f - 0x1p-16f, kLatticeShift = 0.5f - 0x1p-13f;
HG_HOST_DEVICE uint32_t lattice_cell(float p) {
    const float x = p + 0x1.8p23f;
    uint32_t b;
    memcpy(&b, &x, 4);
    return b & 15u;
}

// Whether cut c of a path is made: candidates 0 .. c in path order by their numbers, at times t (minus infinity where there is
// none) in leaves `leaf`.  A cut is made when it lies later than the last one made and in another leaf (the path
// starts at t0 in leaf0).
HG_HOST_DEVICE bool cut_made(const float *t, const int32_t *leaf, int c, float t0, int32_t leaf0) {
    bool made = false;
    for (int j = 0; j <= c; j++) {
        made = t[j] > t0 && leaf[j] != leaf0;
        t0 = made ? t[j] : t0;
        leaf0 = made ? leaf[j] : leaf0;
    }
    return made;
}

}  // namespace hg
