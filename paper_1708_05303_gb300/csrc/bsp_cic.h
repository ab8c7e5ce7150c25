// bsp_cic.h -- where a position outside [0, box) falls on the periodic grid.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define BSP_HD __host__ __device__ __forceinline__
#else
#define BSP_HD inline
#endif

namespace bsp {

// Cell 0 .. n - 1 and fraction 0 .. 1 of coordinate u (cell units) on an axis of n cells, wrapped.
// The wrapped value can round to n itself (u = -1e-15: it is cell 0), and beyond 2^53
// cells it is any remainder of the rounding, or NaN: whatever is not in [0, n) goes to 0,
// so that no position, however wrong, is written outside the grid.
BSP_HD void cic_wrap(double u, int n, int& cell, float& frac) {
    u -= floor(u / n) * n;
    if (!(u >= 0.0 && u < (double)n)) u = 0.0;
    cell = (int)u;
    frac = (float)(u - (double)cell);
}

}  // namespace bsp
