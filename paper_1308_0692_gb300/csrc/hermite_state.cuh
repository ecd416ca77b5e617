// States from moments: the second-order Hermite expansion
//   h_a = w_a [rho' + xi_a . j' + 1/2 sum_ij (P'_ij - rho' delta_ij)(xi_i xi_j - delta_ij)]
// (warm start, lbm_set_moments).  A block takes 32 cells, warp w velocity row w.  Of a row,
//   h = w_x A + (w_x xi_x) B + w_x (xi_x^2 - 1) C,
// A, B, C the row's own: three FP64 operations per velocity (and the conversion), the bound of
// these kernels.  One thread per cell with the sum written out took 55 us for 128^2 x 64.
#pragma once

#include "lbm_internal.h"

namespace hermite {

// moments of a cell in units of u_ref: rho', j', P'
struct Cell {
    double rho, jx, jy, pxx, pxy, pyy;
};

// c[ix] = w_x, w_x xi_x, w_x (xi_x^2 - 1); the block's first m threads, then a barrier
__device__ __forceinline__ void row_table(double (*c)[3], const double *xi1, const double *w1, int m)
{
    if ((int)threadIdx.x < m) {
        const double x = xi1[threadIdx.x], w = w1[threadIdx.x];
        c[threadIdx.x][0] = w;
        c[threadIdx.x][1] = w * x;
        c[threadIdx.x][2] = w * (x * x - 1.0);
    }
    __syncthreads();
}

// velocity row iy of cell (x, y): planar, or (tiled32) the strip-tiled layout of batch cavities, 32
// columns a tile with velocity pairs side by side per cell
template <typename T>
__device__ __forceinline__ void put_row(const Cell &q, const double (*c)[3], double ey, double wy, int iy, int m, int x, int y,
                                        int ny, long pa, long py, T *h, bool tiled32)
{
    const double A = wy * (q.rho + ey * q.jy + 0.5 * (q.pyy - q.rho) * (ey * ey - 1.0));
    const double B = wy * (q.jx + q.pxy * ey), C = 0.5 * wy * (q.pxx - q.rho);
    const long co = tiled32 ? (long)(x >> 5) * (32L * m * m * ny) + y * (32L * m * m) + (x & 31) * 2 : y * py + x;
#pragma unroll 4
    for (int ix = 0; ix < m; ++ix) {
        const double v = c[ix][0] * A + (c[ix][1] * B + c[ix][2] * C);
        const int a = iy * m + ix;
        h[(tiled32 ? (long)(a >> 1) * 64 + (a & 1) : (long)a * pa) + co] = (T)v;
    }
}

}  // namespace hermite
