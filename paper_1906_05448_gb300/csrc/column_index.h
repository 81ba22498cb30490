// Element offsets of the pulls on the column layout (columns.cuh) where
// columns on the faces of the box are swept, without CUDA, so that they are
// checked on the CPU up to the largest grids.
//
// A pull of direction c for the cell (x, y, z) reads element
//   z' + zp (x' + nx y'),  x' = x - c_x and so on, wrapped into the box.
// The plane pointer of the direction carries -(c_z + zp (c_x + nx c_y)) and
// +column_shift, so one signed 32-bit offset per access is left: the cell's
// own element less the shift, plus nz, a row or a plane across the ends.
// With the shift (half a plane) every offset lies within 0.9 of 2^31 (planes
// hold fewer than 2^31 elements, sections at least four columns each way);
// without it those across the low faces overflow on planes of nearly 2^31.
#pragma once

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbmgb {

// Whether the sweeps walk cells across the ends of the columns: 32-cell warps
// of single columns would hold more than a tenth of idle lanes.
LBM_HD bool column_flat(int nz) { return 10LL * nz < 9LL * ((nz + 31) / 32 * 32); }

// Whether pulls that wrap in x and y need the shift.
LBM_HD bool column_shifted(int nx, int zp, long long plane) { return plane + (long long)(nx + 2) * zp >= (1LL << 31); }
LBM_HD int column_shift(long long plane) { return (int)(plane / 2); }

// what a pull adds across the low and the high end of each axis
struct ColumnWrap {
    int xlo, xhi, ylo, yhi, zlo, zhi;
};
LBM_HD ColumnWrap column_wrap(int x, int y, int z, int nx, int ny, int nz, int zp) {
    const int row = nx * zp;
    return ColumnWrap{x == 0 ? row : 0, x == nx - 1 ? row : 0, y == 0 ? row * ny : 0, y == ny - 1 ? row * ny : 0,
                      z == 0 ? nz : 0, z == nz - 1 ? nz : 0};
}
// e: the cell's element less the shift
LBM_HD int column_offset(int e, const ColumnWrap &w, int cx, int cy, int cz) {
    return e + (cz > 0 ? w.zlo : 0) - (cz < 0 ? w.zhi : 0) + (cx > 0 ? w.xlo : 0) - (cx < 0 ? w.xhi : 0) +
           (cy > 0 ? w.ylo : 0) - (cy < 0 ? w.yhi : 0);
}

}  // namespace lbmgb
