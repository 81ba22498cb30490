// Element offsets of the pulls on the column layout (columns.cuh), without
// CUDA, so that they are checked on the CPU up to the largest grids.
//
// A pull of direction c for the cell (x, y, z) reads element
//   z' + zp (x' + nx y'),  x' = x - c_x and so on, wrapped into the box.
// The plane pointer of the direction carries -(c_z + zp (c_x + nx c_y)) and
// -column_bias, so one 32-bit offset per access is left: the cell's own
// element plus the bias plus nz, a row or a plane across the ends. With the
// bias every offset is positive and below 2^32 (the planes hold fewer than
// 2^31 elements and a section has at least four columns each way); without
// it a signed offset overflows on planes of nearly 2^31 elements.
#pragma once

#ifdef __CUDACC__
#define LBM_HD __host__ __device__ __forceinline__
#else
#define LBM_HD inline
#endif

namespace lbmgb {

LBM_HD unsigned column_bias(int nx, int zp) { return (unsigned)(nx + 1) * (unsigned)zp + 1u; }

// what a pull adds across the low and the high end of each axis
struct ColumnWrap {
    unsigned xlo, xhi, ylo, yhi, zlo, zhi;
};
LBM_HD ColumnWrap column_wrap(int x, int y, int z, int nx, int ny, int nz, int zp) {
    const unsigned row = (unsigned)nx * (unsigned)zp, plane = row * (unsigned)ny;
    return ColumnWrap{x == 0 ? row : 0u, x == nx - 1 ? row : 0u, y == 0 ? plane : 0u, y == ny - 1 ? plane : 0u,
                      z == 0 ? (unsigned)nz : 0u, z == nz - 1 ? (unsigned)nz : 0u};
}
// e: the cell's element plus the bias
LBM_HD unsigned column_offset(unsigned e, const ColumnWrap &w, int cx, int cy, int cz) {
    return e + (cz > 0 ? w.zlo : 0u) - (cz < 0 ? w.zhi : 0u) + (cx > 0 ? w.xlo : 0u) - (cx < 0 ? w.xhi : 0u) +
           (cy > 0 ? w.ylo : 0u) - (cy < 0 ? w.yhi : 0u);
}

}  // namespace lbmgb
