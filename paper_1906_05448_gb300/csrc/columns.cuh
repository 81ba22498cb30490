// The column layout of the pipe: populations with z fastest.
//
// The pipe of Sec. 2.1 is the same in every z plane, so a whole column
// (x, y) is either fluid or solid and all cells of a fluid column have the
// same wall links with the same wall fractions. A context with a pipe keeps
// its populations, from its first step with a wall on, as
//   g[i * Np + z + zp * (x + nx * y)],   zp >= nz the column pitch, Np = nx ny zp,
// so that a warp sweeps 32 consecutive z of one column: full, aligned
// sectors on every access, no solid cell touched, and the wall a
// warp-uniform branch with uniform weights. Everything outside the sweeps
// (fields, flags, link and site lists, checkpoint files) keeps x fastest;
// the kernels here convert.
#pragma once

#include "column_index.h"
#include "lbm_internal.cuh"

namespace lbmgb {

// Addresses of a D3Q19 sweep on columns: the pull of direction i for element
// e = z + zp * column of a plane is Ap[i][e], its store Bp[i][e] (one
// address operation per access); pulls across the ends of z, and of x and y
// where columns on the box faces are swept, add a correction; e and the
// pointers are shifted where that would overflow (column_index.h).
struct ColumnPtrs {
    const void *Ap[19];  // A + i Np - (c_z + zp (c_x + nx c_y)) + shift
    void *Bp[19];        // B + i Np + shift
    int nx, ny, nz, zp, shift;
    FastDiv fd_nx;
};

// How threads walk the cells of n columns (of a list, or all of them in
// order): a warp per 32 consecutive z of one column, so that a column's wall
// is uniform over the warp and the accesses are whole sectors; or, where
// such warps would hold too many idle lanes (column_flat), the cells one
// after the other across the ends of the columns, which lie next to each
// other then (zp = nz); that walk also takes planes so large that the pulls
// need shifted offsets (column_shifted). us per step of the IBB pipe with warps
// per column, and so:
//   148 x 148 x 4    FP32 12.3 and 6.2   FP16 13.1 and 6.2   FP64 254 and 41
//   148 x 148 x 16   FP32 12.3 and 10.3  FP16 13.5 and 9.7   FP64 254 and 131
//   300 x 300 x 8    FP32 33.4 and 16.4  FP16 35.6 and 14.4  FP64 1033 and 274
//   300 x 300 x 33   FP32 75.8 and 65.4  FP16 70.5 and 49.5  FP64 2044 and 1071
//   148 x 148 x 58   FP32 37.1 and 31.3  FP16 22.1 and 20.8  FP64 505 and 456
//   148 x 148 x 438  FP32 176.4 and 179.7, FP16 124.7 and 125.1 (14 warps of
//                    32 for 438 cells: the wall and the sectors decide)
// The line at nine tenths of busy lanes is where FP64, bound by its
// arithmetic, would fall behind by more than the flat walk's ends cost FP32.
struct ColumnItems {
    unsigned n, run;  // run: warps, or cells, per column
    FastDiv fd;
    // column and z of this thread (blocks of 256); z may lie past the last plane
    template <bool FLAT>
    __device__ __forceinline__ bool cell(unsigned &ci, int &z) const {
        const unsigned t = FLAT ? blockIdx.x * 256u + threadIdx.x : blockIdx.x * 8 + threadIdx.x / 32;
        ci = fd.div(t);
        if (ci >= n) return false;
        z = FLAT ? (int)(t - ci * run) : (int)(t - ci * run) * 32 + (int)(threadIdx.x & 31);
        return true;
    }
};
inline ColumnItems column_items(const Ctx &c, long long n) {
    const unsigned run = c.col_flat ? (unsigned)c.nz : (unsigned)((c.nz + 31) / 32);
    return ColumnItems{(unsigned)n, run, FastDiv(run)};
}
inline unsigned column_item_blocks(const Ctx &c, const ColumnItems &it) {
    const unsigned long long items = (unsigned long long)it.n * it.run, per = c.col_flat ? 256 : 8;
    return (unsigned)((items + per - 1) / per);
}

inline void column_ptrs(const Ctx &c, ColumnPtrs &p) {
    const long long sb = (long long)storage_bytes(c.storage);
    p.shift = c.col_flat ? column_shift(c.Np) : 0;  // the cell-by-cell walk carries it whatever the size
    for (int i = 0; i < 19; i++) {
        const long long off = cz(i) + (long long)c.zp * (cx(i) + (long long)c.nx * cy(i)) - p.shift;
        p.Ap[i] = (const void *)((const char *)c.fA + sb * (i * c.Np - off));
        p.Bp[i] = (void *)((char *)c.fB + sb * (i * c.Np + p.shift));
    }
    p.nx = c.nx;
    p.ny = c.ny;
    p.nz = c.nz;
    p.zp = c.zp;
    p.fd_nx = FastDiv((unsigned)c.nx);
}

// the cell's element for the pointers above
template <bool SHIFT>
__device__ __forceinline__ int column_element(const ColumnPtrs &p, int col, int z) {
    return SHIFT ? col * p.zp + z - p.shift : col * p.zp + z;
}

// the 19 pulls of the cell (column, z) through ld(const T *); WRAP: the
// column may lie on an x or y face of the box; SHIFT: with p.shift
template <typename T, bool WRAP, bool SHIFT, typename R, typename Ld>
__device__ __forceinline__ void column_pull(R g[19], const ColumnPtrs &p, int col, int z, Ld ld) {
    if constexpr (SHIFT) {
        int x = 1, y = 1;  // no face unless WRAP
        if constexpr (WRAP) {
            y = (int)p.fd_nx.div((unsigned)col);
            x = col - y * p.nx;
        }
        const int e = column_element<true>(p, col, z);
        const ColumnWrap w = column_wrap(x, y, z, WRAP ? p.nx : 4, WRAP ? p.ny : 4, p.nz, p.zp);
#pragma unroll
        for (int i = 0; i < 19; i++) g[i] = ld((const T *)p.Ap[i] + column_offset(e, w, cx(i), cy(i), cz(i)));
        return;
    }
    // (through the functions above, the same offsets without the shift take the IBM pipe 4 % longer)
    const int e = col * p.zp + z;
    const int zlo = z == 0 ? p.nz : 0, zhi = z == p.nz - 1 ? p.nz : 0;
    int xlo = 0, xhi = 0, ylo = 0, yhi = 0;
    if constexpr (WRAP) {
        const int y = (int)p.fd_nx.div((unsigned)col), x = col - y * p.nx;
        const int row = p.nx * p.zp;
        xlo = x == 0 ? row : 0;
        xhi = x == p.nx - 1 ? row : 0;
        ylo = y == 0 ? row * p.ny : 0;
        yhi = y == p.ny - 1 ? row * p.ny : 0;
    }
#pragma unroll
    for (int i = 0; i < 19; i++) {
        int o = e + (cz(i) > 0 ? zlo : 0) - (cz(i) < 0 ? zhi : 0);
        if constexpr (WRAP)
            o += (cx(i) > 0 ? xlo : 0) - (cx(i) < 0 ? xhi : 0) + (cy(i) > 0 ? ylo : 0) - (cy(i) < 0 ? yhi : 0);
        g[i] = ld((const T *)p.Ap[i] + o);
    }
}

constexpr int COL_TILE = 32;  // x by z tile of the conversions, at one y

// blocks: z tiles x x tiles (linear in x, so that no grid limit is met), y
// strided beyond the limit
inline dim3 column_tiles(const Ctx &c) {
    const long long t = (long long)((c.nz + COL_TILE - 1) / COL_TILE) * ((c.nx + COL_TILE - 1) / COL_TILE);
    return dim3((unsigned)t, (unsigned)(c.ny < 65535 ? c.ny : 65535));
}

// body(x, z, value) for the cells of a block's tile in z-fast order, then in
// x-fast order: PUT(x, z) -> V runs with lanes along z, GET(x, z, V) with
// lanes along x (TOX), or the other way round; the values cross through
// shared memory (one pad word per row: no bank conflicts for 4-byte V)
template <typename V, bool TOX, typename Put, typename Get>
__device__ __forceinline__ void column_exchange(V (*sh)[COL_TILE + 1], int nx, int nz, Put put, Get get) {
    const unsigned nzt = (unsigned)((nz + COL_TILE - 1) / COL_TILE);
    const int z0 = (int)(blockIdx.x % nzt) * COL_TILE, x0 = (int)(blockIdx.x / nzt) * COL_TILE;
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5, rows = blockDim.x >> 5;
    for (int r = row; r < COL_TILE; r += rows) {
        const int x = x0 + (TOX ? r : lane), z = z0 + (TOX ? lane : r);
        if (x < nx && z < nz) {
            if (TOX) sh[lane][r] = put(x, z);  // sh[z][x]
            else sh[r][lane] = put(x, z);
        }
    }
    __syncthreads();
    for (int r = row; r < COL_TILE; r += rows) {
        const int x = x0 + (TOX ? lane : r), z = z0 + (TOX ? r : lane);
        if (x < nx && z < nz) get(x, z, TOX ? sh[r][lane] : sh[lane][r]);
    }
    __syncthreads();  // the tile is free for the next exchange
}

// Statistics of the pipe's columns: cylindrical basis and radial bin
// b = floor(r nbins / R) of a column, formed with explicitly rounded
// operations so that a cell on a bin edge falls in the same bin everywhere.
struct PipeColumn {
    double r, ca, sa;  // e_r = (ca, sa, 0), e_theta = (-sa, ca, 0); on the axis (1, 0)
    int bin;
};
// false outside the pipe or beyond the last bin
__device__ __forceinline__ bool pipe_column(const uint8_t *flags, int x, int y, int nx, int ny, double pcx, double pcy,
                                            double R, int nbins, PipeColumn &k) {
    if (x >= nx || y >= ny || (flags[x + nx * y] & FL_SOLID)) return false;
    const double dx = __dsub_rn((double)x, pcx), dy = __dsub_rn((double)y, pcy);
    k.r = sqrt(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
    k.bin = (int)floor(__ddiv_rn(__dmul_rn(k.r, (double)nbins), R));
    if (k.bin < 0 || k.bin >= nbins) return false;
    k.ca = k.r > 0.0 ? dx / k.r : 1.0;
    k.sa = k.r > 0.0 ? dy / k.r : 0.0;
    return true;
}
// 32 x 8 columns per block, numbered linearly over the section; y: runs of z
constexpr int COL_RUN = 32;  // planes per thread (more where the grid limit asks for it)
inline int column_run(int nz) { return nz / 65535 >= COL_RUN ? nz / 65535 + 1 : COL_RUN; }
inline dim3 column_blocks(int nx, int ny, int nz, int run) {
    return dim3((unsigned)(((nx + 31) / 32) * (long long)((ny + 7) / 8)), (unsigned)((nz + run - 1) / run));
}
__device__ __forceinline__ void column_of_thread(int nx, int &x, int &y) {
    const unsigned nxt = (unsigned)((nx + 31) / 32);
    x = (int)(blockIdx.x % nxt) * 32 + (int)(threadIdx.x & 31);
    y = (int)(blockIdx.x / nxt) * 8 + (int)(threadIdx.x >> 5);
}

}  // namespace lbmgb
