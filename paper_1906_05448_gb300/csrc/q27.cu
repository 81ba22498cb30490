// D3Q27 on a periodic box: the velocity set of the paper's pipe solver
// (Sec. 2.1: D3Q27 MRT run with a single relaxation parameter, i.e. BGK).
// Same storage (shifted g = f - w_i, FP64 or FP32), pull streaming, Guo
// forcing and post-collision stored state as the D3Q19 path.
//
// Velocity order (the interface of populations in and out): rest, the 6
// faces, the 12 edges, the 8 corners; within a group the triples
// (c_x, c_y, c_z) over {-1, 0, 1}^3 in lexicographic order (c_x slowest).
// Weights 8/27, 2/27, 1/54, 1/216 by |c|^2 = 0 .. 3.
#include "columns.cuh"

#include <vector>

namespace lbmgb {

namespace {

// components as characters '0', '1', '2' for -1, 0, 1 (compile-time lookups)
__host__ __device__ constexpr int q27x(int i) { return "101111200001111222200002222"[i] - '1'; }
__host__ __device__ constexpr int q27y(int i) { return "110112101120022011200220022"[i] - '1'; }
__host__ __device__ constexpr int q27z(int i) { return "111021110210202102102020202"[i] - '1'; }
__host__ __device__ constexpr double q27w(int i) {
    return i == 0 ? 8.0 / 27.0 : (i <= 6 ? 2.0 / 27.0 : (i <= 18 ? 1.0 / 54.0 : 1.0 / 216.0));
}
static_assert(q27x(1) == -1 && q27y(1) == 0 && q27z(1) == 0, "first face");
static_assert(q27x(26) == 1 && q27y(26) == 1 && q27z(26) == 1, "last corner");
static_assert(q27x(7) * q27x(7) + q27y(7) * q27y(7) + q27z(7) * q27z(7) == 2, "first edge");
static_assert(q27x(19) * q27x(19) + q27y(19) * q27y(19) + q27z(19) * q27z(19) == 3, "first corner");

constexpr int Q27 = 27;

template <int S>
__global__ void q27_init_kernel(void *A, const double *u, double rho0, long long N) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const double ux = u[c], uy = u[N + c], uz = u[2 * N + c];
    const double u2 = ux * ux + uy * uy + uz * uz;
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        const double cu = q27x(i) * ux + q27y(i) * uy + q27z(i) * uz;
        const double feq = q27w(i) * rho0 * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * u2);
        Store<S>::st((T *)A + (size_t)i * N + c, R(feq - q27w(i)));
    }
}

template <int S>
__global__ void q27_plane_kernel(void *A, double *v, long long N, int i, int to_f64) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    T *p = (T *)A + (size_t)i * N + c;
    const double w = q27w(i);
    if (to_f64) v[c] = (double)Store<S>::ld(p) + w;
    else Store<S>::st(p, R(v[c] - w));
}

// rho and u of the post-collision state: sum f c = rho u + F/2
template <int S>
__global__ void q27_macro_kernel(const void *A, float4 *rec, double *rho_o, double *u_o, long long N, double F0, double F1,
                                 double F2) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const T *P = (const T *)A;
    R r = R(0), j0 = R(0), j1 = R(0), j2 = R(0);
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        const R g = Store<S>::ld(P + (size_t)i * N + c);
        r += g;
        j0 += g * R(q27x(i));
        j1 += g * R(q27y(i));
        j2 += g * R(q27z(i));
    }
    const R rho = R(1) + r, ir = R(1) / rho;
    if (rec) {
        rec[c] = make_float4(float((j0 - R(0.5) * R(F0)) * ir), float((j1 - R(0.5) * R(F1)) * ir),
                             float((j2 - R(0.5) * R(F2)) * ir), float(rho));
        return;
    }
    rho_o[c] = double(rho);
    u_o[c] = double((j0 - R(0.5) * R(F0)) * ir);
    u_o[N + c] = double((j1 - R(0.5) * R(F1)) * ir);
    u_o[2 * N + c] = double((j2 - R(0.5) * R(F2)) * ir);
}

// the same on the column layout (columns.cuh): read along z, written along x.
// Solid columns are never swept and their populations are undefined (calls
// that use the idle buffer as scratch leave their bytes there): they report
// the state at rest, g = 0.
template <int S>
__global__ void __launch_bounds__(256) q27_column_macro_kernel(const void *A, const unsigned *colmask, float4 *rec, double *rho_o,
                                                               double *u_o, int nx, int ny, int nz, int zp, long long N,
                                                               long long Np, double F0, double F1, double F2) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    struct V {
        R rho, ux, uy, uz;
    };
    __shared__ V sh[COL_TILE][COL_TILE + 1];
    for (int y = blockIdx.y; y < ny; y += gridDim.y)
        column_exchange<V, true>(
            sh, nx, nz,
            [&](int x, int z) {
                const T *P = (const T *)A + (size_t)(x + nx * y) * zp + z;
                R r = R(0), j0 = R(0), j1 = R(0), j2 = R(0);
                if (!(__ldg(colmask + x + nx * y) & 1u)) {
#pragma unroll
                    for (int i = 0; i < Q27; i++) {
                        const R g = Store<S>::ld(P + i * Np);
                        r += g;
                        j0 += g * R(q27x(i));
                        j1 += g * R(q27y(i));
                        j2 += g * R(q27z(i));
                    }
                }
                const R rho = R(1) + r, ir = R(1) / rho;
                return V{rho, (j0 - R(0.5) * R(F0)) * ir, (j1 - R(0.5) * R(F1)) * ir, (j2 - R(0.5) * R(F2)) * ir};
            },
            [&](int x, int z, const V &v) {
                const long long c = x + (long long)nx * (y + (long long)ny * z);
                if (rec) {
                    rec[c] = make_float4(float(v.ux), float(v.uy), float(v.uz), float(v.rho));
                    return;
                }
                rho_o[c] = double(v.rho);
                u_o[c] = double(v.ux);
                u_o[N + c] = double(v.uy);
                u_o[2 * N + c] = double(v.uz);
            });
}

struct Q27Args {
    const void *A;
    void *B;
    long long N;
    int nx, ny, nz;
    FastDiv fx, fxy;  // division by nx and nx * ny
    double om;        // 1 / tau
    double F[3];
    unsigned *status;
};

// one cell per thread: pull f_i(x) = f*_i(x - c_i) (periodic), BGK with the
// Guo source, store the post-collision values
template <int S, bool FORCE>
__global__ void __launch_bounds__(256) q27_sweep_kernel(Q27Args a) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.N) return;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const unsigned zq = a.fxy.div((unsigned)c), rem = (unsigned)c - zq * (unsigned)(nx * ny);
    const unsigned yq = a.fx.div(rem);
    const int z = (int)zq, y = (int)yq, x = (int)(rem - yq * (unsigned)nx);
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
    const int zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
    const T *__restrict__ A = (const T *)a.A;
    T *__restrict__ B = (T *)a.B;
    const size_t N = (size_t)a.N;
    R g[Q27];
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        const int xs = q27x(i) > 0 ? xm : (q27x(i) < 0 ? xp : x);
        const int ys = q27y(i) > 0 ? ym : (q27y(i) < 0 ? yp : y);
        const int zs = q27z(i) > 0 ? zm : (q27z(i) < 0 ? zp : z);
        g[i] = Store<S>::ld(A + (i * N + (size_t)(xs + nx * (ys + ny * zs))));
    }
    R drho = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        drho += g[i];
        if (q27x(i)) jx += q27x(i) > 0 ? g[i] : -g[i];
        if (q27y(i)) jy += q27y(i) > 0 ? g[i] : -g[i];
        if (q27z(i)) jz += q27z(i) > 0 ? g[i] : -g[i];
    }
    const R Fx = FORCE ? R(a.F[0]) : R(0), Fy = FORCE ? R(a.F[1]) : R(0), Fz = FORCE ? R(a.F[2]) : R(0);
    const R rho = R(1) + drho, ir = R(1) / rho;
    const R ux = (jx + R(0.5) * Fx) * ir, uy = (jy + R(0.5) * Fy) * ir, uz = (jz + R(0.5) * Fz) * ir;
    const R u2 = ux * ux + uy * uy + uz * uz;
    // g_eq = f_eq - w = w (drho - 1.5 rho u^2 + c.u (3 rho + 4.5 rho c.u))
    const R om = R(a.om), c1 = R(1) - R(0.5) * om;
    const R base = drho - rho * R(1.5) * u2, r3 = R(3) * rho, r45 = R(4.5) * rho;
    const R uF3 = FORCE ? R(3) * (ux * Fx + uy * Fy + uz * Fz) : R(0);
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        const R cu = R(q27x(i)) * ux + R(q27y(i)) * uy + R(q27z(i)) * uz;
        const R geq = R(q27w(i)) * (base + cu * (r3 + r45 * cu));
        R v = g[i] + om * (geq - g[i]);
        if (FORCE) {
            const R cF = R(q27x(i)) * Fx + R(q27y(i)) * Fy + R(q27z(i)) * Fz;
            v += (c1 * R(q27w(i))) * (R(3) * cF - uF3 + R(9) * cu * cF);
        }
        Store<S>::st(B + (i * N + (size_t)c), v);
    }
    watchdog(rho, ux, uy, uz, a.status);
}

__host__ __device__ constexpr int q27opp(int i) {
    // the opposite velocity has every component negated: search the table
    int o = 0;
    for (int j = 0; j < Q27; j++)
        if (q27x(j) == -q27x(i) && q27y(j) == -q27y(i) && q27z(j) == -q27z(i)) o = j;
    return o;
}
static_assert(q27opp(0) == 0 && q27opp(1) == 6 && q27opp(26) == 19, "opposites");

// The pipe wall of the paper's runs (Sec. 2.1) on D3Q27: cells with
// (x - c_x)^2 + (y - c_y)^2 >= R^2 are solid. A link (x_f, i) joins a fluid
// cell to a solid x_f + c_i; the wall sits at x_f + q c_i, q in (0, 1] the
// exit root of the cylinder equation along c_i (FP64). The population
// j = opp(i) that cannot be pulled from x_f + c_i is the linear
// interpolated bounce-back (Bouzidi et al. 2001) from post-collision values
// at the wall at rest:
//   q < 1/2: 2q f*_i(x_f) + (1 - 2q) f*_i(x_f - c_i), x_f - c_i fluid, else f*_i(x_f);
//   q >= 1/2: f*_i(x_f) / (2q) + (2q - 1)/(2q) f*_j(x_f).
// The geometry is the same in every z plane: per (x, y) column a 27-bit
// mask (bit i: the column x + c_i, y + c_i is solid; bit 0: the column
// itself) tells which pulls come from the wall. Solid cells are not swept.
// The weights of the two populations of each wall link are formed once, at
// set-up (q27_coef_kernel), per column and direction: (2q, 1 - 2q) with
// f*_i(x_f - c_i), (1, 0) for the halfway fallback, and
// (1/(2q), (2q - 1)/(2q)) with f*_j(x_f), the last two flagged in hmask.
struct Q27PipeArgs {
    Q27Args b;
    const unsigned *colmask, *hmask;
    const void *coef;  // per column x 27 directions: two weights in the arithmetic type
    const int2 *cols;  // fluid columns: x + nx y, nonzero if the column has wall links
    ColumnItems items;
    int zp;
    long long Np;
    // the pull of direction i for element e of a plane is Ap[i][e] (plus nz
    // or minus nz across the z ends), its store Bp[i][e]
    const void *Ap[Q27];  // A + i Np - (c_z + zp (c_x + nx c_y))
    void *Bp[Q27];        // B + i Np
};

template <typename R>
struct Q27Coef {
    R k1, k2;
};

template <int S>
__global__ void q27_coef_kernel(const unsigned *colmask, unsigned *hmask, void *coefv, int nx, int ny, double pcx,
                                double pcy, double R2) {
    typedef typename Store<S>::R R;
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    if (col >= nx * ny) return;
    const unsigned m = colmask[col];
    Q27Coef<R> *coef = (Q27Coef<R> *)coefv + (size_t)col * Q27;
    unsigned h = 0;
    if (!(m & 1u) && m) {
        const int x = col % nx, y = col / nx;
        const double dx = (double)x - pcx, dy = (double)y - pcy;
        const double c0 = dx * dx + dy * dy - R2;
        for (int i = 1; i < Q27; i++) {
            if (!((m >> i) & 1u)) continue;
            const double aa = (double)(q27x(i) * q27x(i) + q27y(i) * q27y(i));
            const double b = q27x(i) * dx + q27y(i) * dy;
            const double q = (-b + sqrt(b * b - aa * c0)) / aa;
            Q27Coef<R> k;
            if (q < 0.5) {
                if ((m >> q27opp(i)) & 1u) {  // x_f - c_i solid too: halfway
                    k.k1 = R(1);
                    k.k2 = R(0);
                    h |= 1u << i;
                } else {
                    k.k1 = R(2.0 * q);
                    k.k2 = R(1.0 - 2.0 * q);
                }
            } else {
                k.k1 = R(1.0 / (2.0 * q));
                k.k2 = R((2.0 * q - 1.0) / (2.0 * q));
                h |= 1u << i;
            }
            coef[i] = k;
        }
    }
    hmask[col] = h;
}

// On the column layout (columns.cuh): a warp takes 32 consecutive z of a
// fluid column, whose mask and weights are uniform over it. What
// bounds it: HBM. 0.259 ms per step on the benchmark pipe (148 x 148 x 438,
// R = 73, FP32): 6.12 TB/s of its 216 B per fluid cell; the sweep over
// x-fast cells, whose warps mixed fluid, wall and solid cells, took 0.386.
// Registers for 4 resident blocks of 256 per SM (64, no spills); 3, 5 and 6
// blocks took 0.283, 0.267 (32 bytes spilled) and 0.315 ms.
constexpr int q27_min_blocks(int S) { return S == LBM_F32 ? 4 : 2; }

// WRAP: fluid columns touch an x or y face of the box
template <int S, bool FORCE, bool WRAP, bool FLAT>
__global__ void __launch_bounds__(256, q27_min_blocks(S)) q27_columns_kernel(Q27PipeArgs pa) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    const Q27Args &a = pa.b;
    unsigned ci;
    int z;
    if (!pa.items.cell<FLAT>(ci, z)) return;
    const int2 col = __ldg(pa.cols + ci);
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    if (z >= nz) return;
    const int c = col.x * pa.zp + z;
    const int zlo = z == 0 ? nz : 0, zhi = z == nz - 1 ? nz : 0;
    const T *__restrict__ A = (const T *)a.A;
    const size_t N = (size_t)pa.Np;
    R g[Q27];
    if constexpr (WRAP) {
        const int y = (int)a.fx.div((unsigned)col.x), x = col.x - y * nx;
        const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
        const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
#pragma unroll
        for (int i = 0; i < Q27; i++) {
            const int xs = q27x(i) > 0 ? xm : (q27x(i) < 0 ? xp : x);
            const int ys = q27y(i) > 0 ? ym : (q27y(i) < 0 ? yp : y);
            const int zs = z - q27z(i) + (q27z(i) > 0 ? zlo : 0) - (q27z(i) < 0 ? zhi : 0);
            g[i] = Store<S>::ld(A + i * N + (xs + nx * ys) * pa.zp + zs);
        }
    } else {
#pragma unroll
        for (int i = 0; i < Q27; i++)
            g[i] = Store<S>::ld((const T *)pa.Ap[i] + (c + (q27z(i) > 0 ? zlo : 0) - (q27z(i) < 0 ? zhi : 0)));
    }
    const unsigned rem = (unsigned)col.x;
    if (col.y) {  // wall column (uniform over a warp of one column): the populations coming back from the wall
        const unsigned m = __ldg(pa.colmask + rem);
        const unsigned h = __ldg(pa.hmask + rem);
        const Q27Coef<R> *kc = (const Q27Coef<R> *)pa.coef + (size_t)rem * Q27;
#pragma unroll
        for (int i = 1; i < Q27; i++) {
            if (!((m >> i) & 1u)) continue;
            const int j = q27opp(i);
            const Q27Coef<R> k = kc[i];
            const R fi = Store<S>::ld(A + (i * N + (size_t)c));  // f*_i(x_f)
            // q < 1/2: f*_i(x_f - c_i), the regular pull of direction i;
            // q >= 1/2 and the halfway fallback (weight 0; its pull is a solid
            // cell's, which may hold anything): f*_j(x_f)
            const R second = ((h >> i) & 1u) ? Store<S>::ld(A + (j * N + (size_t)c)) : g[i];
            // the bounce-back acts on f, the storage holds g = f - w with w_i = w_j
            g[j] = k.k1 * fi + k.k2 * second;
        }
    }
    R drho = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        drho += g[i];
        if (q27x(i)) jx += q27x(i) > 0 ? g[i] : -g[i];
        if (q27y(i)) jy += q27y(i) > 0 ? g[i] : -g[i];
        if (q27z(i)) jz += q27z(i) > 0 ? g[i] : -g[i];
    }
    const R Fx = FORCE ? R(a.F[0]) : R(0), Fy = FORCE ? R(a.F[1]) : R(0), Fz = FORCE ? R(a.F[2]) : R(0);
    const R rho = R(1) + drho, ir = R(1) / rho;
    const R ux = (jx + R(0.5) * Fx) * ir, uy = (jy + R(0.5) * Fy) * ir, uz = (jz + R(0.5) * Fz) * ir;
    const R u2 = ux * ux + uy * uy + uz * uz;
    const R om = R(a.om), c1 = R(1) - R(0.5) * om;
    const R base = drho - rho * R(1.5) * u2, r3 = R(3) * rho, r45 = R(4.5) * rho;
    const R uF3 = FORCE ? R(3) * (ux * Fx + uy * Fy + uz * Fz) : R(0);
#pragma unroll
    for (int i = 0; i < Q27; i++) {
        const R cu = R(q27x(i)) * ux + R(q27y(i)) * uy + R(q27z(i)) * uz;
        const R geq = R(q27w(i)) * (base + cu * (r3 + r45 * cu));
        R v = g[i] + om * (geq - g[i]);
        if (FORCE) {
            const R cF = R(q27x(i)) * Fx + R(q27y(i)) * Fy + R(q27z(i)) * Fz;
            v += (c1 * R(q27w(i))) * (R(3) * cF - uF3 + R(9) * cu * cF);
        }
        Store<S>::st((T *)pa.Bp[i] + c, v);
    }
    watchdog(rho, ux, uy, uz, a.status);
}

}  // namespace

template <int S>
static cudaError_t q27_step_s(Ctx &c, const Q27Args &a, bool force) {
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    if (force) q27_sweep_kernel<S, true><<<nb, 256, 0, c.stream>>>(a);
    else q27_sweep_kernel<S, false><<<nb, 256, 0, c.stream>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_q27_step(Ctx &c) {
    Q27Args a;
    a.A = c.fA;
    a.B = c.fB;
    a.N = c.N;
    a.nx = c.nx;
    a.ny = c.ny;
    a.nz = c.nz;
    a.fx = FastDiv((unsigned)c.nx);
    a.fxy = FastDiv((unsigned)(c.nx * c.ny));
    a.om = 1.0 / c.tau;
    for (int d = 0; d < 3; d++) a.F[d] = c.F[d];
    a.status = c.d_status;
    const bool force = c.F[0] != 0.0 || c.F[1] != 0.0 || c.F[2] != 0.0;
    count_launch(c, G_BULK);
    if (c.has_pipe) {
        Q27PipeArgs pa;
        pa.b = a;
        pa.colmask = c.q27_colmask;
        pa.hmask = c.q27_hmask;
        pa.coef = c.q27_coef;
        pa.cols = c.col_list;
        pa.items = column_items(c, c.ncols);
        pa.zp = c.zp;
        pa.Np = c.Np;
        const long long sb = (long long)storage_bytes(c.storage);
        for (int i = 0; i < Q27; i++) {
            const long long off = q27z(i) + (long long)c.zp * (q27x(i) + (long long)c.nx * q27y(i));
            pa.Ap[i] = (const void *)((const char *)c.fA + sb * (i * c.Np - off));
            pa.Bp[i] = (void *)((char *)c.fB + sb * (i * c.Np));
        }
        const unsigned nb = column_item_blocks(c, pa.items);
        if (nb == 0) return cudaSuccess;
#define QC(S, W, L)                                                                    \
    if (force) q27_columns_kernel<S, true, W, L><<<nb, 256, 0, c.stream>>>(pa);        \
    else q27_columns_kernel<S, false, W, L><<<nb, 256, 0, c.stream>>>(pa)
#define QS(S)                                                                          \
    if (c.col_flat) {                                                                  \
        if (c.pipe_nowrap) { QC(S, false, true); } else { QC(S, true, true); }         \
    } else {                                                                           \
        if (c.pipe_nowrap) { QC(S, false, false); } else { QC(S, true, false); }       \
    }
        if (c.storage == LBM_F64) { QS(LBM_F64) } else { QS(LBM_F32) }
#undef QS
#undef QC
        return cudaGetLastError();
    }
    return c.storage == LBM_F64 ? q27_step_s<LBM_F64>(c, a, force) : q27_step_s<LBM_F32>(c, a, force);
}

// per (x, y) column: bit i set when the column (x + c_x, y + c_y) of
// direction i is outside the pipe (bit 0: the column itself); FP64 test as
// the D3Q19 pipe flags
void q27_pipe_colmask(const Ctx &c, std::vector<unsigned> &mask) {
    mask.assign((size_t)c.nx * c.ny, 0u);
    auto solid = [&](int x, int y) {
        x = (x % c.nx + c.nx) % c.nx;
        y = (y % c.ny + c.ny) % c.ny;
        const double dx = (double)x - c.pipe_cx, dy = (double)y - c.pipe_cy;
        return dx * dx + dy * dy >= c.pipe_R * c.pipe_R;
    };
    for (int y = 0; y < c.ny; y++)
        for (int x = 0; x < c.nx; x++) {
            unsigned m = 0;
            for (int i = 0; i < Q27; i++)
                if (solid(x + q27x(i), y + q27y(i))) m |= 1u << i;
            mask[(size_t)x + (size_t)c.nx * y] = m;
        }
}

// the wall weights of the pipe (after the column masks are uploaded)
cudaError_t launch_q27_coef(Ctx &c) {
    const unsigned nb = (unsigned)((c.nx * c.ny + 255) / 256);
    const double R2 = c.pipe_R * c.pipe_R;
    if (c.storage == LBM_F64)
        q27_coef_kernel<LBM_F64><<<nb, 256, 0, c.stream>>>(c.q27_colmask, c.q27_hmask, c.q27_coef, c.nx, c.ny,
                                                            c.pipe_cx, c.pipe_cy, R2);
    else
        q27_coef_kernel<LBM_F32><<<nb, 256, 0, c.stream>>>(c.q27_colmask, c.q27_hmask, c.q27_coef, c.nx, c.ny,
                                                            c.pipe_cx, c.pipe_cy, R2);
    return cudaGetLastError();
}

cudaError_t launch_q27_init(Ctx &c, const double *u_dev, double rho0) {
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    if (c.storage == LBM_F64) q27_init_kernel<LBM_F64><<<nb, 256, 0, c.stream>>>(c.fA, u_dev, rho0, c.N);
    else q27_init_kernel<LBM_F32><<<nb, 256, 0, c.stream>>>(c.fA, u_dev, rho0, c.N);
    return cudaGetLastError();
}

// one population plane to or from the FP64 scratch c.rho_f (unshifted f)
cudaError_t q27_plane_copy(Ctx &c, int i, bool to_f64) {
    if (c.zlay) return column_plane_copy(c, i, q27w(i), to_f64);
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    if (c.storage == LBM_F64) q27_plane_kernel<LBM_F64><<<nb, 256, 0, c.stream>>>(c.fA, c.rho_f, c.N, i, to_f64);
    else q27_plane_kernel<LBM_F32><<<nb, 256, 0, c.stream>>>(c.fA, c.rho_f, c.N, i, to_f64);
    return cudaGetLastError();
}

cudaError_t launch_q27_macro(Ctx &c, float4 *rec) {
    count_launch(c, G_STATS);
    if (c.zlay) {
#define MK(S)                                                                                                      \
    q27_column_macro_kernel<S><<<column_tiles(c), 256, 0, c.stream>>>(c.fA, c.q27_colmask, rec, c.rho_f, c.u_f, c.nx, c.ny, c.nz, \
                                                                    c.zp, c.N, c.Np, c.F[0], c.F[1], c.F[2])
        if (c.storage == LBM_F64) MK(LBM_F64);
        else MK(LBM_F32);
#undef MK
        return cudaGetLastError();
    }
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    if (c.storage == LBM_F64)
        q27_macro_kernel<LBM_F64><<<nb, 256, 0, c.stream>>>(c.fA, rec, c.rho_f, c.u_f, c.N, c.F[0], c.F[1], c.F[2]);
    else
        q27_macro_kernel<LBM_F32><<<nb, 256, 0, c.stream>>>(c.fA, rec, c.rho_f, c.u_f, c.N, c.F[0], c.F[1], c.F[2]);
    return cudaGetLastError();
}

}  // namespace lbmgb
