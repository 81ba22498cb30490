// The immersed boundary pipe (Sec. 2.1) on the column layout (columns.cuh).
//
// The ring of markers is the same in every z plane and sits at integer z,
// so the support cells are whole columns, the x-y weight of a (marker,
// support column) pair is the same in all planes, and the z factor of the
// 4-point kernel takes the constants phi(0) = 1/2, phi(+-1) = 1/4
// (phi(+-2) = 0). A step:
//   sweep    pull and collide of all other columns; at support columns rho
//            and u* = (sum f c + F_ext/2)/rho of the pulled populations
//            (first half of the direct forcing)
//   3 x      U*_l, rho_l at the markers and F_l = 2 rho_l (U_d - U*_l), U_d = 0;
//            then F(x) = sum F_l delta dV_l and u* += F/(2 rho) at the columns
//   collide  pull again and collide the support columns with body + IBM force
// Every access is a run of consecutive z of one column, marker or site:
//   sites (k, z):   (rho, u*) at 4 (k nz + z), force planes F_d at d S + k nz + z (S = sp nz sites)
//   markers (j, z): force planes at d M + j nz + z (M = nc nz markers)
//
// What bounds it: HBM for the sweep and the collision (support columns read
// their populations twice and write them once; left in the stream of the
// sweep and collided in place they were read twice and written twice), L2
// and launch latency for the passes. Benchmark pipe (148 x 148 x 438,
// R = 73, IBM-B, FP32), per step: sweep 0.215 ms (6.4 TB/s), passes 0.071,
// collision 0.030, together 0.311 ms. With x fastest (rows through the ring,
// tiles of 6 planes, scattered support cells): 0.246 + 0.164 + 0.093 = 0.498.
#include "columns.cuh"

namespace lbmgb {

struct IbmColumnArgs {
    ColumnPtrs p;
    const int *info;   // per column: (support index + 1) << 1 | solid
    const int *sites;  // support columns in order (the first sp cells of the site list)
    void *ru;          // (rho, u*) per site
    const void *sF;    // IBM force planes
    long long S;       // sites
    ColumnItems items;  // of all columns, or of the support columns
    unsigned *status;
    Rates rt;
    double F[3];
    float Fs[3];
};

__device__ __forceinline__ void st_site4(float *p, float a, float b, float c, float d) {
    *(float4 *)p = make_float4(a, b, c, d);
}
__device__ __forceinline__ void st_site4(double *p, double a, double b, double c, double d) {
    ((double2 *)p)[0] = make_double2(a, b);
    ((double2 *)p)[1] = make_double2(c, d);
}
__device__ __forceinline__ void ld_site4(const float *p, float q[4]) {
    const float4 v = *(const float4 *)p;
    q[0] = v.x;
    q[1] = v.y;
    q[2] = v.z;
    q[3] = v.w;
}
__device__ __forceinline__ void ld_site4(const double *p, double q[4]) {
    const double2 v0 = ((const double2 *)p)[0], v1 = ((const double2 *)p)[1];
    q[0] = v0.x;
    q[1] = v0.y;
    q[2] = v1.x;
    q[3] = v1.y;
}

// resident blocks of 256 per SM: FP32 on the benchmark pipe, whole step:
// 0.3158 ms at 3, 0.3156 at 4, 0.3113 at 5, 0.3184 at 6
constexpr int ibm_column_min_blocks(int S) { return S == LBM_F64 ? 2 : 5; }

template <int S, bool FORCE, bool SRT, bool FLAT>
__global__ void __launch_bounds__(256, ibm_column_min_blocks(S)) ibm_columns_sweep(IbmColumnArgs a) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    unsigned col;
    int z;
    if (!a.items.cell<FLAT>(col, z)) return;
    const int info = __ldg(a.info + col);
    if (z >= a.p.nz) return;
    R g[19];
    column_pull<T, true, FLAT>(g, a.p, (int)col, z, [](const T *p) -> R { return Store<S>::ld(p); });
    const bool fluid = !(info & 1);
    if (info >> 1) {  // support column (uniform over a warp of one column)
        R drho = g[0];
#pragma unroll
        for (int i = 1; i < 19; i++) drho += g[i];
        R jx = (g[1] - g[2]) + (g[7] - g[8]) + (g[9] - g[10]) + (g[11] - g[12]) + (g[13] - g[14]);
        R jy = (g[3] - g[4]) + (g[7] - g[8]) - (g[9] - g[10]) + (g[15] - g[16]) + (g[17] - g[18]);
        R jz = (g[5] - g[6]) + (g[11] - g[12]) - (g[13] - g[14]) + (g[15] - g[16]) - (g[17] - g[18]);
        if (FORCE && fluid) {
            jx += R(0.5) * body_force<R>(a, 0);
            jy += R(0.5) * body_force<R>(a, 1);
            jz += R(0.5) * body_force<R>(a, 2);
        }
        const R rho = R(1) + drho, ir = R(1) / rho;
        st_site4((R *)a.ru + 4 * ((size_t)((info >> 1) - 1) * a.p.nz + z), rho, jx * ir, jy * ir, jz * ir);
        return;
    }
    R rho, ux, uy, uz;
    const R fs = fluid ? R(1) : R(0);  // the body force acts on fluid cells only
    collide<R, FORCE, SRT>(g, fs * body_force<R>(a, 0), fs * body_force<R>(a, 1), fs * body_force<R>(a, 2), a.rt, rho, ux,
                           uy, uz);
    watchdog(rho, ux, uy, uz, a.status);
    const int e = column_element<FLAT>(a.p, (int)col, z);
#pragma unroll
    for (int i = 0; i < 19; i++) Store<S>::st((T *)a.p.Bp[i] + e, g[i]);
}

template <int S, bool SRT, bool FLAT>
__global__ void __launch_bounds__(256, ibm_column_min_blocks(S)) ibm_columns_collide(IbmColumnArgs a) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    unsigned k;
    int z;
    if (!a.items.cell<FLAT>(k, z)) return;
    const int col = __ldg(a.sites + k);
    if (z >= a.p.nz) return;
    R g[19];
    column_pull<T, true, FLAT>(g, a.p, col, z, [](const T *p) -> R { return Store<S>::ld(p); });
    const R fs = (__ldg(a.info + col) & 1) ? R(0) : R(1);
    const R *sF = (const R *)a.sF + (size_t)k * a.p.nz + z;
    const R Fx = fs * body_force<R>(a, 0) + sF[0];
    const R Fy = fs * body_force<R>(a, 1) + sF[a.S];
    const R Fz = fs * body_force<R>(a, 2) + sF[2 * a.S];
    R rho, ux, uy, uz;
    collide<R, true, SRT>(g, Fx, Fy, Fz, a.rt, rho, ux, uy, uz);
    watchdog(rho, ux, uy, uz, a.status);
    const int e = column_element<FLAT>(a.p, col, z);
#pragma unroll
    for (int i = 0; i < 19; i++) Store<S>::st((T *)a.p.Bp[i] + e, g[i]);
}

// The passes: a block takes one ring marker (or support column) and a run of
// blockDim.x - 2 planes; each thread forms the x-y sum of its plane once, the
// first and the last those of the halo planes, and the z factor combines
// three neighbours through shared memory.
struct IbmPassArgs {
    int nz, pass, nc, sp;  // a launch: nc markers or sp columns for each run of planes in turn
    // markers: 16 (support column, x-y weight) entries each
    const int *it_k;
    const void *it_w;
    void *mF, *mAcc;  // F_l dV_l of the pass, F_l summed over the passes
    long long M;
    double dV;
    // support columns: range of the marker list
    const int *sites, *xy_start, *xy_j;
    const void *xy_w;
    void *ru, *sF;
    long long S;
};

// plane of thread t of a block: z0 - 1 + t, wrapped
__device__ __forceinline__ int pass_plane(int z0, int nz) {
    const int z = (z0 - 1 + (int)threadIdx.x) % nz;
    return z < 0 ? z + nz : z;
}

template <typename R>
__global__ void __launch_bounds__(256) ibm_columns_interp(IbmPassArgs a) {
    __shared__ R P[4][256];
    const int j = (int)(blockIdx.x % (unsigned)a.nc), t = threadIdx.x;
    const int z0 = (int)(blockIdx.x / (unsigned)a.nc) * (int)(blockDim.x - 2), z = pass_plane(z0, a.nz);
    const R *tw = (const R *)a.it_w + 16 * (size_t)j;
    const int *tk = a.it_k + 16 * (size_t)j;
    const R *ru = (const R *)a.ru + 4 * (size_t)z;
    R q[4] = {R(0), R(0), R(0), R(0)};
    R v[16][4];
    // all 16 loads in flight (an entry without a column has weight 0 and index 0)
#pragma unroll
    for (int e = 0; e < 16; e++) ld_site4(ru + 4 * (size_t)__ldg(tk + e) * a.nz, v[e]);
#pragma unroll
    for (int e = 0; e < 16; e++) {
        const R w = __ldg(tw + e);
        if (w != R(0))
            for (int d = 0; d < 4; d++) q[d] += w * v[e][d];
    }
    for (int d = 0; d < 4; d++) P[d][t] = q[d];
    __syncthreads();
    if (t < 1 || t > (int)blockDim.x - 2 || z0 - 1 + t >= a.nz) return;
    for (int d = 0; d < 4; d++) q[d] = R(0.25) * P[d][t - 1] + R(0.5) * P[d][t] + R(0.25) * P[d][t + 1];
    R *mF = (R *)a.mF + (size_t)j * a.nz + z, *acc = (R *)a.mAcc + (size_t)j * a.nz + z;
    const R dVl = R(a.dV);
    for (int d = 0; d < 3; d++) {
        const R Fl = R(2) * q[0] * (R(0) - q[1 + d]);
        mF[d * a.M] = Fl * dVl;  // spread weight F_l dV_l
        acc[d * a.M] = a.pass == 0 ? Fl : acc[d * a.M] + Fl;
    }
}

template <typename R>
__global__ void __launch_bounds__(256) ibm_columns_spread(IbmPassArgs a) {
    __shared__ R Q[3][256];
    const int k = (int)(blockIdx.x % (unsigned)a.sp), t = threadIdx.x;
    const int z0 = (int)(blockIdx.x / (unsigned)a.sp) * (int)(blockDim.x - 2), z = pass_plane(z0, a.nz);
    const int xy = __ldg(a.sites + k);
    const int e0 = __ldg(a.xy_start + xy), e1 = __ldg(a.xy_start + xy + 1);
    const R *xw = (const R *)a.xy_w, *mF = (const R *)a.mF + z;
    R q[3] = {R(0), R(0), R(0)};
    for (int e = e0; e < e1; e++) {
        const R w = __ldg(xw + e);
        const R *f = mF + (size_t)__ldg(a.xy_j + e) * a.nz;
        for (int d = 0; d < 3; d++) q[d] += f[d * a.M] * w;
    }
    for (int d = 0; d < 3; d++) Q[d][t] = q[d];
    __syncthreads();
    if (t < 1 || t > (int)blockDim.x - 2 || z0 - 1 + t >= a.nz) return;
    const size_t s = (size_t)k * a.nz + z;
    R *ru = (R *)a.ru + 4 * s, *sF = (R *)a.sF + s;
    R r[4];
    ld_site4(ru, r);
    const R ir = R(0.5) / r[0];
    for (int d = 0; d < 3; d++) {
        const R F = R(0.25) * Q[d][t + 1] + R(0.5) * Q[d][t] + R(0.25) * Q[d][t - 1];
        r[1 + d] += F * ir;
        sF[d * a.S] = a.pass == 0 ? F : sF[d * a.S] + F;
    }
    st_site4(ru, r[0], r[1], r[2], r[3]);
}

// ------------------------------------------------------------- launchers ---
static void fill_args(const Ctx &c, IbmColumnArgs &a, long long n) {
    column_ptrs(c, a.p);
    a.info = c.col_ibm;
    a.sites = c.site_cell;
    a.ru = c.sup_ru;
    a.sF = c.sup_F;
    a.S = (long long)c.pipe_sp * c.nz;
    a.items = column_items(c, n);
    a.status = c.d_status;
    a.rt = c.rt;
    for (int d = 0; d < 3; d++) {
        a.F[d] = c.F[d];
        a.Fs[d] = (float)c.F[d];
    }
}

template <int S, bool FLAT>
static cudaError_t sweep_t(Ctx &c) {
    IbmColumnArgs a;
    fill_args(c, a, (long long)c.nx * c.ny);
    const unsigned nb = column_item_blocks(c, a.items);
    const bool force = c.F[0] != 0.0 || c.F[1] != 0.0 || c.F[2] != 0.0, srt = c.rates == LBM_RATES_SRT;
    count_launch(c, G_BULK);
    if (srt && force) ibm_columns_sweep<S, true, true, FLAT><<<nb, 256, 0, c.stream>>>(a);
    else if (srt) ibm_columns_sweep<S, false, true, FLAT><<<nb, 256, 0, c.stream>>>(a);
    else if (force) ibm_columns_sweep<S, true, false, FLAT><<<nb, 256, 0, c.stream>>>(a);
    else ibm_columns_sweep<S, false, false, FLAT><<<nb, 256, 0, c.stream>>>(a);
    return cudaGetLastError();
}

template <int S, bool FLAT>
static cudaError_t collide_t(Ctx &c) {
    IbmColumnArgs a;
    fill_args(c, a, c.pipe_sp);
    const unsigned nb = column_item_blocks(c, a.items);
    count_launch(c, G_IBMCOL);
    if (c.rates == LBM_RATES_SRT) ibm_columns_collide<S, true, FLAT><<<nb, 256, 0, c.stream>>>(a);
    else ibm_columns_collide<S, false, FLAT><<<nb, 256, 0, c.stream>>>(a);
    return cudaGetLastError();
}

template <typename R>
static cudaError_t passes_t(Ctx &c) {
    IbmPassArgs a{c.nz, 0, c.pipe_nc, c.pipe_sp, c.pipe_it_k, c.pipe_it_w, c.mFr, c.mFaccR, (long long)c.pipe_nc * c.nz, c.pipe_dV,
                  c.site_cell, c.pipe_xy_start, c.pipe_xy_j, c.pipe_xy_w, c.sup_ru, c.sup_F, (long long)c.pipe_sp * c.nz};
    // equal runs of at most 254 planes, whole warps with the two halo threads
    const int tiles = (c.nz + 253) / 254, run = (c.nz + tiles - 1) / tiles;
    const unsigned tb = (unsigned)((run + 2 + 31) / 32 * 32);
    const unsigned ty = (unsigned)((c.nz + (int)tb - 3) / ((int)tb - 2));
    for (int pass = 0; pass < 3; pass++) {
        a.pass = pass;
        count_launch(c, G_IBM, 2);
        ibm_columns_interp<R><<<(unsigned)c.pipe_nc * ty, tb, 0, c.stream>>>(a);
        ibm_columns_spread<R><<<(unsigned)c.pipe_sp * ty, tb, 0, c.stream>>>(a);
    }
    c.markers_stale = 1;
    return cudaGetLastError();
}

cudaError_t launch_ibm_columns_sweep(Ctx &c) {
    switch (c.storage) {
    case LBM_F64: return c.col_flat ? sweep_t<LBM_F64, true>(c) : sweep_t<LBM_F64, false>(c);
    case LBM_F32: return c.col_flat ? sweep_t<LBM_F32, true>(c) : sweep_t<LBM_F32, false>(c);
    case LBM_F16S: return c.col_flat ? sweep_t<LBM_F16S, true>(c) : sweep_t<LBM_F16S, false>(c);
    default: return c.col_flat ? sweep_t<LBM_BF16S, true>(c) : sweep_t<LBM_BF16S, false>(c);
    }
}
cudaError_t launch_ibm_columns_collide(Ctx &c) {
    switch (c.storage) {
    case LBM_F64: return c.col_flat ? collide_t<LBM_F64, true>(c) : collide_t<LBM_F64, false>(c);
    case LBM_F32: return c.col_flat ? collide_t<LBM_F32, true>(c) : collide_t<LBM_F32, false>(c);
    case LBM_F16S: return c.col_flat ? collide_t<LBM_F16S, true>(c) : collide_t<LBM_F16S, false>(c);
    default: return c.col_flat ? collide_t<LBM_BF16S, true>(c) : collide_t<LBM_BF16S, false>(c);
    }
}
cudaError_t launch_ibm_columns_passes(Ctx &c) {
    return c.storage == LBM_F64 ? passes_t<double>(c) : passes_t<float>(c);
}

// ------------------------------- the layouts seen from outside the sweeps --
// F_l of the last step per marker l = z nc + j, three FP64 components
template <typename R>
__global__ void markers_out_kernel(double *out, const R *acc, int nc, int nz) {
    const long long M = (long long)nc * nz, l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= M) return;
    const long long z = l / nc, j = l - z * nc;
    for (int d = 0; d < 3; d++) out[3 * l + d] = (double)acc[d * M + j * nz + z];
}

cudaError_t refresh_markers(Ctx &c) {
    if (!c.markers_stale) return cudaSuccess;
    const unsigned nb = (unsigned)((c.nm + 255) / 256);
    if (c.storage == LBM_F64) markers_out_kernel<double><<<nb, 256, 0, c.stream>>>(c.mFacc, (const double *)c.mFaccR, c.pipe_nc, c.nz);
    else markers_out_kernel<float><<<nb, 256, 0, c.stream>>>(c.mFacc, (const float *)c.mFaccR, c.pipe_nc, c.nz);
    c.markers_stale = 0;
    return cudaGetLastError();
}

// the site forces in the order of the site list (s = z sp + k, three
// components each), from the planes or into them
template <typename R, bool OUT>
__global__ void site_force_kernel(R *list, R *planes, int sp, int nz) {
    const long long S = (long long)sp * nz, s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const long long z = s / sp, k = s - z * sp;
    for (int d = 0; d < 3; d++) {
        if (OUT) list[3 * s + d] = planes[d * S + k * nz + z];
        else planes[d * S + k * nz + z] = list[3 * s + d];
    }
}

cudaError_t copy_site_force(Ctx &c, void *list, bool out) {
    const unsigned nb = (unsigned)(((long long)c.pipe_sp * c.nz + 255) / 256);
    if (c.storage == LBM_F64) {
        if (out) site_force_kernel<double, true><<<nb, 256, 0, c.stream>>>((double *)list, (double *)c.sup_F, c.pipe_sp, c.nz);
        else site_force_kernel<double, false><<<nb, 256, 0, c.stream>>>((double *)list, (double *)c.sup_F, c.pipe_sp, c.nz);
    } else {
        if (out) site_force_kernel<float, true><<<nb, 256, 0, c.stream>>>((float *)list, (float *)c.sup_F, c.pipe_sp, c.nz);
        else site_force_kernel<float, false><<<nb, 256, 0, c.stream>>>((float *)list, (float *)c.sup_F, c.pipe_sp, c.nz);
    }
    return cudaGetLastError();
}

}  // namespace lbmgb
