// Component-wise TKE budget of the pipe (Eq. 1a-c, Sec. 2.2): production,
// turbulent transport, pressure work, viscous diffusion and dissipation of
// the streamwise, radial and azimuthal velocity fluctuations, per radial
// bin of one snapshot.
//
// Local quantities of a cell (statistics velocity, central differences):
//   G_ab = d u_a / d x_b, T_ij = e_i . G . e_j, s_ij = (T_ij + T_ji) / 2,
//   du_i/dr = T_ir, du_i/dz = T_iz, (1/r) du_z/dtheta = T_ztheta,
//   (1/r) du_r/dtheta = T_rtheta + u_theta / r,
//   (1/r) du_theta/dtheta = T_thetatheta - u_r / r,
//   p = c_s^2 rho.
//
// What bounds it: the FP64 pipe (two multiply-adds per clock and SM). So the
// work is arranged around the columns (x, y), whose radius, basis and bin
// are the same in every plane:
//   1. sums over z of u and rho per column (four additions per cell);
//   2. the bin means: every quantity averaged is linear in u and rho and the
//      basis is constant along z, so its column sum follows from the sums of
//      the column and its four neighbours (the z derivatives add up to zero
//      over the periodic length);
//   3. 14 products of fluctuations per cell, in registers over a run of z:
//      the bin means, turned back into the Cartesian frame of the column, are
//      taken off u and G before these are rotated, so that the rotation
//      gives the fluctuations directly (about 80 FP64 operations per cell);
//   4. the columns' sums go to one of BUD_REP copies of the bins (global FP64
//      reductions, one per column run, not per cell) and the copies are
//      added in order.
// The host then takes the radial derivatives of the binned profiles
// (central differences over the bin centres, one-sided at the ends).
// Benchmark pipe (7.34 M cells, 64 bins): 11.4 ms with 20 shared-memory FP64
// atomics and about 250 FP64 operations per cell and pass, 1.8 ms now, of
// which the product pass is 1.46 (1.0 by its FP64 operations alone).
#include "columns.cuh"

#include <vector>

namespace lbmgb {

namespace {

constexpr int BQ = 20;          // values per bin and copy
constexpr int BUD_REP = 32;     // copies of the bins

// per bin: count, means of the linear quantities (T rows: i, columns: j of e_i . G . e_j)
enum { M_ONE, M_UZ, M_UR, M_UT, M_P, M_T /* 9: rr rt rz tr tt tz zr zt zz */, M_URR = M_T + 9 /* u_r / r */, M_UTR /* u_t / r */, M_N };
static_assert(M_N <= BQ, "mean table");
// per bin: products of fluctuations; D*: s_ij dissipation sums of a component
enum { P_ZR, P_ZZR, P_P_DZZ, P_Z_SZR, P_DZ, P_RRR, P_R_P, P_P_DRR, P_R_SRR, P_DR, P_TTR, P_P_DTHT, P_T_SRT, P_DT, P_N };

struct BudgetArgs {
    const double *u, *rho;
    const uint8_t *flags;
    double *colsum;      // 4 x nx ny: sums over z of u_x, u_y, u_z, rho
    double *part;        // BUD_REP x nbins x BQ
    const double *mean;  // nbins x BQ
    int nx, ny, nz;
    long long N;
    double cx, cy, R;
    int nbins, run;
};

// the column's basis and bin; false outside the pipe, on the axis or beyond the last bin
__device__ __forceinline__ bool budget_column(const BudgetArgs &a, int x, int y, PipeColumn &k) {
    return pipe_column(a.flags, x, y, a.nx, a.ny, a.cx, a.cy, a.R, a.nbins, k) && k.r > 0.0;
}

__global__ void __launch_bounds__(256) budget_colsum_kernel(BudgetArgs a) {
    const long long nxy = (long long)a.nx * a.ny;
    const long long c = (long long)blockIdx.x * 32 + (threadIdx.x & 31);
    const int w = threadIdx.x >> 5;  // 8 warps share the planes of 32 columns
    double s[4] = {0, 0, 0, 0};
    if (c < nxy)
        for (int z = w; z < a.nz; z += 8) {
            const long long e = c + nxy * z;
            s[0] += a.u[e];
            s[1] += a.u[a.N + e];
            s[2] += a.u[2 * a.N + e];
            s[3] += a.rho[e];
        }
    __shared__ double sh[8][4][32];
    for (int q = 0; q < 4; q++) sh[w][q][threadIdx.x & 31] = s[q];
    __syncthreads();
    if (w >= 4 || c >= nxy) return;
    double t = 0.0;
    for (int v = 0; v < 8; v++) t += sh[v][w][threadIdx.x & 31];  // warp w adds quantity w
    a.colsum[w * nxy + c] = t;
}

__device__ __forceinline__ void bin_add(double *p, double v) { atomicAdd(p, v); }

__global__ void __launch_bounds__(256) budget_mean_kernel(BudgetArgs a) {
    int x, y;
    column_of_thread(a.nx, x, y);
    PipeColumn k;
    if (!budget_column(a, x, y, k)) return;
    const long long nxy = (long long)a.nx * a.ny;
    const int c = x + a.nx * y;
    const int xm = x == 0 ? c + a.nx - 1 : c - 1, xp = x == a.nx - 1 ? c - a.nx + 1 : c + 1;
    const int ym = y == 0 ? c + a.nx * (a.ny - 1) : c - a.nx, yp = y == a.ny - 1 ? c - a.nx * (a.ny - 1) : c + a.nx;
    double G[3][2];
    for (int d = 0; d < 3; d++) {
        const double *s = a.colsum + d * nxy;
        G[d][0] = 0.5 * (s[xp] - s[xm]);
        G[d][1] = 0.5 * (s[yp] - s[ym]);
    }
    const double ca = k.ca, sa = k.sa;
    const double ux = a.colsum[c], uy = a.colsum[nxy + c];
    const double rx = ca * G[0][0] + sa * G[0][1], ry = ca * G[1][0] + sa * G[1][1];     // (G e_r)
    const double tx = ca * G[0][1] - sa * G[0][0], ty = ca * G[1][1] - sa * G[1][0];     // (G e_theta)
    const double ur = ca * ux + sa * uy, ut = ca * uy - sa * ux;
    const double v[M_N] = {(double)a.nz,
                          a.colsum[2 * nxy + c],
                          ur,
                          ut,
                          a.colsum[3 * nxy + c] * (1.0 / 3.0),  // p = c_s^2 rho
                          ca * rx + sa * ry, ca * tx + sa * ty, 0.0,
                          ca * ry - sa * rx, ca * ty - sa * tx, 0.0,
                          ca * G[2][0] + sa * G[2][1], ca * G[2][1] - sa * G[2][0], 0.0, ur / k.r, ut / k.r};
    double *row = a.part + ((size_t)(blockIdx.x % BUD_REP) * a.nbins + k.bin) * BQ;
    for (int q = 0; q < M_N; q++)
        if (v[q] != 0.0) bin_add(row + q, v[q]);
}

__global__ void __launch_bounds__(256) budget_product_kernel(BudgetArgs a) {
    int x, y;
    column_of_thread(a.nx, x, y);
    PipeColumn k;
    if (!budget_column(a, x, y, k)) return;
    const double ca = k.ca, sa = k.sa, ir = 1.0 / k.r;
    const long long nxy = (long long)a.nx * a.ny, N = a.N;
    const int c = x + a.nx * y;
    const int oxm = x == 0 ? a.nx - 1 : -1, oxp = x == a.nx - 1 ? 1 - a.nx : 1;
    const int oym = y == 0 ? a.nx * (a.ny - 1) : -a.nx, oyp = y == a.ny - 1 ? -a.nx * (a.ny - 1) : a.nx;
    // the bin's means in the Cartesian frame of this column
    const double *m = a.mean + (size_t)k.bin * BQ, *T = m + M_T;
    const double mu[3] = {ca * m[M_UR] - sa * m[M_UT], sa * m[M_UR] + ca * m[M_UT], m[M_UZ]}, mp = m[M_P];
    // (1/r) times the mean is not the mean of the quotient: r varies in a bin
    const double kr = m[M_URR] - m[M_UR] * ir, kt = m[M_UT] * ir - m[M_UTR];
    double M[3][3];
    {
        const double xr = ca * T[0] - sa * T[3], xt = ca * T[1] - sa * T[4];  // rows x of Q T
        const double yr = sa * T[0] + ca * T[3], yt = sa * T[1] + ca * T[4];
        M[0][0] = ca * xr - sa * xt;
        M[0][1] = sa * xr + ca * xt;
        M[1][0] = ca * yr - sa * yt;
        M[1][1] = sa * yr + ca * yt;
        M[0][2] = ca * T[2] - sa * T[5];
        M[1][2] = sa * T[2] + ca * T[5];
        M[2][0] = ca * T[6] - sa * T[7];
        M[2][1] = sa * T[6] + ca * T[7];
        M[2][2] = T[8];
    }
    double P[P_N];
    for (int q = 0; q < P_N; q++) P[q] = 0.0;
    const int z0 = blockIdx.y * a.run, z1 = min(a.nz, z0 + a.run);
    const int zb = z0 == 0 ? a.nz - 1 : z0 - 1;
    const double *u = a.u + c;
    double um[3], uc[3];
    for (int d = 0; d < 3; d++) {
        um[d] = u[d * N + nxy * zb];
        uc[d] = u[d * N + nxy * z0];
    }
    for (int z = z0; z < z1; z++) {
        const long long e = nxy * z, ep = z == a.nz - 1 ? 0 : e + nxy;
        double up[3], G[3][3], v[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const double *ud = u + d * N;
            up[d] = ud[ep];
            G[d][0] = fma(0.5, ud[e + oxp] - ud[e + oxm], -M[d][0]);
            G[d][1] = fma(0.5, ud[e + oyp] - ud[e + oym], -M[d][1]);
            G[d][2] = fma(0.5, up[d] - um[d], -M[d][2]);
            v[d] = uc[d] - mu[d];
            um[d] = uc[d];
            uc[d] = up[d];
        }
        const double p = fma(a.rho[c + e], 1.0 / 3.0, -mp);
        const double ur = ca * v[0] + sa * v[1], ut = ca * v[1] - sa * v[0], uz = v[2];
        const double rx = ca * G[0][0] + sa * G[0][1], ry = ca * G[1][0] + sa * G[1][1];
        const double tx = ca * G[0][1] - sa * G[0][0], ty = ca * G[1][1] - sa * G[1][0];
        const double Trr = ca * rx + sa * ry, Ttr = ca * ry - sa * rx, Trt = ca * tx + sa * ty, Ttt = ca * ty - sa * tx;
        const double Trz = ca * G[0][2] + sa * G[1][2], Ttz = ca * G[1][2] - sa * G[0][2];
        const double Tzr = ca * G[2][0] + sa * G[2][1], Tzt = ca * G[2][1] - sa * G[2][0], Tzz = G[2][2];
        const double szr = 0.5 * (Tzr + Trz), szt = 0.5 * (Tzt + Ttz), srt = 0.5 * (Trt + Ttr);
        const double dthr = fma(ut, ir, Trt) + kt, dtht = fma(-ur, ir, Ttt) + kr;
        const double zr = uz * ur;
        P[P_ZR] += zr;
        P[P_ZZR] = fma(uz, zr, P[P_ZZR]);
        P[P_P_DZZ] = fma(p, Tzz, P[P_P_DZZ]);
        P[P_Z_SZR] = fma(uz, szr, P[P_Z_SZR]);
        P[P_DZ] = fma(szr, Tzr, fma(szt, Tzt, fma(Tzz, Tzz, P[P_DZ])));
        P[P_RRR] = fma(ur * ur, ur, P[P_RRR]);
        P[P_R_P] = fma(ur, p, P[P_R_P]);
        P[P_P_DRR] = fma(p, Trr, P[P_P_DRR]);
        P[P_R_SRR] = fma(ur, Trr, P[P_R_SRR]);
        P[P_DR] = fma(Trr, Trr, fma(srt, dthr, fma(szr, Trz, P[P_DR])));
        P[P_TTR] = fma(ut * ut, ur, P[P_TTR]);
        P[P_P_DTHT] = fma(p, dtht, P[P_P_DTHT]);
        P[P_T_SRT] = fma(ut, srt, P[P_T_SRT]);
        P[P_DT] = fma(Ttt, dtht, fma(srt, Ttr, fma(szt, Ttz, P[P_DT])));
    }
    const unsigned blk = blockIdx.x + gridDim.x * blockIdx.y;
    double *row = a.part + ((size_t)(blk % BUD_REP) * a.nbins + k.bin) * BQ;
    for (int q = 0; q < P_N; q++) bin_add(row + q, P[q]);
}

// the copies added in order; a bin's sums over its count. The mean pass
// keeps the count itself in column M_ONE.
__global__ void budget_bins_kernel(const double *part, double *out, const double *cnt, int nbins, int means) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nbins * BQ) return;
    const int b = i / BQ, q = i - b * BQ;
    double s = 0.0, n = 0.0;
    for (int r = 0; r < BUD_REP; r++) s += part[(size_t)r * nbins * BQ + i];
    if (means)
        for (int r = 0; r < BUD_REP; r++) n += part[((size_t)r * nbins + b) * BQ + M_ONE];
    else
        n = cnt[(size_t)b * BQ + M_ONE];
    out[i] = (means && q == M_ONE) ? s : (n > 0.0 ? s / n : 0.0);
}

}  // namespace

// what the call asks of the idle population buffer (a limit of the ABI: the
// layout below needs less for every grid that passes it: 4 nx ny sums and
// BUD_REP + 2 sets of bins, against 19 nx ny nz stored values of 2 bytes or
// more that are at least 305 sets of bins)
size_t tke_budget_scratch_bytes(int nbins) { return sizeof(double) * ((size_t)304 + 1) * nbins * BQ; }


// scratch: the population buffer that the next step overwrites (column
// sums, copies of the bins, bin means, bin products)
cudaError_t run_tke_budget(Ctx &c, int flags, int nbins, double *out) {
    cudaError_t e;
    if ((e = launch_macro(c)) != cudaSuccess) return e;
    const int ibm = c.armed_bc == LBM_BC_IBM_U || c.armed_bc == LBM_BC_IBM_B;
    if (!(ibm && (flags & LBM_STATS_UNMASK)))
        if ((e = launch_mask(c)) != cudaSuccess) return e;
    const size_t nxy = (size_t)c.nx * c.ny, set = (size_t)nbins * BQ;
    BudgetArgs a{c.u_f, c.rho_f, c.flags, (double *)c.fB, (double *)c.fB + 4 * nxy, nullptr, c.nx, c.ny, c.nz, c.N,
                 c.pipe_cx, c.pipe_cy, c.pipe_R, nbins, column_run(c.nz)};
    double *dmean = a.part + BUD_REP * set, *dprod = dmean + set;
    a.mean = dmean;
    const dim3 cols = column_blocks(c.nx, c.ny, c.nz, a.run);
    const unsigned nbb = (unsigned)((set + 255) / 256);
    count_launch(c, G_STATS, 5);
    budget_colsum_kernel<<<(unsigned)((nxy + 31) / 32), 256, 0, c.stream>>>(a);
    if ((e = cudaMemsetAsync(a.part, 0, sizeof(double) * BUD_REP * set, c.stream)) != cudaSuccess) return e;
    budget_mean_kernel<<<cols.x, 256, 0, c.stream>>>(a);
    budget_bins_kernel<<<nbb, 256, 0, c.stream>>>(a.part, dmean, nullptr, nbins, 1);
    if ((e = cudaMemsetAsync(a.part, 0, sizeof(double) * BUD_REP * set, c.stream)) != cudaSuccess) return e;
    budget_product_kernel<<<cols, 256, 0, c.stream>>>(a);
    budget_bins_kernel<<<nbb, 256, 0, c.stream>>>(a.part, dprod, dmean, nbins, 0);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    std::vector<double> both(2 * set), cnt(nbins);
    if ((e = cudaMemcpyAsync(both.data(), dmean, sizeof(double) * both.size(), cudaMemcpyDeviceToHost, c.stream)) !=
        cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(c.stream)) != cudaSuccess) return e;
    const double *mean = both.data(), *prod = mean + set;
    for (int b = 0; b < nbins; b++) cnt[b] = mean[(size_t)b * BQ + M_ONE];

    // radial derivative over the bin centres r_b = (b + 1/2) R / nbins:
    // central differences, one-sided at the first and last bins
    const int n = nbins;
    const double R = c.pipe_R, h = R / n, nu = (c.tau - 0.5) / 3.0;
    std::vector<double> rb(n);
    for (int b = 0; b < n; b++) rb[b] = ((b + 0.5) * R) / n;
    auto ddr = [&](const std::vector<double> &F) {
        std::vector<double> g(n, 0.0);
        if (n > 1) {
            g[0] = (F[1] - F[0]) / h;
            g[n - 1] = (F[n - 1] - F[n - 2]) / h;
            for (int b = 1; b < n - 1; b++) g[b] = (F[b + 1] - F[b - 1]) / (2.0 * h);
        }
        return g;
    };
    auto div_r = [&](const std::vector<double> &F) {  // (1/r) d/dr (r F)
        std::vector<double> rF(n);
        for (int b = 0; b < n; b++) rF[b] = rb[b] * F[b];
        std::vector<double> g = ddr(rF);
        for (int b = 0; b < n; b++) g[b] /= rb[b];
        return g;
    };
    auto pm = [&](int k, double f) {  // f times a pass-2 column
        std::vector<double> v(n);
        for (int b = 0; b < n; b++) v[b] = f * prod[(size_t)b * BQ + k];
        return v;
    };
    auto P = [&](int b, int k) { return prod[(size_t)b * BQ + k]; };
    std::vector<double> uz_mean(n);
    for (int b = 0; b < n; b++) uz_mean[b] = mean[(size_t)b * BQ + M_UZ];
    const std::vector<double> dUz = ddr(uz_mean), Tz = div_r(pm(P_ZZR, 0.5)), Vz = div_r(pm(P_Z_SZR, 1.0)),
                              Tr = div_r(pm(P_RRR, 0.5)), dRP = ddr(pm(P_R_P, 1.0)), Vr = div_r(pm(P_R_SRR, 1.0)),
                              Tt = div_r(pm(P_TTR, 0.5)), Vt = div_r(pm(P_T_SRT, 1.0));
    for (int b = 0; b < n; b++) {
        double *o = out + (size_t)b * LBM_BUDGET_NT;
        o[0] = cnt[b];
        if (!(cnt[b] > 0.0)) {
            for (int k = 1; k < LBM_BUDGET_NT; k++) o[k] = 0.0;
            continue;
        }
        o[1] = -P(b, P_ZR) * dUz[b];
        o[2] = -Tz[b];
        o[3] = P(b, P_P_DZZ);
        o[4] = 2.0 * nu * Vz[b];
        o[5] = -2.0 * nu * P(b, P_DZ);
        o[6] = -Tr[b];
        o[7] = -dRP[b] + P(b, P_P_DRR);
        o[8] = 2.0 * nu * Vr[b];
        o[9] = -2.0 * nu * P(b, P_DR);
        o[10] = -Tt[b];
        o[11] = P(b, P_P_DTHT);
        o[12] = 2.0 * nu * Vt[b];
        o[13] = -2.0 * nu * P(b, P_DT);
    }
    return cudaSuccess;
}

}  // namespace lbmgb
