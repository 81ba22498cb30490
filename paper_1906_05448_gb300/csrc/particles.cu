// Particle-side kernels. Particle state and equations are FP64; sums over
// links, markers and box cells form their terms in the storage's arithmetic
// type and add them up in FP64:
//  - gimem_reduce: per-particle sum of the per-link momentum exchange
//    (Galilean-invariant form of Wen et al. 2014, Sec. 3.1);
//  - release_kernel: initial particle velocity = fluid velocity averaged
//    over the particle volume (Sec. 3.1);
//  - contact_kernel / eom_kernel: normal-only soft-sphere contacts and the
//    rigid-body update (Sec. 3.1);
//  - IBM: marker placement, support-cell marking, the three direct-forcing
//    passes (interpolate with the Peskin 4-point delta, force, spread;
//    Sec. 2.1 / 3.1) and the particle force with Kempe's inner-fluid term.
// All reductions are block trees in a fixed order (bitwise reproducible for
// a given launch configuration); only the IBM spreading adds to the support
// cells with atomics (of the storage's arithmetic type).
#include "lbm_internal.cuh"

#include <algorithm>

namespace lbmgb {

// wrap a coordinate in [-n, 2n) into [0, n)
__device__ __forceinline__ int pwrap(int a, int n) {
    a = a < 0 ? a + n : a;
    return a >= n ? a - n : a;
}

constexpr int PB = 256;  // threads per particle block (as many as slot_sums has partial sums)

// Sums of NV quantities over SLOTS partial sums each, in FP64 and in a fixed
// order: sh[k * SLOTS + i] holds partial i of quantity k, warp k adds them up
// as a binary tree (halves first, the last five levels by shuffles). The
// particle kernels used to run that tree over the block with a barrier per
// level, which was most of their time.
constexpr int SLOTS = 256;
template <int NV, typename Rl>
__device__ __forceinline__ void slot_sums(const Rl *sh, double *tot /* shared, NV */) {
    const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k < NV) {
        double t[SLOTS / 32];
#pragma unroll
        for (int i = 0; i < SLOTS / 32; i++) {
            if constexpr (sizeof(Rl) == 8) t[i] = sh[k * SLOTS + 32 * i + lane];
            else t[i] = to_double(sh[k * SLOTS + 32 * i + lane]);
        }
#pragma unroll
        for (int o = SLOTS / 64; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < o; i++) t[i] += t[i + o];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
        if (lane == 0) tot[k] = t[0];
    }
}
// the same for one partial sum per thread of a block of SLOTS threads
template <int NV, typename Rl>
__device__ __forceinline__ void block_sum(const Rl v[NV], Rl *sh /* NV * SLOTS, shared */, double out[NV]) {
    static_assert(NV <= SLOTS / 32, "a warp per quantity");
    __shared__ double tot[NV];
    for (int k = 0; k < NV; k++) sh[k * SLOTS + threadIdx.x] = v[k];
    __syncthreads();
    slot_sums<NV>(sh, tot);
    __syncthreads();
    for (int k = 0; k < NV; k++) out[k] = tot[k];
}

// ------------------------------------------------------------ GIMEM ------
struct GimemArgs {
    const uint8_t *flags;
    const int *aux, *site_first, *link_pid;
    const unsigned *site_mask;
    const void *link_dP, *link_dT;  // arithmetic type of the storage
    const double *X, *R;
    double *Fh, *Th;
    int nx, ny, nz;
    long long max_sites;
};

// One block per particle. What bounds it is the chain of dependent loads
// flags -> site -> first link -> links: a thread per box cell that walked it
// cell by cell took 78 us for 2000 spheres of radius 4, and 40 us for the one
// of a 32^3 box. So each level is read for several cells at a time into
// shared memory, and the links by eight lanes per partial sum, one component
// each (consecutive addresses): 67 us, and 11 for the one sphere.
// Partial sum s of a component adds up, in the storage's arithmetic type,
// the links of the box cells s, s + 256, ... in that order, whatever the
// block's size.
constexpr int GIMEM_CELLS = 4096;  // box cells per round
template <typename Rl, int TB>
__global__ void __launch_bounds__(TB) gimem_reduce_kernel(GimemArgs a) {
    constexpr int CELLS = 8;  // cells of a thread whose loads are in flight together
    __shared__ int first[GIMEM_CELLS];
    __shared__ unsigned char links[GIMEM_CELLS];
    __shared__ unsigned some[SLOTS];  // bit j: cell s + 256 j of the round has links
    __shared__ Rl sum[6 * SLOTS];
    __shared__ int head[4];
    __shared__ float centre[4];
    __shared__ double tot[6];
    const int p = blockIdx.x, tid = threadIdx.x;
    if (tid < 3) {  // the box, once per block
        const double X = a.X[3 * p + tid], Rp = a.R[p];
        const int r = (int)ceil(Rp) + 2, b = (int)floor(X) - r;
        head[tid] = b;
        head[3] = 2 * r + 2;
        centre[tid] = (float)(X - b);
        centre[3] = (float)Rp + 1.5f;  // a link of p starts within R_p + sqrt 2 of its centre
    }
    for (int k = tid; k < 6 * SLOTS; k += TB) sum[k] = Rl(0);
    for (int k = tid; k < SLOTS; k += TB) some[k] = 0u;
    __syncthreads();
    const int bx = head[0], by = head[1], bz = head[2], w = head[3], total = w * w * w;
    const float fX0 = centre[0], fX1 = centre[1], fX2 = centre[2], reach2 = centre[3] * centre[3];
    const FastDiv fw((unsigned)w);
    // lanes 0 .. 2 of eight add up dP, 3 .. 5 dT
    const int comp = tid & 7;
    const Rl *e = comp < 3 ? (const Rl *)a.link_dP + comp : (const Rl *)a.link_dT + (comp - 3);
    for (int t0 = 0; t0 < total; t0 += GIMEM_CELLS) {
        for (int i0 = tid; i0 < GIMEM_CELLS && t0 + i0 - tid < total; i0 += CELLS * TB) {
            int c[CELLS];
            unsigned char fl[CELLS];
#pragma unroll
            for (int j = 0; j < CELLS; j++) {
                const int i = i0 + j * TB, t = t0 + i;
                int ix, iy, iz;
                box_coords(t, fw, w, ix, iy, iz);
                const float ex = ix - fX0, ey = iy - fX1, ez = iz - fX2;
                c[j] = i < GIMEM_CELLS && t < total && ex * ex + ey * ey + ez * ez <= reach2
                           ? pwrap(bx + ix, a.nx) + a.nx * (pwrap(by + iy, a.ny) + a.ny * pwrap(bz + iz, a.nz))
                           : -1;
                fl[j] = c[j] >= 0 ? a.flags[c[j]] : (unsigned char)0;
            }
#pragma unroll
            for (int j = 0; j < CELLS; j++) {
                c[j] = (fl[j] & FL_BND) ? a.aux[c[j]] : -1;
                if (c[j] >= a.max_sites) c[j] = -1;
            }
            int f[CELLS];
            unsigned m[CELLS];
#pragma unroll
            for (int j = 0; j < CELLS; j++) {
                f[j] = c[j] >= 0 ? a.site_first[c[j]] : 0;
                m[j] = c[j] >= 0 ? a.site_mask[c[j]] : 0u;
            }
#pragma unroll
            for (int j = 0; j < CELLS; j++) {
                const int i = i0 + j * TB;
                if (m[j] == 0u) continue;
                first[i] = f[j];
                links[i] = (unsigned char)__popc(m[j]);
                atomicOr(&some[i & (SLOTS - 1)], 1u << (i / SLOTS));
            }
        }
        __syncthreads();
        // the four groups of a warp in step (their cells and links differ in
        // number): loops they leave one by one would run once per group
        for (int s = tid >> 3; s < SLOTS; s += TB / 8) {
            unsigned cells = some[s];
            if (__all_sync(0xffffffffu, cells == 0u)) continue;
            Rl v = comp < 6 ? sum[comp * SLOTS + s] : Rl(0);
            do {
                const int i = s + SLOTS * (cells ? __ffs(cells) - 1 : 0);
                const int n = cells ? links[i] : 0;
                const int k0 = n ? first[i] : 0;
                cells &= cells - 1u;
                const int most = __reduce_max_sync(0xffffffffu, n);
#pragma unroll 4
                for (int k = 0; k < most; k++) {
                    const bool on = k < n && comp < 6;
                    const int own = on ? a.link_pid[k0 + k] : -1;
                    const Rl x = on ? e[3 * (size_t)(k0 + k)] : Rl(0);
                    v += own == p ? x : Rl(0);
                }
            } while (__any_sync(0xffffffffu, cells));
            if (comp < 6) sum[comp * SLOTS + s] = v;
        }
        __syncthreads();
        for (int k = tid; k < SLOTS; k += TB) some[k] = 0u;
        __syncthreads();
    }
    slot_sums<6>(sum, tot);
    __syncthreads();
    if (tid < 6) (tid < 3 ? a.Fh : a.Th)[3 * p + tid % 3] = tot[tid];
}

cudaError_t launch_gimem(Ctx &c) {
    if (c.np == 0) return cudaSuccess;
    GimemArgs a{c.flags, c.aux, c.site_first, c.link_pid, c.site_mask, c.link_dP, c.link_dT,
                c.X, c.R, c.Fh, c.Th, c.nx, c.ny, c.nz, c.max_sites};
    count_launch(c, G_PART);
    // 1024 threads while there is no more than a block per SM (a fixed sphere
    // of radius 4 in FP32: 14.9 us, with 256 threads 22, launch gap included),
    // 512 beyond (2000 spheres: 67 us, with 256 threads 75, with 128 96)
    const bool wide = c.np <= 152;
    if (c.storage == LBM_F64) {
        if (wide) gimem_reduce_kernel<double, 1024><<<c.np, 1024, 0, c.stream>>>(a);
        else gimem_reduce_kernel<double, 512><<<c.np, 512, 0, c.stream>>>(a);
    } else {
        if (wide) gimem_reduce_kernel<float, 1024><<<c.np, 1024, 0, c.stream>>>(a);
        else gimem_reduce_kernel<float, 512><<<c.np, 512, 0, c.stream>>>(a);
    }
    return cudaGetLastError();
}

// ----------------------------------------------------- solid fraction ----
// Kempe et al. (2012): alpha = sum(-phi H(-phi)) / sum|phi| over the 8 cell
// corners, phi = |x - X| - R (x relative to the particle, minimum image),
// in the arithmetic type R of the storage.
template <typename R>
__device__ R solid_fraction(R rx, R ry, R rz, R Rp) {
    R num = 0, den = 0;
    for (int m = 0; m < 8; m++) {
        const R ax = rx + ((m & 1) ? R(0.5) : R(-0.5)), ay = ry + ((m & 2) ? R(0.5) : R(-0.5)),
                az = rz + ((m & 4) ? R(0.5) : R(-0.5));
        const R phi = sqrt(ax * ax + ay * ay + az * az) - Rp;
        if (phi < R(0)) num += -phi;
        den += fabs(phi);
    }
    return den > R(0) ? num / den : R(0);
}

// velocity of the post-collision state of cell c: (sum f c - F/2) / rho
template <int S>
__device__ void cell_velocity(const void *A, size_t N, long long c, double Fx, double Fy, double Fz, double &rho,
                              double u[3]) {
    typedef typename Store<S>::T T;
    const T *P = (const T *)A;
    double r = 0.0, j0 = 0.0, j1 = 0.0, j2 = 0.0;
    for (int i = 0; i < 19; i++) {
        double g;
        if (S == LBM_F64) g = *(const double *)(P + i * N + c);
        else if (S == LBM_F32) g = *(const float *)(P + i * N + c);
        else if (S == LBM_F16S) g = (double)__half2float(*(const __half *)(P + i * N + c)) / (double)F16_SCALE;
        else g = (double)__bfloat162float(*(const __nv_bfloat16 *)(P + i * N + c));
        r += g;
        j0 += g * cx(i);
        j1 += g * cy(i);
        j2 += g * cz(i);
    }
    rho = 1.0 + r;
    u[0] = (j0 - 0.5 * Fx) / rho;
    u[1] = (j1 - 0.5 * Fy) / rho;
    u[2] = (j2 - 0.5 * Fz) / rho;
}

struct VolArgs {
    const void *A;
    const uint8_t *flags;
    const int *aux;
    const void *sup_ru;  // (rho, u*) per support site, arithmetic type of the storage
    const double *X, *R;
    double *out_u, *out_r;  // per particle (3): sum alpha u and sum alpha r x u (or averages)
    int nx, ny, nz;
    long long N;
    double F[3];
    int mode;  // 0: release average from populations, 1: Kempe integrals from populations, 2: from sup_u
    long long max_sites;
};

template <int S>
__global__ void __launch_bounds__(PB, S == LBM_F64 ? 2 : 4) volume_kernel(VolArgs a) {
    typedef typename Store<S>::R Rt;
    __shared__ Rt sh[7 * PB];
    const int p = blockIdx.x;
    const double *Xp = a.X + 3 * p;
    const double Rp = a.R[p];
    // the box once per block: FP64 in every thread costs more than the barrier
    __shared__ int head[4];
    __shared__ double frac[3];
    if (threadIdx.x < 3) {
        const double X = Xp[threadIdx.x], f = floor(X);
        const int r1 = (int)ceil(Rp) + 1;
        head[threadIdx.x] = (int)f - r1;
        head[3] = r1;
        frac[threadIdx.x] = X - f;
    }
    __syncthreads();
    const int r = head[3], bx = head[0], by = head[1], bz = head[2];
    const int w = 2 * r + 2;
    // cell offsets relative to the particle: integer part exact, fraction in Rt
    const double fx = frac[0], fy = frac[1], fz = frac[2];
    Rt v[7] = {0, 0, 0, 0, 0, 0, 0};
    const Rt *su = (const Rt *)a.sup_ru;
    const FastDiv fw((unsigned)w);
    const Rt ro = Rt(Rp) + Rt(0.9), ri = Rt(Rp) > Rt(0.9) ? Rt(Rp) - Rt(0.9) : Rt(0), ro2 = ro * ro, ri2 = ri * ri;
    for (int t = threadIdx.x; t < w * w * w; t += PB) {
        int ix, iy, iz;
        box_coords(t, fw, w, ix, iy, iz);
        const int x = pwrap(bx + ix, a.nx), y = pwrap(by + iy, a.ny), z = pwrap(bz + iz, a.nz);
        const Rt rx = Rt(ix - r) - Rt(fx), ry = Rt(iy - r) - Rt(fy), rz = Rt(iz - r) - Rt(fz);
        // a cell whose corners (0.87 from its centre) are all inside has
        // fraction 1, all outside 0: the eight distances are formed near the surface only
        const Rt d2 = rx * rx + ry * ry + rz * rz;
        if (d2 > ro2) continue;
        const Rt al = d2 < ri2 ? Rt(1) : solid_fraction<Rt>(rx, ry, rz, Rt(Rp));
        if (al <= Rt(0)) continue;
        const long long c = (long long)x + (long long)a.nx * (y + (long long)a.ny * z);
        Rt u[3];
        if (a.mode == 2) {
            const int s = a.aux[c];
            if (s < 0 || s >= a.max_sites) continue;
            u[0] = su[4 * s + 1];
            u[1] = su[4 * s + 2];
            u[2] = su[4 * s + 3];
        } else {
            double rho, ud[3];
            const bool fluid = a.mode == 0 ? true : !(a.flags[c] & FL_SOLID);
            cell_velocity<S>(a.A, (size_t)a.N, c, fluid ? a.F[0] : 0.0, fluid ? a.F[1] : 0.0, fluid ? a.F[2] : 0.0,
                             rho, ud);
            u[0] = Rt(ud[0]);
            u[1] = Rt(ud[1]);
            u[2] = Rt(ud[2]);
        }
        v[0] += al * u[0];
        v[1] += al * u[1];
        v[2] += al * u[2];
        v[3] += al * (ry * u[2] - rz * u[1]);
        v[4] += al * (rz * u[0] - rx * u[2]);
        v[5] += al * (rx * u[1] - ry * u[0]);
        v[6] += al;
    }
    double vd[7];
    block_sum<7>(v, sh, vd);
    if (threadIdx.x == 0) {
        if (a.mode == 0) {
            for (int d = 0; d < 3; d++) a.out_u[3 * p + d] = vd[6] > 0.0 ? vd[d] / vd[6] : 0.0;
        } else {
            for (int d = 0; d < 3; d++) {
                a.out_u[3 * p + d] = vd[d];
                a.out_r[3 * p + d] = vd[3 + d];
            }
        }
    }
}

static cudaError_t launch_volume(Ctx &c, int mode, double *out_u, double *out_r) {
    if (c.np == 0) return cudaSuccess;
    count_launch(c, G_PART);
    VolArgs a{c.fA, c.flags, c.aux, c.sup_ru, c.X, c.R, out_u, out_r, c.nx, c.ny, c.nz, c.N,
              {c.F[0], c.F[1], c.F[2]}, mode, c.max_sites};
    switch (c.storage) {
    case LBM_F64: volume_kernel<LBM_F64><<<c.np, PB, 0, c.stream>>>(a); break;
    case LBM_F32: volume_kernel<LBM_F32><<<c.np, PB, 0, c.stream>>>(a); break;
    case LBM_F16S: volume_kernel<LBM_F16S><<<c.np, PB, 0, c.stream>>>(a); break;
    default: volume_kernel<LBM_BF16S><<<c.np, PB, 0, c.stream>>>(a); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_release(Ctx &c) { return launch_volume(c, 0, c.U, nullptr); }

// ------------------------------------------------------- contacts, EOM ----
struct EomArgs {
    double *X, *Xold, *U, *W, *Fh, *Th, *Fprev, *Tprev, *Fc;
    const double *R, *mass, *inertia;
    int *has_prev;
    int np, nx, ny, nz;
    float4 *Xf;  // FP32 copies of the centres and radii for the contact search's cull
};

// FP32 centre and radius of every particle: the contact search culls pairs
// on these (one FP64-to-FP32 conversion per particle instead of per pair)
__global__ void xf_kernel(EomArgs a) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < a.np) a.Xf[p] = make_float4((float)a.X[3 * p], (float)a.X[3 * p + 1], (float)a.X[3 * p + 2], (float)a.R[p]);
}

// Normal-only soft-sphere contact (Sec. 3.1): for a gap below zeta = 1, a
// spring-dashpot along the line of centres, k_n = m (pi^2 + ln^2 e)/Tc^2,
// eta_n = -2 m ln e / Tc, m the reduced mass, e = 0.97, Tc = 10 steps.
// One warp per particle; lanes stride over partners, cull in FP32 with a
// margin and evaluate the few close pairs in FP64 (each pair as (a < b));
// the lane sums are reduced in a fixed butterfly order.
__global__ void __launch_bounds__(256) contact_kernel(EomArgs a) {
    const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (p >= a.np) return;
    const double zeta = 1.0, e = 0.97, Tc = 10.0, PI = 3.14159265358979323846;
    const float hx = 0.5f * a.nx, hy = 0.5f * a.ny, hz = 0.5f * a.nz;
    const float4 P = a.Xf[p];
    double F[3] = {0.0, 0.0, 0.0};
    // the culling data of four partners at a time: their loads overlap (one
    // by one the search took 25 us for 2000 particles, so 16)
    for (int q0 = lane; q0 < a.np; q0 += 128) {
        float4 Qs[4];
#pragma unroll
        for (int j = 0; j < 4; j++) Qs[j] = a.Xf[min(q0 + 32 * j, a.np - 1)];
        unsigned close = 0u;
#pragma unroll
        for (int j = 0; j < 4; j++) {
            const float4 Q = Qs[j];
            float dx = P.x - Q.x, dy = P.y - Q.y, dz = P.z - Q.z;
            dx = dx > hx ? dx - a.nx : (dx < -hx ? dx + a.nx : dx);
            dy = dy > hy ? dy - a.ny : (dy < -hy ? dy + a.ny : dy);
            dz = dz > hz ? dz - a.nz : (dz < -hz ? dz + a.nz : dz);
            const float reach = P.w + Q.w + (float)zeta + 0.01f;
            const int q = q0 + 32 * j;
            // not "less than": a NaN distance is evaluated
            if (!(dx * dx + dy * dy + dz * dz >= reach * reach) && q != p && q < a.np) close |= 1u << j;
        }
        for (; close; close &= close - 1u) {
            const int q = q0 + 32 * (__ffs(close) - 1);
            const int ia = q < p ? q : p, ib = q < p ? p : q;  // pair evaluated as (a < b)
            const double d0 = min_image(a.X[3 * ia] - a.X[3 * ib], a.nx),
                         d1 = min_image(a.X[3 * ia + 1] - a.X[3 * ib + 1], a.ny),
                         d2 = min_image(a.X[3 * ia + 2] - a.X[3 * ib + 2], a.nz);
            const double dist = sqrt(d0 * d0 + d1 * d1 + d2 * d2);
            const double gap = dist - (a.R[ia] + a.R[ib]);
            if (gap >= zeta || dist <= 0.0) continue;
            const double n0 = d0 / dist, n1 = d1 / dist, n2 = d2 / dist;
            const double vn = (a.U[3 * ia] - a.U[3 * ib]) * n0 + (a.U[3 * ia + 1] - a.U[3 * ib + 1]) * n1 +
                              (a.U[3 * ia + 2] - a.U[3 * ib + 2]) * n2;
            const double meff = a.mass[ia] * a.mass[ib] / (a.mass[ia] + a.mass[ib]);
            const double le = log(e);
            const double kn = meff * (PI * PI + le * le) / (Tc * Tc);
            const double eta = -2.0 * meff * le / Tc;
            const double Fm = kn * (zeta - gap) - eta * vn;
            const double sg = q < p ? -1.0 : 1.0;
            F[0] += sg * (Fm * n0);
            F[1] += sg * (Fm * n1);
            F[2] += sg * (Fm * n2);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        for (int d = 0; d < 3; d++) F[d] += __shfl_xor_sync(0xffffffffu, F[d], o);
    if (lane == 0)
        for (int d = 0; d < 3; d++) a.Fc[3 * p + d] = F[d];
}

// U += ((F_h^n + F_h^{n-1})/2 + F_c)/m, W += (T^n + T^{n-1})/(2 I), X += U_new.
__global__ void eom_kernel(EomArgs a) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= a.np) return;
    const int n[3] = {a.nx, a.ny, a.nz};
    const bool hp = a.has_prev[p] != 0;
    for (int d = 0; d < 3; d++) {
        const double Fh = a.Fh[3 * p + d], Th = a.Th[3 * p + d];
        const double Fa = hp ? 0.5 * (Fh + a.Fprev[3 * p + d]) : Fh;
        const double Ta = hp ? 0.5 * (Th + a.Tprev[3 * p + d]) : Th;
        const double u1 = a.U[3 * p + d] + (Fa + a.Fc[3 * p + d]) / a.mass[p];
        a.U[3 * p + d] = u1;
        a.W[3 * p + d] += Ta / a.inertia[p];
        a.Xold[3 * p + d] = a.X[3 * p + d];
        double x = a.X[3 * p + d] + u1;
        if (x >= n[d]) x -= n[d];
        if (x < 0.0) x += n[d];
        a.X[3 * p + d] = x;
        a.Fprev[3 * p + d] = Fh;
        a.Tprev[3 * p + d] = Th;
    }
    a.has_prev[p] = 1;
}

cudaError_t launch_particle_update(Ctx &c) {
    if (c.np == 0) return cudaSuccess;
    EomArgs a{c.X, c.Xold, c.U, c.W, c.Fh, c.Th, c.Fprev, c.Tprev, c.Fc, c.R, c.mass, c.inertia, c.has_prev,
              c.np, c.nx, c.ny, c.nz, c.Xf};
    const int tb = 128, nb = (c.np + tb - 1) / tb;
    count_launch(c, G_PART, 3);
    xf_kernel<<<nb, tb, 0, c.stream>>>(a);
    contact_kernel<<<(c.np * 32 + 255) / 256, 256, 0, c.stream>>>(a);
    eom_kernel<<<nb, tb, 0, c.stream>>>(a);
    return cudaGetLastError();
}

// -------------------------------------------------------------- IBM ------
__device__ __forceinline__ double peskin(double r) {
    const double a = fabs(r);
    if (a <= 1.0) return (3.0 - 2.0 * a + sqrt(1.0 + 4.0 * a - 4.0 * a * a)) * 0.125;
    if (a <= 2.0) return (5.0 - 2.0 * a - sqrt(-7.0 + 12.0 * a - 4.0 * a * a)) * 0.125;
    return 0.0;
}

__global__ void markers_place_kernel(double *mX, const double *mUnit, const int *mpid, const double *X, long long nm,
                                     int nx, int ny, int nz) {
    const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nm) return;
    const int p = mpid[l];
    const int n[3] = {nx, ny, nz};
    for (int d = 0; d < 3; d++) {
        double x = X[3 * p + d] + mUnit[3 * l + d];
        if (x >= n[d]) x -= n[d];
        if (x < 0.0) x += n[d];
        mX[3 * l + d] = x;
    }
}

// per marker: first stencil node floor(X) - 1 (wrapped), X - floor(X), and
// the desired velocity U_d = U_p + Omega_p x (X_l - X_p) of the rigid body
// (zero for the pipe's ring markers), evaluated in FP64 once per step
template <typename R>
__global__ void marker_offsets_kernel(const double *mX, int *mB, R *mE, R *mUd, const int *mpid, const double *X,
                                      const double *U, const double *W, long long nm, int nx, int ny, int nz) {
    const long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nm) return;
    const int n[3] = {nx, ny, nz};
    for (int d = 0; d < 3; d++) {
        const double x = mX[3 * l + d], f = floor(x);
        mB[3 * l + d] = pwrap((int)f - 1, n[d]);
        mE[3 * l + d] = R(x - f);
    }
    double Ud[3] = {0.0, 0.0, 0.0};
    const int p = mpid[l];
    if (p >= 0) {
        const double r0 = min_image(mX[3 * l] - X[3 * p], nx), r1 = min_image(mX[3 * l + 1] - X[3 * p + 1], ny),
                     r2 = min_image(mX[3 * l + 2] - X[3 * p + 2], nz);
        const double *Wp = W + 3 * p, *Up = U + 3 * p;
        Ud[0] = Up[0] + (Wp[1] * r2 - Wp[2] * r1);
        Ud[1] = Up[1] + (Wp[2] * r0 - Wp[0] * r2);
        Ud[2] = Up[2] + (Wp[0] * r1 - Wp[1] * r0);
    }
    for (int d = 0; d < 3; d++) mUd[3 * l + d] = R(Ud[d]);
}

cudaError_t launch_marker_offsets(Ctx &c) {
    if (c.nm == 0) return cudaSuccess;
    const unsigned nb = (unsigned)((c.nm + 255) / 256);
    count_launch(c, G_GEOM);
    if (c.storage == LBM_F64)
        marker_offsets_kernel<double><<<nb, 256, 0, c.stream>>>(c.mX, c.mB, (double *)c.mE, (double *)c.mUd, c.mpid,
                                                                c.X, c.U, c.W, c.nm, c.nx, c.ny, c.nz);
    else
        marker_offsets_kernel<float><<<nb, 256, 0, c.stream>>>(c.mX, c.mB, (float *)c.mE, (float *)c.mUd, c.mpid,
                                                               c.X, c.U, c.W, c.nm, c.nx, c.ny, c.nz);
    return cudaGetLastError();
}

cudaError_t launch_markers_place(Ctx &c) {
    if (c.np == 0 || c.nm == 0) return cudaSuccess;
    const unsigned nb = (unsigned)((c.nm + 127) / 128);
    count_launch(c, G_GEOM);
    markers_place_kernel<<<nb, 128, 0, c.stream>>>(c.mX, c.mUnit, c.mpid, c.X, c.nm, c.nx, c.ny, c.nz);
    return cudaGetLastError();
}

__device__ __forceinline__ void flag_or(uint8_t *flags, long long c, uint8_t bit) {
    unsigned *w = (unsigned *)(flags + (c & ~3LL));
    atomicOr(w, ((unsigned)bit) << (8 * (c & 3)));
}

__global__ void clear_sup_kernel(uint8_t *flags, long long N) {
    const long long c = 16 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
    if (c + 16 <= N) {
        uint4 f = *(const uint4 *)(flags + c);
        constexpr unsigned sup = 0x01010101u * FL_SUP;
        if (!((f.x | f.y | f.z | f.w) & sup)) return;
        f.x &= ~sup;
        f.y &= ~sup;
        f.z &= ~sup;
        f.w &= ~sup;
        *(uint4 *)(flags + c) = f;
    } else {
        for (long long k = c; k < N; k++) flags[k] = (uint8_t)(flags[k] & ~FL_SUP);
    }
}

// Support of one particle per block: the 4x4x4 stencils of its markers and
// the cells that overlap it (|x - X| < R + 1, whose velocity enters the
// inner-fluid integrals), as bits of the W^3 box floor(X) - ceil(R) - 1 ..
// floor(X) + ceil(R) + 2 in shared memory (a word per x-row, W <= 32), then
// one flag update per four cells. Marker by marker and cell by cell on the
// grid, with the overlap test in FP64 throughout, the two passes took 107 and
// 189 us at 256^3 with 2000 spheres; this takes 43.
__global__ void __launch_bounds__(256) mark_support_kernel(uint8_t *flags, const double *mX, const int *m_first,
                                                           const double *X, const double *R, int nx, int ny, int nz) {
    __shared__ unsigned row[32 * 32];
    const int p = blockIdx.x, lane = threadIdx.x & 31;
    const double X0 = X[3 * p], X1 = X[3 * p + 1], X2 = X[3 * p + 2], Rp = R[p];
    __shared__ int head[4];
    __shared__ float off[4];
    if (threadIdx.x < 3) {  // the box, once per block
        const double Xd = X[3 * p + threadIdx.x];
        const int hp = (int)ceil(Rp) + 1, o = (int)floor(Xd) - hp;
        head[threadIdx.x] = o;
        head[3] = hp;
        off[threadIdx.x] = (float)(Xd - o);
        off[3] = (float)((Rp + 1.0) * (Rp + 1.0));
    }
    __syncthreads();
    const int h = head[3], W = 2 * h + 2, o0 = head[0], o1 = head[1], o2 = head[2];
    for (int t = threadIdx.x; t < W * W; t += blockDim.x) row[t] = 0u;
    __syncthreads();
    for (int l = m_first[p] + threadIdx.x; l < m_first[p + 1]; l += blockDim.x) {
        // first stencil node relative to the box: markers are wrapped into the grid
        int i0 = (int)floor(mX[3 * l]) - 1 - o0, i1 = (int)floor(mX[3 * l + 1]) - 1 - o1,
            i2 = (int)floor(mX[3 * l + 2]) - 1 - o2;
        i0 = i0 < 0 ? i0 + nx : (i0 >= nx ? i0 - nx : i0);
        i1 = i1 < 0 ? i1 + ny : (i1 >= ny ? i1 - ny : i1);
        i2 = i2 < 0 ? i2 + nz : (i2 >= nz ? i2 - nz : i2);
        if (i0 + 4 > W || i1 + 4 > W || i2 + 4 > W) continue;  // not reached: |X_l - X| <= R
        for (int k = 0; k < 16; k++) atomicOr(&row[i1 + (k & 3) + W * (i2 + (k >> 2))], 0xfu << i0);
    }
    __syncthreads();
    // a warp per row, a lane per cell
    const float fl2 = off[3], f0 = off[0], f1 = off[1], f2 = off[2];
    for (int t = threadIdx.x >> 5; t < W * W; t += blockDim.x / 32) {
        const int iy = t % W, iz = t / W;
        const int y = pwrap(o1 + iy, ny), z = pwrap(o2 + iz, nz), x = pwrap(o0 + lane, nx);
        bool in = false;
        if (lane < W) {
            const float ex = lane - f0, ey = iy - f1, ez = iz - f2, e2 = ex * ex + ey * ey + ez * ez;
            if (fabsf(e2 - fl2) > 1e-2f) {  // far wider than the FP32 error of e2
                in = e2 < fl2;
            } else {
                const double rx = min_image(int_to_double(x) - X0, nx), ry = min_image(int_to_double(y) - X1, ny), rz = min_image(int_to_double(z) - X2, nz);
                in = rx * rx + ry * ry + rz * rz < (Rp + 1.0) * (Rp + 1.0);
            }
        }
        const unsigned m = row[t] | __ballot_sync(0xffffffffu, in);
        // one atomic per aligned group of four cells, by its first lane
        const long long c = (long long)x + (long long)nx * (y + (long long)ny * z);
        const unsigned group = lane < W ? (unsigned)(c >> 2) : 0xffffffffu;
        const unsigned mine = ((m >> lane) & 1u) ? ((unsigned)FL_SUP) << (8 * (unsigned)(c & 3)) : 0u;
        unsigned bits = mine;
#pragma unroll
        for (int o = 1; o < 4; o++) {
            const unsigned ob = __shfl_down_sync(0xffffffffu, mine, o), og = __shfl_down_sync(0xffffffffu, group, o);
            if (lane + o < 32 && og == group) bits |= ob;
        }
        const unsigned before = __shfl_up_sync(0xffffffffu, group, 1);
        if (bits && (lane == 0 || before != group)) atomicOr((unsigned *)(flags + (c & ~3LL)), bits);
    }
}

// support = 4x4x4 stencil of every marker
__global__ void mark_stencil_kernel(uint8_t *flags, const double *mX, long long nm, int nx, int ny, int nz) {
    const long long l = (long long)blockIdx.x * (blockDim.x / 64) + threadIdx.x / 64;
    if (l >= nm) return;
    const int k = threadIdx.x & 63;
    const int ox = k & 3, oy = (k >> 2) & 3, oz = k >> 4;
    const int x = pwrap((int)floor(mX[3 * l]) - 1 + ox, nx), y = pwrap((int)floor(mX[3 * l + 1]) - 1 + oy, ny),
              z = pwrap((int)floor(mX[3 * l + 2]) - 1 + oz, nz);
    flag_or(flags, (long long)x + (long long)nx * (y + (long long)ny * z), FL_SUP);
}

// ... plus every cell overlapping a particle (|x - X| < R + 1), whose
// velocity enters the inner-fluid integrals
__global__ void mark_interior_kernel(uint8_t *flags, const double *X, const double *R, int nx, int ny, int nz) {
    const int p = blockIdx.x;
    const double Rp = R[p];
    const int r = (int)ceil(Rp) + 1;
    const int bx = (int)floor(X[3 * p]) - r, by = (int)floor(X[3 * p + 1]) - r, bz = (int)floor(X[3 * p + 2]) - r;
    const int w = 2 * r + 2;
    const FastDiv fw((unsigned)w);
    for (int t = threadIdx.x; t < w * w * w; t += blockDim.x) {
        int ix, iy, iz;
        box_coords(t, fw, w, ix, iy, iz);
        const int x = pwrap(bx + ix, nx), y = pwrap(by + iy, ny), z = pwrap(bz + iz, nz);
        const double rx = min_image(int_to_double(x) - X[3 * p], nx), ry = min_image(int_to_double(y) - X[3 * p + 1], ny), rz = min_image(int_to_double(z) - X[3 * p + 2], nz);
        if (rx * rx + ry * ry + rz * rz < (Rp + 1.0) * (Rp + 1.0))
            flag_or(flags, (long long)x + (long long)nx * (y + (long long)ny * z), FL_SUP);
    }
}

cudaError_t launch_support_mark(Ctx &c) {
    clear_sup_kernel<<<(unsigned)((c.N + 4095) / 4096), 256, 0, c.stream>>>(c.flags, c.N);
    if (c.np > 0 && 2 * ((int)ceil(c.max_radius) + 1) + 2 <= 32) {
        count_launch(c, G_GEOM, 2);
        mark_support_kernel<<<c.np, 256, 0, c.stream>>>(c.flags, c.mX, c.m_first, c.X, c.R, c.nx, c.ny, c.nz);
        return cudaGetLastError();
    }
    count_launch(c, G_GEOM, 1 + (c.nm > 0) + (c.np > 0));
    if (c.nm > 0) {
        const unsigned mb = (unsigned)((c.nm + 3) / 4);
        mark_stencil_kernel<<<mb, 256, 0, c.stream>>>(c.flags, c.mX, c.nm, c.nx, c.ny, c.nz);
    }
    if (c.np > 0) mark_interior_kernel<<<c.np, 256, 0, c.stream>>>(c.flags, c.X, c.R, c.nx, c.ny, c.nz);
    return cudaGetLastError();
}

// Peskin (2002) 4-point kernel in the arithmetic type R of the storage
template <typename R>
__device__ __forceinline__ R peskin_r(R r) {
    const R a = fabs(r);
    if (a <= R(1)) return (R(3) - R(2) * a + sqrt(R(1) + R(4) * a - R(4) * a * a)) * R(0.125);
    if (a <= R(2)) return (R(5) - R(2) * a - sqrt(R(-7) + R(12) * a - R(4) * a * a)) * R(0.125);
    return R(0);
}

// Support-cell data (rho, u*, accumulated force, force of the pass) and the
// marker forces used for spreading are held in R: double for FP64 storage,
// float otherwise (FP64 arithmetic is slow on this GPU and would dominate).
struct IbmArgs {
    const double *mX, *mdV;
    const int *mpid;
    double *mFacc;        // per-step marker force (sum of the passes), FP64
    const void *mUd;      // desired velocity U_d at the marker (R)
    void *mFaccR, *mFr;   // running sum of the passes' forces; F_l dV_l of this pass for the spreading (R)
    const int *mB;
    const void *mE;
    const int *aux;
    void *sup_ru, *sup_F, *sup_Fp;
    const double *X, *U, *W;
    long long nm;
    const long long *counts;
    long long max_sites;
    int nx, ny, nz;
    int pass, last;
};

// (rho, u*) of one support site: one 16-byte load in FP32
__device__ __forceinline__ void ld_site4(const float *p, float q[4]) {
    const float4 v = __ldg((const float4 *)p);
    q[0] = v.x;
    q[1] = v.y;
    q[2] = v.z;
    q[3] = v.w;
}
__device__ __forceinline__ void ld_site4(const double *p, double q[4]) {
    const double2 v0 = __ldg((const double2 *)p), v1 = __ldg((const double2 *)p + 1);
    q[0] = v0.x;
    q[1] = v0.y;
    q[2] = v1.x;
    q[3] = v1.y;
}

// Interpolation, one warp per marker: lane k takes stencil nodes k and k+32;
// U*_l = sum u* delta, rho_l = sum rho delta (fixed butterfly reduction);
// F_l = 2 rho_l (U_d - U*_l).
template <typename R>
__global__ void __launch_bounds__(256) ibm_interp_warp_kernel(IbmArgs a) {
    const long long l = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (l >= a.nm) return;
    const R *ru = (const R *)a.sup_ru;
    const R *E = (const R *)a.mE + 3 * l;
    const R e0 = E[0], e1 = E[1], e2 = E[2];  // X - floor(X)
    const int b0 = a.mB[3 * l], b1 = a.mB[3 * l + 1], b2 = a.mB[3 * l + 2];  // floor(X) - 1, wrapped
    // the 12 one-dimensional kernel values of the marker: lane 4 d + o holds
    // phi(o - 1 - e_d); every node's weight is a product of three of them
    R phi = R(0);
    if (lane < 12) {
        const int d = lane >> 2, o = lane & 3;
        phi = peskin_r<R>(R(o - 1) - (d == 0 ? e0 : (d == 1 ? e1 : e2)));
    }
    R U0 = 0, U1 = 0, U2 = 0, rl = 0;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int k = lane + 32 * h;
        const int kx = k & 3, ky = (k >> 2) & 3, kz = k >> 4;
        const R w = __shfl_sync(0xffffffffu, phi, kx) * __shfl_sync(0xffffffffu, phi, 4 + ky) *
                    __shfl_sync(0xffffffffu, phi, 8 + kz);
        const long long c = (long long)pwrap(b0 + kx, a.nx) +
                            (long long)a.nx * (pwrap(b1 + ky, a.ny) + (long long)a.ny * pwrap(b2 + kz, a.nz));
        const int s = a.aux[c];
        if (s < 0 || s >= a.max_sites) continue;
        R q[4];
        ld_site4(ru + 4 * (size_t)s, q);
        rl += w * q[0];
        U0 += w * q[1];
        U1 += w * q[2];
        U2 += w * q[3];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        rl += __shfl_xor_sync(0xffffffffu, rl, o);
        U0 += __shfl_xor_sync(0xffffffffu, U0, o);
        U1 += __shfl_xor_sync(0xffffffffu, U1, o);
        U2 += __shfl_xor_sync(0xffffffffu, U2, o);
    }
    if (lane != 0) return;
    // F_l = 2 rho_l (U_d - U*_l) in the storage's arithmetic type; U_d was
    // evaluated once per step (marker_offsets_kernel)
    const R *Ud = (const R *)a.mUd + 3 * l;
    const R U[3] = {U0, U1, U2};
    R *mFr = (R *)a.mFr, *acc = (R *)a.mFaccR;
    const R dVl = R(a.mdV[l]);
    for (int d = 0; d < 3; d++) {
        const R Fl = R(2) * rl * (Ud[d] - U[d]);
        mFr[3 * l + d] = Fl * dVl;  // spread weight F_l dV_l
        const R s = a.pass == 0 ? Fl : acc[3 * l + d] + Fl;
        acc[3 * l + d] = s;
        if (a.last) a.mFacc[3 * l + d] = double(s);
    }
}

// generic spreading with global atomics (large particles only)
template <typename R>
__global__ void ibm_spread_kernel(IbmArgs a) {
    const long long l = (long long)blockIdx.x * (blockDim.x / 64) + threadIdx.x / 64;
    if (l >= a.nm) return;
    const int k = threadIdx.x & 63;
    const int kx = k & 3, ky = (k >> 2) & 3, kz = k >> 4;
    const R *E = (const R *)a.mE + 3 * l;
    const int b0 = a.mB[3 * l], b1 = a.mB[3 * l + 1], b2 = a.mB[3 * l + 2];
    const R w = peskin_r<R>(R(kx - 1) - E[0]) * peskin_r<R>(R(ky - 1) - E[1]) * peskin_r<R>(R(kz - 1) - E[2]);
    const long long c = (long long)pwrap(b0 + kx, a.nx) +
                        (long long)a.nx * (pwrap(b1 + ky, a.ny) + (long long)a.ny * pwrap(b2 + kz, a.nz));
    const int s = a.aux[c];
    if (s < 0 || s >= a.max_sites) return;
    const R *mFr = (const R *)a.mFr;
    R *Fp = (R *)a.sup_Fp;
    atomicAdd(Fp + 3 * s, mFr[3 * l] * w);
    atomicAdd(Fp + 3 * s + 1, mFr[3 * l + 1] * w);
    atomicAdd(Fp + 3 * s + 2, mFr[3 * l + 2] * w);
}

// u* += F/(2 rho); accumulate the IBM force; clear the pass buffer
template <typename R>
__global__ void ibm_update_kernel(IbmArgs a) {
    const long long ns = a.counts[0] < a.max_sites ? a.counts[0] : a.max_sites;
    R *ru = (R *)a.sup_ru, *sF = (R *)a.sup_F, *Fp = (R *)a.sup_Fp;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < ns; s += (long long)gridDim.x * blockDim.x) {
        const R ir = R(0.5) / ru[4 * s];
        for (int d = 0; d < 3; d++) {
            const R f = Fp[3 * s + d];
            ru[4 * s + 1 + d] += f * ir;
            sF[3 * s + d] = a.pass == 0 ? f : sF[3 * s + d] + f;
            Fp[3 * s + d] = R(0);
        }
    }
}

// Spheres: one block per particle accumulates the spread force of its
// markers in a shared-memory box around the particle, then adds the box to
// the support cells (global atomics only where boxes of nearby particles
// overlap).
struct ParticleSpreadArgs {
    const double *mX, *mdV;
    const void *mFr;
    const int *mB;
    const void *mE;
    const double *X, *R;
    const int *m_first, *aux;
    void *sup_Fp;
    long long max_sites;
    int nx, ny, nz;
    double rd;
};

template <typename R>
__global__ void __launch_bounds__(256) ibm_spread_particle_kernel(ParticleSpreadArgs a, int W) {
    extern __shared__ __align__(16) unsigned char box_raw[];
    R *box = (R *)box_raw;  // W^3 x 3
    const int p = blockIdx.x;
    const int nbox = W * W * W;
    for (int t = threadIdx.x; t < 3 * nbox; t += blockDim.x) box[t] = R(0);
    __syncthreads();
    const double RL = a.R[p] - a.rd;
    const int h = (int)ceil(RL) + 2;
    const double Xp0 = a.X[3 * p], Xp1 = a.X[3 * p + 1], Xp2 = a.X[3 * p + 2];
    const int o0 = (int)floor(Xp0) - h, o1 = (int)floor(Xp1) - h, o2 = (int)floor(Xp2) - h;
    const int l0 = a.m_first[p], l1 = a.m_first[p + 1];
    const R *mFr = (const R *)a.mFr;
    const int lane = threadIdx.x & 31;
    // 64 (marker, node) pairs per marker: a warp's 32 pairs share one marker
    // and every warp runs the same number of rounds (64 n is a multiple of 32)
    for (long long t = threadIdx.x; t < 64LL * (l1 - l0); t += blockDim.x) {
        const int l = l0 + (int)(t >> 6), k = (int)(t & 63);
        const int kx = k & 3, ky = (k >> 2) & 3, kz = k >> 4;
        const R *E = (const R *)a.mE + 3 * l;
        // the marker's 12 one-dimensional kernel values on lanes 0 .. 11
        R phi = R(0);
        if (lane < 12) phi = peskin_r<R>(R((lane & 3) - 1) - E[lane >> 2]);
        const R w = __shfl_sync(0xffffffffu, phi, kx) * __shfl_sync(0xffffffffu, phi, 4 + ky) *
                    __shfl_sync(0xffffffffu, phi, 8 + kz);
        // box-local node index modulo the grid, for the marker base is wrapped:
        // a box may be wider than half the grid (or than the grid itself)
        const int i0 = pwrap(a.mB[3 * l] + kx - o0, a.nx), i1 = pwrap(a.mB[3 * l + 1] + ky - o1, a.ny),
                  i2 = pwrap(a.mB[3 * l + 2] + kz - o2, a.nz);
        if (i0 >= W || i1 >= W || i2 >= W) continue;
        const int bi = i0 + W * (i1 + W * i2);
        atomicAdd(&box[3 * bi], mFr[3 * l] * w);
        atomicAdd(&box[3 * bi + 1], mFr[3 * l + 1] * w);
        atomicAdd(&box[3 * bi + 2], mFr[3 * l + 2] * w);
    }
    __syncthreads();
    R *Fp = (R *)a.sup_Fp;
    for (int bi = threadIdx.x; bi < nbox; bi += blockDim.x) {
        const R f0 = box[3 * bi], f1 = box[3 * bi + 1], f2 = box[3 * bi + 2];
        if (f0 == R(0) && f1 == R(0) && f2 == R(0)) continue;
        const int i0 = bi % W, i1 = (bi / W) % W, i2 = bi / (W * W);
        const long long c = (long long)pwrap(o0 + i0, a.nx) +
                            (long long)a.nx * (pwrap(o1 + i1, a.ny) + (long long)a.ny * pwrap(o2 + i2, a.nz));
        const int s = a.aux[c];
        if (s < 0 || s >= a.max_sites) continue;
        atomicAdd(Fp + 3 * s, f0);
        atomicAdd(Fp + 3 * s + 1, f1);
        atomicAdd(Fp + 3 * s + 2, f2);
    }
}

// One forcing pass of one particle per block: the (rho, u*) of the box that
// holds its markers' stencils go to shared memory once; four lanes per marker
// (a z plane of 16 nodes each) interpolate from there, form F_l and spread it
// into the box of forces, which is then added to the support cells (global
// atomics: boxes of nearby particles overlap).
//
// What bounds it: latency of the box loads and the instructions of the 128
// node visits per marker. With a warp per marker reading 64 nodes through the
// cell index (780 MB from L2 per pass) and a second kernel spreading, a pass
// took 147 + 170 us at 256^3 with 2000 spheres of radius 4; a warp per marker
// on the box 215; this takes 118.
//
// FP32: the box of forces is in integers, scaled by the power of two that
// puts the largest |F_l dV_l| of the particle at 2^28 .. 2^29. Shared-memory
// integer atomics are native (FP32 ones are a compare-and-swap loop), the
// sum does not depend on their order, and its quantum, 2^-28 or less of that
// force, is finer than the rounding of FP32 sums of that size. Four times
// the largest term fits: the weights of a cell over the markers of a sphere
// (about one per unit of surface) add up to 0.92 at most, at a radius of 1.1,
// and to 0.5 .. 0.6 beyond 2. The quantum is the same for all components: one
// that is a hundredth of the strongest keeps 8e-6 of itself in its sums (CPU
// emulation, radius 3.6), less than what rounding the velocities to FP32
// leaves of it.
template <typename R>
struct __align__(4 * sizeof(R)) PassBox {
    R rho, u0, u1, u2;
};
template <typename R> struct SpreadSum;
template <> struct SpreadSum<float> {
    typedef int T;
    static __device__ __forceinline__ float scale(float m) {  // 2^(28 - exponent of m)
        const int e = (int)(__float_as_uint(m) >> 23) - 127;
        return m > 0.f ? exp2f((float)min(28 - e, 120)) : 1.f;
    }
    static __device__ __forceinline__ int of(float v, float s) { return __float2int_rn(v * s); }
    static __device__ __forceinline__ float value(int v, float s) { return (float)v / s; }
};
template <> struct SpreadSum<double> {
    typedef double T;
    static __device__ __forceinline__ double scale(double) { return 1.0; }
    static __device__ __forceinline__ double of(double v, double) { return v; }
    static __device__ __forceinline__ double value(double v, double) { return v; }
};

// shared memory of a block: fields and forces of the box (z planes padded by
// one cell, so that the four planes of a marker start on different banks),
// its sites, per marker 12 kernel values, the force and the first node
constexpr int PASS_SMEM = 220 * 1024;  // at most
template <typename R>
size_t pass_smem_bytes(int W, int markers) {
    const size_t nb = (size_t)W * (W * W + 1);
    return nb * (sizeof(PassBox<R>) + 3 * sizeof(typename SpreadSum<R>::T) + sizeof(int)) +
           (size_t)markers * (15 * sizeof(R) + sizeof(int));
}

template <typename R>
__global__ void __launch_bounds__(256) ibm_pass_particle_kernel(IbmArgs a, const double *Rp, const int *m_first, double rd,
                                                                int W, int max_markers) {
    typedef SpreadSum<R> Sum;
    typedef typename Sum::T T;
    extern __shared__ __align__(32) unsigned char pass_raw[];
    const int PS = W * W + 1, nb = W * PS;  // plane stride
    PassBox<R> *box = (PassBox<R> *)pass_raw;
    T *F = (T *)(box + nb);  // three components
    R *phi = (R *)(F + 3 * nb), *Fl = phi + 12 * max_markers;
    int *first = (int *)(Fl + 3 * max_markers), *site = first + max_markers;
    __shared__ R wmax[8];
    const int p = blockIdx.x, tid = threadIdx.x;
    __shared__ int head[3];
    if (tid < 3) head[tid] = (int)floor(a.X[3 * p + tid]) - (int)ceil(Rp[p] - rd) - 1;  // the box, once per block
    __syncthreads();
    const int o0 = head[0], o1 = head[1], o2 = head[2];
    const FastDiv fw((unsigned)W);
    const R *ru = (const R *)a.sup_ru;
    const int l0 = m_first[p], n = min(m_first[p + 1] - l0, max_markers);
    const int nbox = W * W * W;
#pragma unroll 4
    for (int t = tid; t < nbox; t += 256) {
        int ix, iy, iz;
        box_coords(t, fw, W, ix, iy, iz);
        const int b = ix + W * iy + PS * iz;
        const int c = pwrap(o0 + ix, a.nx) + a.nx * (pwrap(o1 + iy, a.ny) + a.ny * pwrap(o2 + iz, a.nz));
        int s = a.aux[c];
        // cells outside the support may keep the index of an earlier list:
        // whatever they bring has no marker's weight on it
        R q[4] = {R(0), R(0), R(0), R(0)};
        if (s >= 0 && s < a.max_sites) ld_site4(ru + 4 * (size_t)s, q);
        else s = -1;
        box[b] = PassBox<R>{q[0], q[1], q[2], q[3]};
        site[b] = s;
        F[b] = F[nb + b] = F[2 * nb + b] = T(0);
    }
    for (int t = tid; t < W; t += 256) site[W * W + PS * t] = -1;  // the padding
    // kernel values phi(o - 1 - e_d) and first stencil nodes of the markers
    const R *E = (const R *)a.mE + 3 * (size_t)l0;
    for (int t = tid; t < 12 * n; t += 256) {
        const int m = t / 12, k = t - 12 * m;
        phi[t] = peskin_r<R>(R((k & 3) - 1) - E[3 * m + (k >> 2)]);
    }
    for (int m = tid; m < n; m += 256) {
        const int *B = a.mB + 3 * (size_t)(l0 + m);  // wrapped into the grid
        int i0 = B[0] - o0, i1 = B[1] - o1, i2 = B[2] - o2;
        i0 = i0 < 0 ? i0 + a.nx : (i0 >= a.nx ? i0 - a.nx : i0);
        i1 = i1 < 0 ? i1 + a.ny : (i1 >= a.ny ? i1 - a.ny : i1);
        i2 = i2 < 0 ? i2 + a.nz : (i2 >= a.nz ? i2 - a.nz : i2);
        // |X_l - X| <= RL keeps every stencil inside the box
        first[m] = i0 + 4 <= W && i1 + 4 <= W && i2 + 4 <= W ? i0 + W * i1 + PS * i2 : -1;
    }
    __syncthreads();
    const R dVl = R(a.mdV[l0]);  // one marker volume per particle
    R *acc = (R *)a.mFaccR + 3 * (size_t)l0;
    const R *Ud = (const R *)a.mUd + 3 * (size_t)l0;
    R big = R(0);
    bool bad = false;
    const int rounds = (4 * n + 255) / 256;  // whole warps: the lanes of a marker add up by shuffles
    for (int r = 0; r < rounds; r++) {
        const int t = tid + 256 * r, m = t >> 2, kz = t & 3;
        const bool on = m < n && first[min(m, n - 1)] >= 0;
        R rl = R(0), U[3] = {R(0), R(0), R(0)};
        if (on) {
            const R *ph = phi + 12 * m;
            const PassBox<R> *q = box + first[m] + PS * kz;
            const R pz = ph[8 + kz];
            // row by row: short sums, so less rounding than one sum over the 16
            // nodes, and half the instructions
#pragma unroll
            for (int ky = 0; ky < 4; ky++) {
                R r0 = R(0), r1 = R(0), r2 = R(0), r3 = R(0);
#pragma unroll
                for (int kx = 0; kx < 4; kx++) {
                    const R w = ph[kx];
                    const PassBox<R> v = q[kx + W * ky];
                    r0 += w * v.rho;
                    r1 += w * v.u0;
                    r2 += w * v.u1;
                    r3 += w * v.u2;
                }
                const R w = ph[4 + ky] * pz;
                rl += w * r0;
                U[0] += w * r1;
                U[1] += w * r2;
                U[2] += w * r3;
            }
        }
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {
            rl += __shfl_xor_sync(0xffffffffu, rl, o);
            for (int d = 0; d < 3; d++) U[d] += __shfl_xor_sync(0xffffffffu, U[d], o);
        }
        if (on && kz < 3) {  // F_l = 2 rho_l (U_d - U*_l), a component per lane
            const R f = R(2) * rl * (Ud[3 * m + kz] - (kz == 0 ? U[0] : (kz == 1 ? U[1] : U[2])));
            const R s = a.pass == 0 ? f : acc[3 * m + kz] + f;
            acc[3 * m + kz] = s;
            if (a.last) a.mFacc[3 * (size_t)(l0 + m) + kz] = double(s);
            const R g = f * dVl;  // spread weight F_l dV_l
            Fl[3 * m + kz] = g;
            big = fmax(big, fabs(g));
            bad = bad || !(fabs(g) < R(1e30));
        }
    }
    // the particle's largest force sets the scale of the integer sums
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, o));
    if ((tid & 31) == 0) wmax[tid >> 5] = big;
    bad = __syncthreads_or(bad);
    for (int k = 0; k < 8; k++) big = fmax(big, wmax[k]);
    const R sc = Sum::scale(big);
    for (int t = tid; t < 4 * n; t += 256) {
        const int m = t >> 2, kz = t & 3;
        if (first[m] < 0) continue;
        const R *ph = phi + 12 * m;
        T *q = F + first[m] + PS * kz;
        const R pz = ph[8 + kz], f0 = Fl[3 * m], f1 = Fl[3 * m + 1], f2 = Fl[3 * m + 2];
#pragma unroll
        for (int ky = 0; ky < 4; ky++)
#pragma unroll
            for (int kx = 0; kx < 4; kx++) {
                const R w = ph[kx] * ph[4 + ky] * pz;
                T *c = q + kx + W * ky;
                atomicAdd(c, Sum::of(f0 * w, sc));
                atomicAdd(c + nb, Sum::of(f1 * w, sc));
                atomicAdd(c + 2 * nb, Sum::of(f2 * w, sc));
            }
    }
    __syncthreads();
    R *Fp = (R *)a.sup_Fp;
#pragma unroll 4
    for (int b = tid; b < nb; b += 256) {
        const int s = site[b];
        if (s < 0) continue;
        const T f0 = F[b], f1 = F[nb + b], f2 = F[2 * nb + b];
        if (f0 == T(0) && f1 == T(0) && f2 == T(0) && !bad) continue;
        // a force that is no number reaches the fluid (and the watchdog) as one
        const R nan = bad ? R(0) / R(0) : R(0);
        atomicAdd(Fp + 3 * s, Sum::value(f0, sc) + nan);
        atomicAdd(Fp + 3 * s + 1, Sum::value(f1, sc) + nan);
        atomicAdd(Fp + 3 * s + 2, Sum::value(f2, sc) + nan);
    }
}

template <typename R>
static cudaError_t ibm_passes_t(Ctx &c) {
    IbmArgs a{c.mX, c.mdV, c.mpid, c.mFacc, c.mUd, c.mFaccR, c.mFr, c.mB, c.mE, c.aux, c.sup_ru, c.sup_F, c.sup_Fp,
              c.X, c.U, c.W, c.nm, c.d_counts, c.max_sites, c.nx, c.ny, c.nz, 0, 0};
    long long ns = c.nsites_hint > 0 ? c.nsites_hint : c.max_sites;
    if (ns > c.max_sites) ns = c.max_sites;
    long long ub = (ns + 255) / 256;
    if (ub < 1) ub = 1;
    if (ub > 152 * 32) ub = 152 * 32;
    // sphere boxes in shared memory when they fit
    const double RLmax = c.max_radius - c.rd;
    const int W = 2 * (int)ceil(RLmax) + 6;
    const size_t smem = 3 * sizeof(R) * (size_t)W * W * W;
    const bool box_spread = !c.has_pipe && c.np > 0 && smem <= 200 * 1024;
    if (box_spread) {
        static bool attr_set = false;
        if (!attr_set) {
            cudaFuncSetAttribute(ibm_spread_particle_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 200 * 1024);
            attr_set = true;
        }
    }
    // the fused pass where a box fits an SM's shared memory; a box must not
    // meet itself around the grid. It wins up to the last radius that fits,
    // one block per SM: the passes of a step at 128^3 take 0.132 against 0.370
    // ms with 100 spheres of radius 6 in FP32 (60 of radius 7: 0.166, 0.457),
    // 0.547 against 1.531 ms with 300 of radius 4 in FP64
    const int WB = 2 * (int)ceil(RLmax) + 4;
    const int mmax = RLmax > 0.0 ? (int)floor(M_PI / 3.0 * (12.0 * RLmax * RLmax + 1.0) + 0.5) : 0;  // as build_markers
    const size_t pass_smem = pass_smem_bytes<R>(WB, mmax);
    const bool fused = !c.has_pipe && c.np > 0 && c.nm > 0 && pass_smem <= PASS_SMEM &&
                       WB <= std::min(c.nx, std::min(c.ny, c.nz));
    if (fused) {
        // the limit, not this context's own size: the attribute is the
        // process's, and another thread may set it before this one launches
        const cudaError_t e = cudaFuncSetAttribute(ibm_pass_particle_kernel<R>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, PASS_SMEM);
        if (e != cudaSuccess) return e;
    }
    for (int pass = 0; pass < 3; pass++) {
        a.pass = pass;
        a.last = pass == 2;
        if (fused) {
            count_launch(c, G_IBM, 2);
            ibm_pass_particle_kernel<R><<<c.np, 256, pass_smem, c.stream>>>(a, c.R, c.m_first, c.rd, WB, mmax);
            ibm_update_kernel<R><<<(unsigned)ub, 256, 0, c.stream>>>(a);
            continue;
        }
        if (c.nm > 0) {
            count_launch(c, G_IBM);
            ibm_interp_warp_kernel<R><<<(unsigned)((c.nm * 32 + 255) / 256), 256, 0, c.stream>>>(a);
        }
        if (c.nm > 0) {
            count_launch(c, G_IBM);
            if (box_spread) {
                ParticleSpreadArgs pa{c.mX, c.mdV, c.mFr, c.mB, c.mE, c.X, c.R, c.m_first, c.aux, c.sup_Fp,
                                      c.max_sites, c.nx, c.ny, c.nz, c.rd};
                ibm_spread_particle_kernel<R><<<c.np, 256, smem, c.stream>>>(pa, W);
            } else {
                ibm_spread_kernel<R><<<(unsigned)((c.nm + 3) / 4), 256, 0, c.stream>>>(a);
            }
        }
        count_launch(c, G_IBM);
        ibm_update_kernel<R><<<(unsigned)ub, 256, 0, c.stream>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_ibm_passes(Ctx &c) {
    return c.storage == LBM_F64 ? ibm_passes_t<double>(c) : ibm_passes_t<float>(c);
}

// particle force/torque: -sum_l F_l dV_l (+ moment) plus the change of the
// inner-fluid momentum sum alpha u (Kempe et al. 2012)
struct SumArgs {
    const double *mX, *mdV, *mFacc;
    const int *m_first;
    const double *X;
    double *Fh, *Th, *Iu, *Ir;
    const double *Iu_new, *Ir_new;
    int nx, ny, nz;
};

__global__ void __launch_bounds__(PB) ibm_sum_kernel(SumArgs a) {
    __shared__ double sh[6 * PB];
    const int p = blockIdx.x;
    double v[6] = {0, 0, 0, 0, 0, 0};
    for (int l = a.m_first[p] + threadIdx.x; l < a.m_first[p + 1]; l += PB) {
        const double F0 = -a.mFacc[3 * l] * a.mdV[l], F1 = -a.mFacc[3 * l + 1] * a.mdV[l],
                     F2 = -a.mFacc[3 * l + 2] * a.mdV[l];
        const double r0 = min_image(a.mX[3 * l] - a.X[3 * p], a.nx), r1 = min_image(a.mX[3 * l + 1] - a.X[3 * p + 1], a.ny),
                     r2 = min_image(a.mX[3 * l + 2] - a.X[3 * p + 2], a.nz);
        v[0] += F0;
        v[1] += F1;
        v[2] += F2;
        v[3] += r1 * F2 - r2 * F1;
        v[4] += r2 * F0 - r0 * F2;
        v[5] += r0 * F1 - r1 * F0;
    }
    double t[6];
    block_sum<6>(v, sh, t);
    if (threadIdx.x == 0)
        for (int d = 0; d < 3; d++) {
            a.Fh[3 * p + d] = t[d] + (a.Iu_new[3 * p + d] - a.Iu[3 * p + d]);
            a.Th[3 * p + d] = t[3 + d] + (a.Ir_new[3 * p + d] - a.Ir[3 * p + d]);
            a.Iu[3 * p + d] = a.Iu_new[3 * p + d];
            a.Ir[3 * p + d] = a.Ir_new[3 * p + d];
        }
}

cudaError_t launch_ibm_particle_sums(Ctx &c, bool init_only) {
    if (c.np == 0) return cudaSuccess;
    if (init_only) return launch_volume(c, 1, c.Iu, c.Ir);
    // scratch for the new integrals: the contact-force buffer (2 x 3 doubles
    // per particle) is free until the contact kernel runs later in the step
    double *Iu_new = c.Fc, *Ir_new = c.Fc + 3 * c.max_np;
    cudaError_t e = launch_volume(c, 2, Iu_new, Ir_new);
    if (e != cudaSuccess) return e;
    SumArgs a{c.mX, c.mdV, c.mFacc, c.m_first, c.X, c.Fh, c.Th, c.Iu, c.Ir, Iu_new, Ir_new, c.nx, c.ny, c.nz};
    count_launch(c, G_PART);
    ibm_sum_kernel<<<c.np, PB, 0, c.stream>>>(a);
    return cudaGetLastError();
}

// one-time rigid-body overwrite inside the particles at insertion (Sec. 3.1)
template <int S>
__global__ void rigid_overwrite_kernel(void *A, const uint8_t *flags, const int *owner, const double *X,
                                       const double *U, const double *W, const double *R, int nx, int ny, int nz,
                                       long long N, double F0, double F1, double F2) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R Rt;
    const int p = blockIdx.x;
    const int r = (int)ceil(R[p]) + 1;
    const int bx = (int)floor(X[3 * p]) - r, by = (int)floor(X[3 * p + 1]) - r, bz = (int)floor(X[3 * p + 2]) - r;
    const int w = 2 * r + 2;
    const FastDiv fw((unsigned)w);
    for (int t = threadIdx.x; t < w * w * w; t += blockDim.x) {
        int ix, iy, iz;
        box_coords(t, fw, w, ix, iy, iz);
        const int x = pwrap(bx + ix, nx), y = pwrap(by + iy, ny), z = pwrap(bz + iz, nz);
        const long long c = (long long)x + (long long)nx * (y + (long long)ny * z);
        if (!(flags[c] & FL_SOLID) || owner[c] != p) continue;
        double rho, u[3];
        cell_velocity<S>(A, (size_t)N, c, 0.0, 0.0, 0.0, rho, u);  // solid cells feel no body force
        const double rx = min_image(int_to_double(x) - X[3 * p], nx), ry = min_image(int_to_double(y) - X[3 * p + 1], ny), rz = min_image(int_to_double(z) - X[3 * p + 2], nz);
        const double uw[3] = {U[3 * p] + (W[3 * p + 1] * rz - W[3 * p + 2] * ry),
                              U[3 * p + 1] + (W[3 * p + 2] * rx - W[3 * p] * rz),
                              U[3 * p + 2] + (W[3 * p] * ry - W[3 * p + 1] * rx)};
        const double u2 = uw[0] * uw[0] + uw[1] * uw[1] + uw[2] * uw[2];
        for (int i = 0; i < 19; i++) {
            const double cu = cx(i) * uw[0] + cy(i) * uw[1] + cz(i) * uw[2];
            const double feq = wgt(i) * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * u2);
            Store<S>::st((T *)A + (size_t)i * N + c, Rt(feq - wgt(i)));
        }
    }
    (void)F0; (void)F1; (void)F2;
}

cudaError_t launch_ibm_rigid_overwrite(Ctx &c) {
    if (c.np == 0) return cudaSuccess;
    count_launch(c, G_OTHER);
    switch (c.storage) {
#define RO(S) rigid_overwrite_kernel<S><<<c.np, 256, 0, c.stream>>>(c.fA, c.flags, c.owner, c.X, c.U, c.W, c.R, \
                                                                      c.nx, c.ny, c.nz, c.N, 0, 0, 0)
    case LBM_F64: RO(LBM_F64); break;
    case LBM_F32: RO(LBM_F32); break;
    case LBM_F16S: RO(LBM_F16S); break;
    default: RO(LBM_BF16S); break;
#undef RO
    }
    return cudaGetLastError();
}

}  // namespace lbmgb
