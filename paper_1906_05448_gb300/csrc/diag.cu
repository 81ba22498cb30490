// Diagnostics (Sec. 3.2, Sec. 2.2): macroscopic fields of the current state,
// rigid-body masking of particle regions, kinetic energy, dissipation
// 2 nu s_ij s_ij from second-order central differences, radial profiles
// around particles and the pipe bulk velocity. The sums of lbm_stats are
// block partials added on the device in a fixed order (deterministic): FP64,
// or pairs of floats of 48 bits for 32- and 16-bit storage. The pipe profiles
// add their columns with global FP64 atomics, in no fixed order.
#include "columns.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

namespace lbmgb {

__device__ __forceinline__ double dmimg(double d, int n) {
    if (d > 0.5 * n) d = __dsub_rn(d, (double)n);
    else if (d < -0.5 * n) d = __dadd_rn(d, (double)n);
    return d;
}
__device__ __forceinline__ int dwrap(int a, int n) {
    a %= n;
    return a < 0 ? a + n : a;
}

// rho and u of the post-collision state: sum f c = rho u + F/2 after a Guo
// collision with total force F (body force on fluid cells + IBM force).
// u32, if not null, receives FP32 records (ux, uy, uz, rho), 16 bytes per
// cell (the closure's gather input, the statistics of 32- and 16-bit
// storage), alone with rec_only.
template <int S>
__global__ void macro_kernel(const void *A, const uint8_t *flags, const int *aux, const void *sup_Fv, double *rho_o,
                             double *u_o, float *u32, long long N, double F0, double F1, double F2, int ibb, int ibm,
                             long long max_sites, int rec_only) {
    typedef typename Store<S>::T T;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= N) return;
    const uint8_t fl = flags[c];
    if (ibb && (fl & FL_SOLID)) {
        if (!rec_only) {
            rho_o[c] = 0.0;
            u_o[c] = u_o[N + c] = u_o[2 * N + c] = 0.0;
        }
        if (u32) reinterpret_cast<float4 *>(u32)[c] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    // arithmetic type of the storage (FP32 for the 32- and 16-bit layouts)
    typedef typename Store<S>::R R;
    const T *P = (const T *)A;
    R r = R(0), j0 = R(0), j1 = R(0), j2 = R(0);
#pragma unroll
    for (int i = 0; i < 19; i++) {
        const R g = Store<S>::ld(P + (size_t)i * N + c);
        r += g;
        j0 += g * R(cx(i));
        j1 += g * R(cy(i));
        j2 += g * R(cz(i));
    }
    const bool fluid = !(fl & FL_SOLID);
    R Fx = fluid ? R(F0) : R(0), Fy = fluid ? R(F1) : R(0), Fz = fluid ? R(F2) : R(0);
    if (ibm && (fl & FL_SUP) && aux[c] >= 0 && aux[c] < max_sites) {
        const R *sup_F = (const R *)sup_Fv;
        const int s = aux[c];
        Fx += sup_F[3 * s];
        Fy += sup_F[3 * s + 1];
        Fz += sup_F[3 * s + 2];
    }
    const R rho = R(1) + r;
    const R ir = R(1) / rho;
    const R ux = (j0 - R(0.5) * Fx) * ir, uy = (j1 - R(0.5) * Fy) * ir, uz = (j2 - R(0.5) * Fz) * ir;
    if (u32) reinterpret_cast<float4 *>(u32)[c] = make_float4(float(ux), float(uy), float(uz), float(rho));
    if (rec_only) return;
    rho_o[c] = double(rho);
    u_o[c] = double(ux);
    u_o[N + c] = double(uy);
    u_o[2 * N + c] = double(uz);
}

cudaError_t launch_macro(Ctx &c, float *u32, bool rec_only) {
    if (c.q == 27) return launch_q27_macro(c, rec_only ? (float4 *)u32 : nullptr);
    if (c.zlay) return launch_column_macro(c, rec_only ? (float4 *)u32 : nullptr);
    count_launch(c, G_STATS);
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    const int ibb = c.armed_bc == LBM_BC_IBB;
    const int ibm = c.armed_bc == LBM_BC_IBM_U || c.armed_bc == LBM_BC_IBM_B;
    switch (c.storage) {
#define MK(S) macro_kernel<S><<<nb, 256, 0, c.stream>>>(c.fA, c.flags, c.aux, c.sup_F, c.rho_f, c.u_f, u32, c.N, c.F[0], \
                                                           c.F[1], c.F[2], ibb, ibm, c.max_sites, rec_only)
    case LBM_F64: MK(LBM_F64); break;
    case LBM_F32: MK(LBM_F32); break;
    case LBM_F16S: MK(LBM_F16S); break;
    default: MK(LBM_BF16S); break;
#undef MK
    }
    return cudaGetLastError();
}

constexpr int SB = 256;     // threads per statistics block
constexpr int SNB = 1024;   // statistics blocks at most (the partial sums of each are kept)
constexpr int NP = 16;      // sums per block
constexpr int NBIN = LBM_NBINS;
// sums of a block: over the cells that carry fluid in the statistics (mass,
// momentum), over fluid and over solid cells (u.u and dissipation), fluid
// cells, u_z of fluid cells; mass and momentum of masked solid cells
enum { ST_MASS, ST_MX, ST_MY, ST_MZ, ST_KF, ST_EF, ST_KS, ST_ES, ST_NF, ST_UZ, ST_SMASS, ST_SX, ST_SY, ST_SZ };

// fixed-order block sum of NV values per thread, results in v of thread 0
template <int NV, int TB>
__device__ void sblock_sum(double v[NV], double *sh /* NV * TB / 32 */) {
#pragma unroll
    for (int k = 0; k < NV; k++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < NV; k++) sh[k * (TB / 32) + (threadIdx.x >> 5)] = v[k];
    __syncthreads();
    if (threadIdx.x == 0)
        for (int k = 0; k < NV; k++) {
            v[k] = 0.0;
            for (int w = 0; w < TB / 32; w++) v[k] += sh[k * (TB / 32) + w];
        }
}

// Replace the velocity of solid cells by the rigid-body velocity (zero
// without an owner: outside the pipe). A block takes runs of 4096 cells, 16
// flags per thread, lists the solid ones and spreads them over its threads.
// part (statistics only): the mass and momentum that the solid cells held.
// REC: the field is FP32 records; cells without an owner become zero there,
// cells of a particle get their velocity as hi + lo of two floats (the
// rigid-body velocity is FP64): hi in the record, whose density then says
// so, lo in a record of its own at u.
constexpr int MASK_RUN = SB * 16;
constexpr float MASKED = -3.402823466e38f;  // no density
template <bool REC>
__global__ void __launch_bounds__(SB) mask_kernel(float4 *rec, double *u, const double *rho, const uint8_t *flags,
                                                  const int *owner, const double *X, const double *U, const double *W,
                                                  int nx, int ny, int nz, FastDiv fdx, FastDiv fdxy, long long N,
                                                  double *part) {
    __shared__ unsigned short list[MASK_RUN];
    __shared__ int wsum[SB / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v[4] = {0, 0, 0, 0};
    for (long long c0 = (long long)blockIdx.x * MASK_RUN; c0 < N; c0 += (long long)gridDim.x * MASK_RUN) {
        const long long b = c0 + 16 * threadIdx.x;
        unsigned w[4] = {0u, 0u, 0u, 0u};
        if (b + 16 <= N) {
            const uint4 q = *(const uint4 *)(flags + b);
            w[0] = q.x;
            w[1] = q.y;
            w[2] = q.z;
            w[3] = q.w;
        } else {
            for (int k = 0; k < 16 && b + k < N; k++) w[k >> 2] |= (unsigned)flags[b + k] << (8 * (k & 3));
        }
        int n = 0;
        for (int k = 0; k < 4; k++) {
            w[k] &= 0x01010101u * FL_SOLID;
            n += __popc(w[k]);
        }
        // positions in cell order: scan over the warp, then over the warps
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int q = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += q;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        int at = inc - n, count = 0;
        for (int k = 0; k < SB / 32; k++) {
            at += k < warp ? wsum[k] : 0;
            count += wsum[k];
        }
        if (n > 0)
            for (int k = 0; k < 16; k++)
                if ((w[k >> 2] >> (8 * (k & 3))) & 1u) list[at++] = (unsigned short)(16 * threadIdx.x + k);
        __syncthreads();
        for (int i = threadIdx.x; i < count; i += SB) {
            const long long c = c0 + list[i];
            if (part) {
                if (REC) {
                    const float4 f = rec[c];
                    const double r = (double)f.w;
                    v[0] += r;
                    v[1] += r * (double)f.x;
                    v[2] += r * (double)f.y;
                    v[3] += r * (double)f.z;
                } else {
                    const double r = rho[c];
                    v[0] += r;
                    v[1] += r * u[c];
                    v[2] += r * u[N + c];
                    v[3] += r * u[2 * N + c];
                }
            }
            const int p = owner[c];
            if (REC && p == NO_OWNER) {
                rec[c] = make_float4(0.f, 0.f, 0.f, 0.f);
                continue;
            }
            double uw[3] = {0, 0, 0};
            if (p != NO_OWNER) {
                const unsigned zq = fdxy.div((unsigned)c), rem = (unsigned)c - zq * (unsigned)(nx * ny);
                const unsigned yq = fdx.div(rem);
                const int x = (int)(rem - yq * (unsigned)nx), y = (int)yq, z = (int)zq;
                const double r0 = dmimg(x - X[3 * p], nx), r1 = dmimg(y - X[3 * p + 1], ny), r2 = dmimg(z - X[3 * p + 2], nz);
                uw[0] = U[3 * p] + (W[3 * p + 1] * r2 - W[3 * p + 2] * r1);
                uw[1] = U[3 * p + 1] + (W[3 * p + 2] * r0 - W[3 * p] * r2);
                uw[2] = U[3 * p + 2] + (W[3 * p] * r1 - W[3 * p + 1] * r0);
            }
            if (REC) {
                const float2 v0 = pair_of(uw[0]), v1 = pair_of(uw[1]), v2 = pair_of(uw[2]);
                rec[c] = make_float4(v0.x, v1.x, v2.x, MASKED);
                ((float4 *)u)[c] = make_float4(v0.y, v1.y, v2.y, 0.f);
            } else {
                u[c] = uw[0];
                u[N + c] = uw[1];
                u[2 * N + c] = uw[2];
            }
        }
        __syncthreads();
    }
    if (!part) return;
    __shared__ double sh[4 * (SB / 32)];
    sblock_sum<4, SB>(v, sh);
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; k++) part[blockIdx.x * NP + ST_SMASS + k] = v[k];
}

// Nearest particle surface of the fluid cells with 0 < s <= reach, s = r -
// R_p (reach: the farthest distance a caller needs, the closure's 2 or the
// last radial bin), in one pass: the 64-bit key of a cell holds the bits
// of s (positive, so ordered as integers) with its low NEAR_PID_BITS bits
// replaced by the particle id, and atomicMin keeps the nearest. Particles
// whose s agree in the upper 44 bits (2^-44 relative) count as tied, and
// the lower id wins. Every particle that could be the nearest of such a
// cell has it in its box, so the minimum is over all of them; cells
// farther out keep the empty key. s is formed in FP32 from the split centre
// (integer part exact, FP32 fraction: error about 1e-6 lu), and in exact
// FP64 where it lies within 1e-4 of 0 or of reach, so every cell's
// membership (0 < s <= reach) is that of the FP64 distance; s itself, the
// order of two particles within 1e-6 of each other and the distance
// feature carry the FP32 error. The closure's own threshold (2) is decided
// the same way when the bins reach farther.
constexpr int NEAR_PID_BITS = 20;
constexpr unsigned long long NEAR_PID_MASK = (1ULL << NEAR_PID_BITS) - 1;
constexpr unsigned long long NEAR_EMPTY = ~0ULL;
__device__ __forceinline__ int near_pid_of(unsigned long long k) { return (int)(k & NEAR_PID_MASK); }
__device__ __forceinline__ double near_s_of(unsigned long long k) {
    return __longlong_as_double((long long)(k & ~NEAR_PID_MASK));
}

__global__ void near_key_kernel(unsigned long long *key, const uint8_t *flags, const double *X, const double *R,
                                int nx, int ny, int nz, double reach) {
    const int p = blockIdx.x;
    const double Rp = R[p];
    const int r = (int)ceil(Rp + reach) + 2;
    const double Xd = X[3 * p], Yd = X[3 * p + 1], Zd = X[3 * p + 2];
    const int bx = (int)floor(Xd) - r, by = (int)floor(Yd) - r, bz = (int)floor(Zd) - r;
    const int w = 2 * r + 2;
    const FastDiv fw((unsigned)w);
    // the centre relative to the box corner: integer part exact, fraction in FP32
    const float fX0 = (float)(Xd - bx), fX1 = (float)(Yd - by), fX2 = (float)(Zd - bz);
    const float Rf = (float)Rp, reachf = (float)reach;
    const float lo = fmaxf(Rf - 2e-3f, 0.f), hi = Rf + reachf + 2e-3f, lo2 = lo * lo, hi2 = hi * hi;
    for (int t = threadIdx.x; t < w * w * w; t += blockDim.x) {
        int ix, iy, iz;
        box_coords(t, fw, w, ix, iy, iz);
        const float ex = ix - fX0, ey = iy - fX1, ez = iz - fX2, e2 = ex * ex + ey * ey + ez * ez;
        if (e2 > hi2 || e2 < lo2) continue;
        const int x = dwrap(bx + ix, nx), y = dwrap(by + iy, ny),
                  z = dwrap(bz + iz, nz);
        const long long c = (long long)x + (long long)nx * (y + (long long)ny * z);
        if (flags[c] & FL_SOLID) continue;
        const float s32 = sqrtf(e2) - Rf;
        double sd;
        if (s32 < 1e-4f || fabsf(s32 - reachf) < 1e-4f || fabsf(s32 - 2.0f) < 1e-4f) {  // 2: the closure's band
            const double dx = dmimg(__dsub_rn((double)x, Xd), nx);
            const double dy = dmimg(__dsub_rn((double)y, Yd), ny);
            const double dz = dmimg(__dsub_rn((double)z, Zd), nz);
            const double rr = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
            sd = __dsub_rn(rr, Rp);
        } else {
            sd = (double)s32;
        }
        if (sd <= 0.0 || sd > reach) continue;
        const unsigned long long k = ((unsigned long long)__double_as_longlong(sd) & ~NEAR_PID_MASK) | (unsigned)p;
        atomicMin(key + c, k);
    }
}

// one counter increment per warp for the lanes with `take`; returns this lane's slot
__device__ __forceinline__ long long warp_slot(bool take, long long *count) {
    const unsigned m = __ballot_sync(__activemask(), take);
    if (!take) return -1;
    const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
    unsigned long long base = 0;
    if (lane == leader) base = atomicAdd((unsigned long long *)count, (unsigned long long)__popc(m));
    base = __shfl_sync(m, base, leader);
    return (long long)base + __popc(m & ((1u << lane) - 1u));
}

// The sums of lbm_stats in one pass over the cells.
//
// What bounds it: FP64 storage, the FP64 pipe (two multiply-adds per clock
// and SM; about 31 operations per cell). 32- and 16-bit storage have FP32
// fields, so there the differences are exact as pairs of floats and sums and
// squares are carried as such pairs (about 48 bits, see pair_add): some 250
// FP32 operations in place of 45 FP64 issues of 16 clocks each (cells with a
// masked particle cell among their neighbours add its low part), and every
// 64 planes the pairs go into FP64 sums.
// A thread takes a column (x, y) over a run of z: every velocity is loaded
// once along z, s_ij s_ij comes from undivided differences, no division. The
// radial bins are private to the thread (shared memory, [bin][thread]: no
// atomics, no bank conflicts); FP64 atomics on 40 shared bins per block,
// contended by the lanes of a warp, were most of the former bins pass. The
// bin index is decided in FP32 from the distance in the cell's key (20 bits
// of mantissa) away from the bin edges and by the exact FP64 quotient near
// one. A plane's loads are issued one plane ahead: only 8 warps per SM
// fit beside the bins.
// 256^3, 2000 spheres, FP32, with bins: 0.7 ms in place of 1.57 (energies) +
// 2.9 (bins); 1.74 ms in FP64, 1.12 without the loads ahead.
constexpr int ST_TB = 128;   // threads: 32 x 4 columns
constexpr int ST_RUN = 64;   // planes per tile

struct StatsArgs {
    const double *u, *rho;  // FP64 fields
    const float4 *rec, *low;  // or FP32 records, and the low parts of masked particle cells' velocities
    const uint8_t *flags;
    const unsigned long long *near_key;
    const double *X, *R;
    float bins_per_unit;  // 1 / (0.05 R) where all particles have one radius, else 0
    float bin_slack;      // how far a bin coordinate may be off, per unit of 1 / (0.05 R), beside 1e-4
    const float *eps_o;  // dissipation from the closure where >= 0, or null
    int nx, ny, nz;
    long long N;
    double nu;
    int pipe, ibb, raw;  // raw: solid cells hold the virtual fluid (no mask) and count in mass and momentum
    double *part, *bpart;
};

// radial bin of a fluid cell from its nearest particle's key, or -1
__device__ __forceinline__ int radial_bin(const StatsArgs &a, unsigned long long key, int x, int y, int z) {
    if (key == NEAR_EMPTY) return -1;
    const int p = near_pid_of(key);
    // the key's distance s with the upper 20 bits of its mantissa
    const unsigned hi = (unsigned)(key >> 32);
    const float s = __uint_as_float((((hi >> 20) - 896u) << 23) | ((hi & 0xfffffu) << 3));
    const float k = a.bins_per_unit > 0.f ? a.bins_per_unit : 20.0f / (float)a.R[p], tb = s * k;  // (r / R - 1) / 0.05
    int b = (int)tb;
    // The key's s carries the FP32 centre of near_key_kernel, rounded at the
    // half width of its box (less than reach + R + 4, R the particle's own),
    // at most 1.8 (reach + R + 4) 2^-24, and the rounding of distances up to
    // 3 R, 14 R 2^-24 with the root; k s that of the 20 bits, 4e-5, and two
    // products. With R = 20 / k: 1.1e-7 (reach + 4) k + 7e-5. A box made for a
    // large particle's reach is coarse for the bins of a small one.
    if (fabsf(tb - rintf(tb)) < 2e-4f + a.bin_slack * k) {
        const double dx = dmimg(__dsub_rn((double)x, a.X[3 * p]), a.nx);
        const double dy = dmimg(__dsub_rn((double)y, a.X[3 * p + 1]), a.ny);
        const double dz = dmimg(__dsub_rn((double)z, a.X[3 * p + 2]), a.nz);
        const double rr = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
        b = (int)floor(__ddiv_rn(__dsub_rn(__ddiv_rn(rr, a.R[p]), 1.0), 0.05));
    }
    return b >= 0 && b < NBIN ? b : -1;
}

// sum of D_aa^2 plus half the sum over a < b of (D_ab + D_ba)^2: 4 s_ij s_ij
__device__ __forceinline__ double strain4(const double D[3][3]) {
    const double sd = fma(D[0][0], D[0][0], fma(D[1][1], D[1][1], D[2][2] * D[2][2]));
    const double sxy = D[0][1] + D[1][0], sxz = D[0][2] + D[2][0], syz = D[1][2] + D[2][1];
    return fma(0.5, fma(sxy, sxy, fma(sxz, sxz, syz * syz)), sd);
}

// What a column's march gives per cell, as FP64 (V = double) or pairs (V = float2)
template <typename V> struct Sums;
template <> struct Sums<double> {
    static __device__ __forceinline__ double zero() { return 0.0; }
    static __device__ __forceinline__ double add(double a, double b) { return a + b; }
    static __device__ __forceinline__ double mul_add(double r, double w, double s) { return fma(r, w, s); }
    static __device__ __forceinline__ double of(double v) { return v; }
    static __device__ __forceinline__ double value(double v) { return v; }
};
template <> struct Sums<float2> {
    static __device__ __forceinline__ float2 zero() { return make_float2(0.f, 0.f); }
    static __device__ __forceinline__ float2 add(float2 a, float2 b) { return pair_add(a, b); }
    static __device__ __forceinline__ float2 mul_add(float r, float w, float2 s) { return pair_add(s, pair_mul(r, w)); }
    static __device__ __forceinline__ float2 of(double v) { return pair_of(v); }
    static __device__ __forceinline__ double value(float2 v) { return pair_value(v); }
};

template <bool BINS, typename V>
__global__ void __launch_bounds__(ST_TB) stats_kernel(StatsArgs a) {
    constexpr bool REC = sizeof(V) == 8 && !std::is_same<V, double>::value;
    typedef Sums<V> M;
    extern __shared__ double acc_raw[];  // BINS: u.u and 4 s_ij s_ij, [2][NBIN][ST_TB], then NBIN counts
    V *acc = reinterpret_cast<V *>(acc_raw);
    int *cnt = (int *)(acc + 2 * NBIN * ST_TB);
    const int t = threadIdx.x;
    if (BINS) {
        for (int i = t; i < 2 * NBIN * ST_TB; i += ST_TB) acc[i] = M::zero();
        for (int i = t; i < NBIN; i += ST_TB) cnt[i] = 0;
        __syncthreads();
    }
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const long long N = a.N, nxy = (long long)nx * ny;
    const long long ntx = (nx + 31) / 32, nty = (ny + 3) / 4, ntz = (nz + ST_RUN - 1) / ST_RUN;
    const double to_eps = 0.5 * a.nu, from_eps = 1.0 / to_eps;  // 2 nu s_ij s_ij = (nu / 2) 4 s_ij s_ij
    double v[10];
    for (int k = 0; k < 10; k++) v[k] = 0.0;
    int nf = 0;
    for (long long tile = blockIdx.x; tile < ntx * nty * ntz; tile += gridDim.x) {
        const int x = (int)(tile % ntx) * 32 + (t & 31), y = (int)((tile / ntx) % nty) * 4 + (t >> 5);
        if (x >= nx || y >= ny) continue;
        const int z0 = (int)(tile / (ntx * nty)) * ST_RUN, z1 = min(nz, z0 + ST_RUN), zb = z0 == 0 ? nz - 1 : z0 - 1;
        const long long c = x + (long long)nx * y;
        const int oxm = x == 0 ? nx - 1 : -1, oxp = x == nx - 1 ? 1 - nx : 1;
        const long long oym = y == 0 ? (long long)nx * (ny - 1) : -nx, oyp = y == ny - 1 ? -(long long)nx * (ny - 1) : nx;
        const double *u = a.u + c;
        const float4 *rec = a.rec + c, *lo = a.low + c;
        double um[3], uc[3];
        float4 fm = make_float4(0.f, 0.f, 0.f, 0.f), fc = fm;
        if constexpr (REC) {
            fm = rec[nxy * zb];
            fc = rec[nxy * z0];
        } else {
            for (int d = 0; d < 3; d++) {
                um[d] = u[d * N + nxy * zb];
                uc[d] = u[d * N + nxy * z0];
            }
        }
        V s[8];
        for (int k = 0; k < 8; k++) s[k] = M::zero();
        V suz = M::zero();
        // the loads of a plane are issued one plane ahead (few warps fit beside the bins)
        float4 nb[5];
        unsigned char nfl;
        float neo = -1.f;
        unsigned long long nkey = NEAR_EMPTY;
        auto fetch = [&](int z) {
            const long long e = nxy * z;
            if constexpr (REC) {
                nb[0] = rec[e + oxp];
                nb[1] = rec[e + oxm];
                nb[2] = rec[e + oyp];
                nb[3] = rec[e + oym];
                nb[4] = rec[z == nz - 1 ? 0 : e + nxy];
            }
            nfl = a.flags[c + e];
            if (a.eps_o) neo = a.eps_o[c + e];
            if (BINS) nkey = a.near_key[c + e];
        };
        fetch(z0);
        for (int z = z0; z < z1; z++) {
            const long long e = nxy * z, ep = z == nz - 1 ? 0 : e + nxy, em = z == 0 ? nxy * (nz - 1) : e - nxy;
            const bool solid = nfl & FL_SOLID;
            const float eo = neo;
            const unsigned long long key = nkey;
            const float4 xp = nb[0], xm = nb[1], yp = nb[2], ym = nb[3], zp = nb[4];
            if (z + 1 < z1) fetch(z + 1);
            V kk, ss;  // u.u, 4 s_ij s_ij
            if constexpr (REC) {
                if (fminf(fminf(fminf(xp.w, xm.w), fminf(yp.w, ym.w)), fminf(fminf(zp.w, fm.w), fc.w)) == MASKED) {
                    // a masked particle cell among them: its velocity has a low part
                    auto low = [&](const float4 &f, long long o) -> float4 {
                        return f.w == MASKED ? lo[o] : make_float4(0.f, 0.f, 0.f, 0.f);
                    };
                    const float4 lxp = low(xp, e + oxp), lxm = low(xm, e + oxm), lyp = low(yp, e + oyp),
                                 lym = low(ym, e + oym), lzp = low(zp, ep), lzm = low(fm, em), lc = low(fc, e);
                    auto diff = [](float a, float b, float la, float lb) -> float2 {
                        return pair_add(pair_diff(a, b), make_float2(la - lb, 0.f));
                    };
                    kk = pair_add(pair_add(pair_square(make_float2(fc.x, lc.x)), pair_square(make_float2(fc.y, lc.y))),
                                  pair_square(make_float2(fc.z, lc.z)));
                    const float2 sxy = pair_add(diff(yp.x, ym.x, lyp.x, lym.x), diff(xp.y, xm.y, lxp.y, lxm.y)),
                                 sxz = pair_add(diff(zp.x, fm.x, lzp.x, lzm.x), diff(xp.z, xm.z, lxp.z, lxm.z)),
                                 syz = pair_add(diff(zp.y, fm.y, lzp.y, lzm.y), diff(yp.z, ym.z, lyp.z, lym.z));
                    const float2 off = pair_add(pair_add(pair_square(sxy), pair_square(sxz)), pair_square(syz));
                    ss = pair_add(pair_add(pair_square(diff(xp.x, xm.x, lxp.x, lxm.x)),
                                           pair_square(diff(yp.y, ym.y, lyp.y, lym.y))),
                                  pair_add(pair_square(diff(zp.z, fm.z, lzp.z, lzm.z)),
                                           make_float2(0.5f * off.x, 0.5f * off.y)));
                } else {
                    kk = pair_add(pair_add(pair_mul(fc.x, fc.x), pair_mul(fc.y, fc.y)), pair_mul(fc.z, fc.z));
                    const float2 sxy = pair_add(pair_diff(yp.x, ym.x), pair_diff(xp.y, xm.y)),
                                 sxz = pair_add(pair_diff(zp.x, fm.x), pair_diff(xp.z, xm.z)),
                                 syz = pair_add(pair_diff(zp.y, fm.y), pair_diff(yp.z, ym.z));
                    const float2 off = pair_add(pair_add(pair_square(sxy), pair_square(sxz)), pair_square(syz));
                    ss = pair_add(pair_add(pair_square(pair_diff(xp.x, xm.x)), pair_square(pair_diff(yp.y, ym.y))),
                                  pair_add(pair_square(pair_diff(zp.z, fm.z)), make_float2(0.5f * off.x, 0.5f * off.y)));
                }
                fm = fc;
                fc = zp;
            } else {
                double D[3][3], w[3];  // differences: twice the gradients
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    const double *ud = u + d * N;
                    const double up = ud[ep];
                    D[d][0] = ud[e + oxp] - ud[e + oxm];
                    D[d][1] = ud[e + oyp] - ud[e + oym];
                    D[d][2] = up - um[d];
                    w[d] = uc[d];
                    um[d] = uc[d];
                    uc[d] = up;
                }
                kk = fma(w[0], w[0], fma(w[1], w[1], w[2] * w[2]));
                ss = strain4(D);
            }
            if (eo >= 0.f) ss = M::of((double)eo * from_eps);
            if (solid) {
                s[ST_KS] = M::add(s[ST_KS], kk);
                s[ST_ES] = M::add(s[ST_ES], ss);
                if (!a.raw) continue;
            }
            if (!solid || (a.raw && !a.ibb)) {
                if constexpr (REC) {  // fm: this cell now
                    s[ST_MASS] = M::add(s[ST_MASS], make_float2(fm.w, 0.f));
                    s[ST_MX] = M::mul_add(fm.w, fm.x, s[ST_MX]);
                    s[ST_MY] = M::mul_add(fm.w, fm.y, s[ST_MY]);
                    s[ST_MZ] = M::mul_add(fm.w, fm.z, s[ST_MZ]);
                } else {
                    const double r = a.rho[c + e];
                    s[ST_MASS] = M::add(s[ST_MASS], r);
                    s[ST_MX] = M::mul_add(r, um[0], s[ST_MX]);
                    s[ST_MY] = M::mul_add(r, um[1], s[ST_MY]);
                    s[ST_MZ] = M::mul_add(r, um[2], s[ST_MZ]);
                }
            }
            if (solid) continue;
            s[ST_KF] = M::add(s[ST_KF], kk);
            s[ST_EF] = M::add(s[ST_EF], ss);
            nf++;
            if (a.pipe) {
                if constexpr (REC) suz = M::add(suz, make_float2(fm.z, 0.f));
                else suz = M::add(suz, um[2]);
            }
            if (BINS) {
                const int b = radial_bin(a, key, x, y, z);
                if (b < 0) continue;
                acc[b * ST_TB + t] = M::add(acc[b * ST_TB + t], kk);
                acc[(NBIN + b) * ST_TB + t] = M::add(acc[(NBIN + b) * ST_TB + t], ss);
                atomicAdd(cnt + b, 1);
            }
        }
        for (int k = 0; k < 8; k++) v[k] += M::value(s[k]);
        v[ST_UZ] += M::value(suz);
    }
    v[ST_NF] = (double)nf;
    v[ST_EF] *= to_eps;
    v[ST_ES] *= to_eps;
    __shared__ double sh[10 * (ST_TB / 32)];
    sblock_sum<10, ST_TB>(v, sh);
    if (t == 0)
        for (int k = 0; k < 10; k++) a.part[blockIdx.x * NP + k] = v[k];
    if (BINS) {
        __syncthreads();
        // one warp per bin and quantity in turn: fixed order
        for (int i = t >> 5; i < 2 * NBIN; i += ST_TB / 32) {
            double q = 0.0;
            for (int k = t & 31; k < ST_TB; k += 32) q += M::value(acc[i * ST_TB + k]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
            if ((t & 31) == 0) a.bpart[blockIdx.x * 3 * NBIN + i] = i < NBIN ? q : q * to_eps;
        }
        for (int i = t; i < NBIN; i += ST_TB) a.bpart[blockIdx.x * 3 * NBIN + 2 * NBIN + i] = (double)cnt[i];
    }
}

// the blocks' sums added in a fixed order: column blockIdx.x of nblk rows
__global__ void __launch_bounds__(SB) stats_reduce_kernel(const double *part, const double *bpart, int nblk, int mblk,
                                                          double *out) {
    const int k = blockIdx.x;
    double v[1] = {0.0};
    if (k < NP) {
        const int n = k >= ST_SMASS ? mblk : nblk;
        for (int b = threadIdx.x; b < n; b += SB) v[0] += part[(size_t)b * NP + k];
    } else {
        for (int b = threadIdx.x; b < nblk; b += SB) v[0] += bpart[(size_t)b * 3 * NBIN + (k - NP)];
    }
    __shared__ double sh[SB / 32];
    sblock_sum<1, SB>(v, sh);
    if (threadIdx.x == 0) out[k] = v[0];
}

__global__ void fill_u64(unsigned long long *p, unsigned long long v, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// ------------------------------------------------------ learned closure --
// Near-surface fluid nodes (distance to the nearest particle surface in
// (0, 2]) and their 85 features: the 27-point stencil of u - u_rb (u_rb the
// rigid-body velocity of the nearest particle), scaled by 1/u_scale, the
// signed distance / h, and u - u_rb at the node.
__global__ void closure_sample_kernel(const double *u, const uint8_t *flags, const unsigned long long *near_key,
                                      const double *X, const double *U, const double *W, int nx, int ny, int nz,
                                      long long N, double inv_us, float *feat, int *cells, long long *count,
                                      long long cap) {
    // whole warps per round (the slot counter is taken once per warp)
    const long long span = (long long)gridDim.x * blockDim.x;
    for (long long c0 = (long long)blockIdx.x * blockDim.x; c0 < N; c0 += span) {
        const long long c = c0 + threadIdx.x;
        const unsigned long long key = c < N && !(flags[c] & FL_SOLID) ? near_key[c] : NEAR_EMPTY;
        const double d = near_s_of(key);  // r - R_p of the nearest particle
        const bool take = key != NEAR_EMPTY && d > 0.0 && d <= 2.0;
        const long long k = warp_slot(take, count);
        if (!take || k >= cap) continue;
        const int p = near_pid_of(key);
        const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / ((long long)nx * ny));
        const double rx = dmimg(x - X[3 * p], nx), ry = dmimg(y - X[3 * p + 1], ny), rz = dmimg(z - X[3 * p + 2], nz);
        cells[k] = (int)c;
        float *f = feat + k * 85;
        int j = 0;
        for (int dz = -1; dz <= 1; dz++)
            for (int dy = -1; dy <= 1; dy++)
                for (int dx = -1; dx <= 1; dx++) {
                    const long long q = (long long)dwrap(x + dx, nx) + (long long)nx * (dwrap(y + dy, ny) + (long long)ny * dwrap(z + dz, nz));
                    const double sx = rx + dx, sy = ry + dy, sz = rz + dz;
                    const double ub0 = U[3 * p] + (W[3 * p + 1] * sz - W[3 * p + 2] * sy);
                    const double ub1 = U[3 * p + 1] + (W[3 * p + 2] * sx - W[3 * p] * sz);
                    const double ub2 = U[3 * p + 2] + (W[3 * p] * sy - W[3 * p + 1] * sx);
                    f[j++] = (float)((u[q] - ub0) * inv_us);
                    f[j++] = (float)((u[N + q] - ub1) * inv_us);
                    f[j++] = (float)((u[2 * N + q] - ub2) * inv_us);
                }
        f[81] = (float)d;
        f[82] = f[3 * 13];
        f[83] = f[3 * 13 + 1];
        f[84] = f[3 * 13 + 2];
    }
}

// 9 velocity gradients du_a/dx_b (central differences) at listed cells,
// scaled by g_scale; NaN where the cell is solid in this state
__global__ void closure_target_kernel(const double *u, const uint8_t *flags, const int *cells, long long n, int nx,
                                      int ny, int nz, long long N, double gs, float *T) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const long long c = cells[k];
    float *t = T + k * 9;
    if (flags[c] & FL_SOLID) {
        for (int e = 0; e < 9; e++) t[e] = __int_as_float(0x7fc00000);
        return;
    }
    const int x = (int)(c % nx), y = (int)((c / nx) % ny), z = (int)(c / ((long long)nx * ny));
    const long long nb[3][2] = {{dwrap(x + 1, nx) + (long long)nx * (y + (long long)ny * z), dwrap(x - 1, nx) + (long long)nx * (y + (long long)ny * z)},
                                {x + (long long)nx * (dwrap(y + 1, ny) + (long long)ny * z), x + (long long)nx * (dwrap(y - 1, ny) + (long long)ny * z)},
                                {x + (long long)nx * (y + (long long)ny * dwrap(z + 1, nz)), x + (long long)nx * (y + (long long)ny * dwrap(z - 1, nz))}};
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) t[3 * a + b] = (float)(0.5 * (u[a * N + nb[b][0]] - u[a * N + nb[b][1]]) * gs);
}

// the near-surface fluid nodes of the fused closure dissipation: cell and
// nearest particle (distance to the surface in (0, 2]); order not fixed
// One slot range per block and 1024 consecutive cells, filled in cell
// order, so that neighbouring samples of the list are mostly neighbouring
// cells (their stencils share lines in the inference kernel's gather).
// (four cells per thread: 119 us per call at 256^3 with one)
__global__ void __launch_bounds__(256) closure_list_kernel(const uint8_t *flags, const unsigned long long *near_key,
                                                           long long N, int *cells, int *pids, long long *count,
                                                           long long cap) {
    __shared__ unsigned wcnt[8];
    __shared__ unsigned long long base;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long c = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
    unsigned long long key[4] = {NEAR_EMPTY, NEAR_EMPTY, NEAR_EMPTY, NEAR_EMPTY};
    if (c + 4 <= N) {
        const ulonglong2 k0 = *(const ulonglong2 *)(near_key + c), k1 = *(const ulonglong2 *)(near_key + c + 2);
        key[0] = k0.x;
        key[1] = k0.y;
        key[2] = k1.x;
        key[3] = k1.y;
    } else {
        for (int k = 0; k < 4; k++)
            if (c + k < N) key[k] = near_key[c + k];
    }
    unsigned take = 0;
    for (int k = 0; k < 4; k++) {
        if (key[k] == NEAR_EMPTY || (flags[c + k] & FL_SOLID)) continue;
        const double d = near_s_of(key[k]);  // r - R_p of the nearest particle
        if (d > 0.0 && d <= 2.0) take |= 1u << k;
    }
    const unsigned n = __popc(take);
    unsigned inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned q = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += q;
    }
    if (lane == 31) wcnt[warp] = inc;
    __syncthreads();
    unsigned before = inc - n, total = 0;
    for (int w = 0; w < 8; w++) {
        before += w < warp ? wcnt[w] : 0u;
        total += wcnt[w];
    }
    if (threadIdx.x == 0) base = total ? atomicAdd((unsigned long long *)count, (unsigned long long)total) : 0ull;
    __syncthreads();
    long long at = (long long)base + before;
    for (int k = 0; k < 4; k++) {
        if (!((take >> k) & 1u)) continue;
        if (at < cap) {
            cells[at] = (int)(c + k);
            pids[at] = near_pid_of(key[k]);
        }
        at++;
    }
}

// dissipation 2 nu s_ij s_ij from predicted gradients (scaled by g_scale)
__global__ void closure_eps_kernel(const float *Y, const int *cells, long long n, double inv_gs, double nu,
                                   float *eps_o) {
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double g[3][3];
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) g[a][b] = (double)Y[k * 9 + 3 * a + b] * inv_gs;
    double ss = 0.0;
    for (int a = 0; a < 3; a++)
        for (int b = 0; b < 3; b++) {
            const double sab = 0.5 * (g[a][b] + g[b][a]);
            ss += sab * sab;
        }
    eps_o[cells[k]] = (float)(2.0 * nu * ss);
}

__global__ void fill_f32(float *p, float v, long long n) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}


static int mask_blocks(const Ctx &c) { return (int)std::min<long long>(SNB, (c.N + MASK_RUN - 1) / MASK_RUN); }
static cudaError_t mask_cells(Ctx &c, double *part, float4 *rec = nullptr) {
    if (c.np == 0 && !c.has_pipe) return cudaSuccess;  // no solid cell
    const FastDiv fdx((unsigned)c.nx), fdxy((unsigned)(c.nx * c.ny));
    if (rec)
        mask_kernel<true><<<mask_blocks(c), SB, 0, c.stream>>>(rec, (double *)(rec + c.N), nullptr, c.flags, c.owner, c.X,
                                                               c.U, c.W, c.nx, c.ny, c.nz, fdx, fdxy, c.N, part);
    else
        mask_kernel<false><<<mask_blocks(c), SB, 0, c.stream>>>(nullptr, c.u_f, c.rho_f, c.flags, c.owner, c.X, c.U, c.W,
                                                                c.nx, c.ny, c.nz, fdx, fdxy, c.N, part);
    return cudaGetLastError();
}

// nearest particle and distance to its surface of the fluid cells within
// `reach` of a surface (key and pid; others NO_OWNER)
static void near_surface(Ctx &c, const unsigned nb, double reach) {
    count_launch(c, G_STATS, 2);
    fill_u64<<<nb, 256, 0, c.stream>>>(c.near_key, NEAR_EMPTY, c.N);
    near_key_kernel<<<c.np, 256, 0, c.stream>>>(c.near_key, c.flags, c.X, c.R, c.nx, c.ny, c.nz, reach);
}

cudaError_t closure_samples(Ctx &c, double u_scale, float *X, int *cells, long long cap, long long *n_out) {
    cudaError_t e;
    if ((e = launch_macro(c)) != cudaSuccess) return e;
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    near_surface(c, nb, 2.0);
    count_launch(c, G_STATS);
    if ((e = cudaMemsetAsync(c.d_counts + 3, 0, sizeof(long long), c.stream)) != cudaSuccess) return e;
    closure_sample_kernel<<<nb, 256, 0, c.stream>>>(c.u_f, c.flags, c.near_key, c.X, c.U, c.W, c.nx, c.ny, c.nz,
                                                    c.N, 1.0 / u_scale, X, cells, c.d_counts + 3, cap);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    long long n = 0;
    if ((e = cudaMemcpyAsync(&n, c.d_counts + 3, sizeof(long long), cudaMemcpyDeviceToHost, c.stream)) != cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(c.stream)) != cudaSuccess) return e;
    *n_out = n;
    return cudaSuccess;
}

cudaError_t closure_targets(Ctx &c, const int *cells, long long n, double g_scale, float *T) {
    cudaError_t e;
    if ((e = launch_macro(c)) != cudaSuccess) return e;
    count_launch(c, G_STATS, 2);
    if ((e = mask_cells(c, nullptr)) != cudaSuccess) return e;
    if (n > 0)
        closure_target_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c.stream>>>(c.u_f, c.flags, cells, n, c.nx, c.ny,
                                                                              c.nz, c.N, g_scale, T);
    return cudaGetLastError();
}

// ------------------------------------------------ pipe radial profiles ----
// Per radial bin b = floor(r nbins / R) of the cells inside the pipe, the
// sums of 1, u_r, u_theta, u_z, their products, rho and 2 nu s_ij s_ij
// (statistics velocity, central differences).
//
// What bounds it: the FP64 pipe. A thread takes a column (x, y), whose basis
// and bin are the same in every plane, over a run of z and keeps the 11 sums
// in registers (about 35 FP64 operations per cell, no division); the columns'
// sums go to one of PROF_REP copies of the bins with global FP64 reductions,
// and the copies are added in order. With every cell adding to shared-memory
// bins a call on the benchmark pipe (7.34 M cells, 64 bins) took 2.9 ms, now
// 0.8 (this kernel 0.57).
constexpr int PROF_NQ = LBM_PROF_NQ;
constexpr int PROF_REP = 32;

__global__ void __launch_bounds__(SB) pipe_profile_kernel(const double *u, const double *rho, const uint8_t *flags,
                                                         int nx, int ny, int nz, long long N, double cx, double cy,
                                                         double R, int nbins, int run, double nu, double *part) {
    int x, y;
    column_of_thread(nx, x, y);
    PipeColumn k;
    if (!pipe_column(flags, x, y, nx, ny, cx, cy, R, nbins, k)) return;
    const double ca = k.ca, sa = k.sa;
    const long long nxy = (long long)nx * ny;
    const int c = x + nx * y;
    const int oxm = x == 0 ? nx - 1 : -1, oxp = x == nx - 1 ? 1 - nx : 1;
    const int oym = y == 0 ? nx * (ny - 1) : -nx, oyp = y == ny - 1 ? -nx * (ny - 1) : nx;
    const int z0 = blockIdx.y * run, z1 = min(nz, z0 + run), zb = z0 == 0 ? nz - 1 : z0 - 1;
    u += c;
    rho += c;
    double um[3], uc[3], s[10], sd = 0.0, so = 0.0;
    for (int d = 0; d < 3; d++) {
        um[d] = u[d * N + nxy * zb];
        uc[d] = u[d * N + nxy * z0];
    }
    for (int q = 0; q < 10; q++) s[q] = 0.0;
    for (int z = z0; z < z1; z++) {
        const long long e = nxy * z, ep = z == nz - 1 ? 0 : e + nxy;
        double D[3][3], v[3];  // differences: twice the gradients
#pragma unroll
        for (int d = 0; d < 3; d++) {
            const double *ud = u + d * N;
            const double up = ud[ep];
            D[d][0] = ud[e + oxp] - ud[e + oxm];
            D[d][1] = ud[e + oyp] - ud[e + oym];
            D[d][2] = up - um[d];
            v[d] = uc[d];
            um[d] = uc[d];
            uc[d] = up;
        }
        const double ur = ca * v[0] + sa * v[1], ut = ca * v[1] - sa * v[0], uz = v[2];
        s[0] += ur;
        s[1] += ut;
        s[2] += uz;
        s[3] = fma(ur, ur, s[3]);
        s[4] = fma(ut, ut, s[4]);
        s[5] = fma(uz, uz, s[5]);
        s[6] = fma(ur, uz, s[6]);
        s[7] = fma(ur, ut, s[7]);
        s[8] = fma(ut, uz, s[8]);
        s[9] += rho[e];
        // s_ij s_ij = (sum of D_aa^2) / 4 + (sum over a < b of (D_ab + D_ba)^2) / 8
        sd = fma(D[0][0], D[0][0], fma(D[1][1], D[1][1], fma(D[2][2], D[2][2], sd)));
        const double sxy = D[0][1] + D[1][0], sxz = D[0][2] + D[2][0], syz = D[1][2] + D[2][1];
        so = fma(sxy, sxy, fma(sxz, sxz, fma(syz, syz, so)));
    }
    double *row = part + ((size_t)((blockIdx.x + gridDim.x * blockIdx.y) % PROF_REP) * nbins + k.bin) * PROF_NQ;
    atomicAdd(row, (double)(z1 - z0));
    for (int q = 0; q < 10; q++) atomicAdd(row + 1 + q, s[q]);
    atomicAdd(row + 11, 2.0 * nu * (0.25 * sd + 0.125 * so));
}

// the copies added in order; sums over the bin's count
__global__ void profile_bins_kernel(const double *part, double *out, int nbins) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nbins * PROF_NQ) return;
    const int b = i / PROF_NQ, q = i - b * PROF_NQ;
    double s = 0.0, n = 0.0;
    for (int r = 0; r < PROF_REP; r++) {
        s += part[(size_t)r * nbins * PROF_NQ + i];
        n += part[((size_t)r * nbins + b) * PROF_NQ];
    }
    out[i] = q == 0 ? s : (n > 0.0 ? s / n : 0.0);
}

// what the call asks of the idle population buffer (a limit of the ABI; the
// bins and their copies need PROF_REP + 1 sets)
size_t pipe_profile_scratch_bytes(int nbins) { return sizeof(double) * (size_t)304 * nbins * PROF_NQ; }

// scratch: the population buffer that the next step overwrites
cudaError_t run_pipe_profiles(Ctx &c, int flags, int nbins, double *out) {
    cudaError_t e;
    if ((e = launch_macro(c)) != cudaSuccess) return e;
    const int ibm = c.armed_bc == LBM_BC_IBM_U || c.armed_bc == LBM_BC_IBM_B;
    if (!(ibm && (flags & LBM_STATS_UNMASK)))
        if ((e = launch_mask(c)) != cudaSuccess) return e;
    const size_t set = (size_t)nbins * PROF_NQ;
    double *part = (double *)c.fB, *res = part + PROF_REP * set;
    const double nu = (c.tau - 0.5) / 3.0;
    const int run = column_run(c.nz);
    count_launch(c, G_STATS, 2);
    if ((e = cudaMemsetAsync(part, 0, sizeof(double) * PROF_REP * set, c.stream)) != cudaSuccess) return e;
    pipe_profile_kernel<<<column_blocks(c.nx, c.ny, c.nz, run), SB, 0, c.stream>>>(
        c.u_f, c.rho_f, c.flags, c.nx, c.ny, c.nz, c.N, c.pipe_cx, c.pipe_cy, c.pipe_R, nbins, run, nu, part);
    profile_bins_kernel<<<(unsigned)((set + 255) / 256), 256, 0, c.stream>>>(part, res, nbins);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    std::vector<double> hp(set);
    if ((e = cudaMemcpyAsync(hp.data(), res, sizeof(double) * set, cudaMemcpyDeviceToHost, c.stream)) != cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(c.stream)) != cudaSuccess) return e;
    std::copy(hp.begin(), hp.end(), out);
    return cudaSuccess;
}

cudaError_t launch_mask(Ctx &c) {
    // the fields of an IBB pipe on columns are zero outside it already
    if (c.zlay && c.q == 19 && c.armed_bc == LBM_BC_IBB) return cudaSuccess;
    count_launch(c, G_STATS);
    return mask_cells(c, nullptr);
}

// The masked fields' sums into res (NP columns, then 3 NBIN of the bins).
// rec: from the FP32 records, else from the FP64 fields (launch_macro wrote
// the one or the other); raw: solid cells keep the virtual fluid.
static cudaError_t stats_sums(Ctx &c, float4 *rec, bool raw, bool bins, double reach, const float *eps_o, double nu,
                              double *res) {
    cudaError_t e;
    const int ibb = c.armed_bc == LBM_BC_IBB;
    count_launch(c, G_STATS, 3);
    // what the masked solid cells held counts in mass and momentum unless the wall is IBB
    const bool solid_held = !raw && !ibb;
    double *bpart = c.partials + (size_t)SNB * NP;
    if (!raw && !(c.zlay && c.q == 19 && ibb))
        if ((e = mask_cells(c, solid_held ? c.partials : nullptr, rec)) != cudaSuccess) return e;
    const int mblk = solid_held && (c.np > 0 || c.has_pipe) ? mask_blocks(c) : 0;
    StatsArgs a{c.u_f, c.rho_f, rec, rec ? rec + c.N : nullptr, c.flags, c.near_key, c.X, c.R,
                c.same_radius ? 20.0f / (float)c.max_radius : 0.f, 2e-7f * (float)(reach + 4.0), eps_o, c.nx, c.ny, c.nz, c.N,
                nu, c.has_pipe, ibb, raw, c.partials, bpart};
    const long long tiles = (long long)((c.nx + 31) / 32) * ((c.ny + 3) / 4) * ((c.nz + ST_RUN - 1) / ST_RUN);
    const int nblk = (int)std::min<long long>(tiles, SNB);
    const size_t smem = bins ? sizeof(double) * 2 * NBIN * ST_TB + sizeof(int) * NBIN : 0;
    void (*kernel)(StatsArgs) = bins ? (rec ? stats_kernel<true, float2> : stats_kernel<true, double>)
                                     : (rec ? stats_kernel<false, float2> : stats_kernel<false, double>);
    if (bins && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
        return e;
    kernel<<<nblk, ST_TB, smem, c.stream>>>(a);
    stats_reduce_kernel<<<NP + (bins ? 3 * NBIN : 0), SB, 0, c.stream>>>(c.partials, bpart, nblk, mblk, res);
    return cudaGetLastError();
}

// Whether sums of float pairs hold what FP64 would: products below 2^-102
// lose their low parts to underflow and those below 2^-149 vanish, which
// shows where the mean square of a sum's terms is below 2^-97 (velocities or
// differences below 2.5e-15: 48 bits of it are left above 2^-149); squares
// beyond FP32's range (an unstable state) show as infinities or NaN. Zero
// sums (a fluid at rest) count as unresolved too: nothing tells them from
// vanished ones.
static bool pairs_resolve(const Ctx &c, const double *s, bool bins, double nu) {
    auto mean = [](double sum, double n) { return n == 0.0 || (sum >= 0x1p-97 * n && std::isfinite(sum)); };
    const double N = (double)c.N, nf = s[ST_NF], four_ss = 1.0 / (0.5 * nu);  // sums hold (nu / 2) 4 s_ij s_ij
    bool ok = std::isfinite(s[ST_MASS] + s[ST_MX] + s[ST_MY] + s[ST_MZ]) && mean(s[ST_KF], nf) && mean(s[ST_EF] * four_ss, nf) &&
              mean(s[ST_KF] + s[ST_KS], N) && mean((s[ST_EF] + s[ST_ES]) * four_ss, N);
    for (int k = 0; bins && k < NBIN; k++) {
        const double *b = s + NP + k;
        ok = ok && mean(b[0], b[2 * NBIN]) && mean(b[NBIN] * four_ss, b[2 * NBIN]);
    }
    return ok;
}

cudaError_t run_stats(Ctx &c, int flags, lbm_stats_t *o) {
    cudaError_t e;
    memset(o, 0, sizeof(*o));
    const int ibm = c.armed_bc == LBM_BC_IBM_U || c.armed_bc == LBM_BC_IBM_B;
    const bool closure = (flags & LBM_STATS_CLOSURE) && c.np > 0 && c.cl_ready && c.max_cl > 0 && c.q == 19;
    // FP32 records of the fields, 16 B per cell: all that 32- and 16-bit
    // storage needs, and the closure's gather input. With such storage they
    // lie in the place of the FP64 fields (rho_f and u_f, 32 B per cell
    // together), the low parts of masked cells behind them; else in the
    // population buffer that the next step overwrites.
    const bool rec = c.storage != LBM_F64;
    float *u32 = rec ? (float *)c.rho_f : (closure ? (float *)c.fB : nullptr);
    if ((e = launch_macro(c, u32, rec)) != cudaSuccess) return e;
    const bool raw = ibm && (flags & LBM_STATS_UNMASK);
    const unsigned nb = (unsigned)((c.N + 255) / 256);
    const double nu = (c.tau - 0.5) / 3.0;
    const bool bins = (flags & LBM_STATS_BINS) && c.np > 0;
    const float *eps_o = nullptr;
    // the bins reach r/R_p = 1 + 0.05 NBIN; the closure 2 lattice units from the surface
    double reach = bins ? 0.05 * NBIN * c.max_radius : 0.0;
    if (closure && reach < 2.0) reach = 2.0;
    if (bins || closure) near_surface(c, nb, reach);
    if (closure) {
        // learned gradients at the near-surface nodes (unmasked velocity in):
        // list the nodes, then one tensor-core kernel gathers each node's
        // features, runs the network and writes the dissipation at the cell
        count_launch(c, G_STATS, 4);
        fill_f32<<<nb, 256, 0, c.stream>>>(c.cl_eps, -1.f, c.N);
        if ((e = cudaMemsetAsync(c.d_counts + 3, 0, sizeof(long long), c.stream)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(c.d_status + 1, 0, sizeof(unsigned), c.stream)) != cudaSuccess) return e;
        int *pids = (int *)c.cl_X;  // the feature buffer is not needed by the fused path
        closure_list_kernel<<<(unsigned)((c.N + 1023) / 1024), 256, 0, c.stream>>>(c.flags, c.near_key, c.N, c.cl_cells, pids, c.d_counts + 3,
                                                      c.max_cl);
        if ((e = mlp_pack_device(c.cl_w, c.cl_pk, c.stream)) != cudaSuccess) return e;
        cudaEvent_t t0 = prof_event(c);
        count_launch(c, G_CLOSURE, 2);  // particle records, inference
        if ((e = closure_eps_tc(c, u32, c.cl_cells, pids, c.d_counts + 3, c.max_cl, c.cl_pk, c.cl_eps,
                                (int *)(c.d_status + 1))) != cudaSuccess)
            return e;
        prof_span(c, G_CLOSURE, t0, prof_event(c));
        eps_o = c.cl_eps;
    }
    double *res = c.partials + (size_t)SNB * (NP + 3 * NBIN);
    if ((e = stats_sums(c, rec ? (float4 *)u32 : nullptr, raw, bins, reach, eps_o, nu, res)) != cudaSuccess) return e;
    const int ncol = NP + (bins ? 3 * NBIN : 0);
    double s[NP + 3 * NBIN] = {0};
    if ((e = cudaMemcpyAsync(s, res, sizeof(double) * ncol, cudaMemcpyDeviceToHost, c.stream)) != cudaSuccess) return e;
    std::vector<double> P(3 * c.np), Uh(3 * c.np), Wh(3 * c.np), Fh(3 * c.np), Th(3 * c.np), mass(c.np), inertia(c.np);
    if (c.np > 0) {
        cudaMemcpyAsync(Uh.data(), c.U, sizeof(double) * 3 * c.np, cudaMemcpyDeviceToHost, c.stream);
        cudaMemcpyAsync(Wh.data(), c.W, sizeof(double) * 3 * c.np, cudaMemcpyDeviceToHost, c.stream);
        cudaMemcpyAsync(Fh.data(), c.Fh, sizeof(double) * 3 * c.np, cudaMemcpyDeviceToHost, c.stream);
        cudaMemcpyAsync(Th.data(), c.Th, sizeof(double) * 3 * c.np, cudaMemcpyDeviceToHost, c.stream);
        cudaMemcpyAsync(mass.data(), c.mass, sizeof(double) * c.np, cudaMemcpyDeviceToHost, c.stream);
        cudaMemcpyAsync(inertia.data(), c.inertia, sizeof(double) * c.np, cudaMemcpyDeviceToHost, c.stream);
    }
    unsigned tc_err = 0;
    if (closure && (e = cudaMemcpyAsync(&tc_err, c.d_status + 1, sizeof(unsigned), cudaMemcpyDeviceToHost,
                                        c.stream)) != cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(c.stream)) != cudaSuccess) return e;
    if (tc_err) return cudaErrorLaunchTimeout;  // a tensor-core wait of the closure ran out
    if (rec && !pairs_resolve(c, s, bins, nu)) {  // the same from FP64 fields and in FP64 sums
        if ((e = launch_macro(c)) != cudaSuccess ||
            (e = stats_sums(c, nullptr, raw, bins, reach, eps_o, nu, res)) != cudaSuccess ||
            (e = cudaMemcpyAsync(s, res, sizeof(double) * ncol, cudaMemcpyDeviceToHost, c.stream)) != cudaSuccess ||
            (e = cudaStreamSynchronize(c.stream)) != cudaSuccess)
            return e;
    }
    o->mass = s[ST_MASS] + s[ST_SMASS];
    for (int d = 0; d < 3; d++) o->momentum[d] = s[ST_MX + d] + s[ST_SX + d];
    o->kinetic_energy = 0.5 * (s[ST_KF] + s[ST_KS]) / (double)c.N;
    o->dissipation = (s[ST_EF] + s[ST_ES]) / (double)c.N;
    o->nfluid = (long long)s[ST_NF];
    o->kinetic_energy_fluid = s[ST_NF] > 0 ? 0.5 * s[ST_KF] / s[ST_NF] : 0.0;
    o->dissipation_fluid = s[ST_NF] > 0 ? s[ST_EF] / s[ST_NF] : 0.0;
    o->bulk_velocity = c.has_pipe && s[ST_NF] > 0 ? s[ST_UZ] / s[ST_NF] : 0.0;
    for (int p = 0; p < c.np; p++) {
        double U2 = 0, W2 = 0;
        for (int d = 0; d < 3; d++) {
            U2 += Uh[3 * p + d] * Uh[3 * p + d];
            W2 += Wh[3 * p + d] * Wh[3 * p + d];
            o->force[d] += Fh[3 * p + d];
            o->torque[d] += Th[3 * p + d];
        }
        o->particle_ke += 0.5 * mass[p] * U2;
        o->particle_ake += 0.5 * inertia[p] * W2;
    }
    if (bins) {
        const double *sk = s + NP, *se = sk + NBIN, *sc = se + NBIN;
        o->nbins = NBIN;
        for (int k = 0; k < NBIN; k++) {
            o->bin_r[k] = 1.0 + 0.05 * (k + 0.5);
            o->bin_count[k] = (long long)sc[k];
            if (sc[k] > 0) {
                const double kf = o->kinetic_energy_fluid > 0 ? o->kinetic_energy_fluid : 1.0;
                const double ef = o->dissipation_fluid > 0 ? o->dissipation_fluid : 1.0;
                o->bin_tke[k] = 0.5 * sk[k] / sc[k] / kf;
                o->bin_eps[k] = se[k] / sc[k] / ef;
            }
        }
    }
    o->nlinks = c.armed_bc == LBM_BC_IBB ? c.nlinks : 0;
    o->nmarkers = c.nm;
    o->step = c.step;
    return cudaSuccess;
}

size_t stats_partials_doubles() { return (size_t)(SNB + 1) * (NP + 3 * NBIN); }

}  // namespace lbmgb
