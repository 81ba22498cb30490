// Three-dimensional spectra of kinetic energy and dissipation (Sec. 3.2:
// the paper compares IBB and IBM spectra with the velocity inside the
// particles masked or not).
//
// The velocity field of the statistics (masked as in lbm_stats) is
// transformed with a hand-written FP32 FFT. Two complex fields carry the
// three real components, u_x + i u_y and u_z: a shell holds k together with
// -k, so the shell sums of |Z|^2 for Z = X + iY are those of |X|^2 + |Y|^2
// and nothing has to be separated.
//
// What bounds it: HBM (88 B per cell: 24 in, 16 out along x; 16 + 16 along
// y; 16 in along z) and the macroscopic fields before it.
//   fft_x   lines along x, read from the FP64 velocity, through shared memory
//   fft_y   lines along y, registers to registers
//   fft_z   lines along z and the shell sums: the transformed values are
//           squared in place and never written
// Lines along y and z are taken L at a time in consecutive x, so that every
// load and store is a run of 64 to 128 bytes. A thread holds 8 points of a
// line; the passes are radix-8 Stockham (a last pass of radix 4 or 2) with
// exchanges through shared memory and twiddles from a table in it.
// Shell sums: FP64. A block takes lines k_x together with -k_x and all k_z,
// so that the four (+-k_x, +-k_z) energies, kept as unevaluated FP32 pairs
// (hi + lo), are added before one FP64 addition per quadruple goes to the
// block's bins; FP64 is the scarce unit here. The blocks' bins are added on
// the host in a fixed order.
// 256^3, 222 shells, the whole call: 6.3 ms with a radix-2 transform per
// component and two shared-memory FP64 atomics per cell and component, 1.22
// ms now.
//
// Scratch: the population buffer that the next step overwrites holds the
// two complex fields (16 bytes per cell of its 38 or more) and the
// per-block sums, so the entry point needs no memory of its own.
#include "lbm_internal.cuh"
#include "spectra_scratch.h"

#include <cmath>
#include <vector>

namespace lbmgb {

// lines per block: runs of 128 bytes, and at most 1024 threads of 8 points
__host__ __device__ constexpr int fft_lines(int logn) { return logn <= 8 ? 16 : 8; }
__host__ __device__ constexpr int fft_threads(int logn) { return (fft_lines(logn) << logn) / 8; }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 mul_mi(float2 a) { return make_float2(a.y, -a.x); }  // a (-i)

__device__ __forceinline__ void fft2(float2 &a, float2 &b) {
    const float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}
// outputs in natural order
__device__ __forceinline__ void fft4(float2 &a0, float2 &a1, float2 &a2, float2 &a3) {
    const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = mul_mi(csub(a1, a3));
    a0 = cadd(t0, t2);
    a1 = cadd(t1, t3);
    a2 = csub(t0, t2);
    a3 = csub(t1, t3);
}
__device__ __forceinline__ void fft8(float2 v[8]) {
    constexpr float h = 0.70710678118654752f;
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    fft4(e0, e1, e2, e3);
    fft4(o0, o1, o2, o3);
    o1 = make_float2(h * (o1.x + o1.y), h * (o1.y - o1.x));   // (1 - i) / sqrt 2
    o2 = mul_mi(o2);
    o3 = make_float2(h * (o3.y - o3.x), -h * (o3.x + o3.y));  // (-1 - i) / sqrt 2
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1);
    v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2);
    v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3);
    v[7] = csub(e3, o3);
}

// One line of n = 2^LOGN points per column l of S ([point][line], LS lines
// apart): thread (j, l) enters with points j + r n/8 in v[r] and leaves with
// the transform in v; OUT(r) is the frequency of v[r].
template <int LOGN>
struct LineFft {
    static constexpr int n = 1 << LOGN, R = LOGN % 3 == 0 ? 8 : (LOGN % 3 == 2 ? 4 : 2);  // last radix
    static constexpr int NsL = n / R;  // length before the last pass
    static __device__ __forceinline__ int out(int j, int r) {
        if (R == 8) return j + r * NsL;                                   // NsL = n/8 > j
        if (R == 4) return (j + (r >> 2) * (n / 8)) + (r & 3) * NsL;      // butterflies j and j + n/8
        return (j + (r >> 1) * (n / 8)) + (r & 1) * NsL;                  // butterflies j + b n/8
    }
    static __device__ __forceinline__ void run(float2 v[8], float2 *S, int LS, const float2 *tw, int j, int l) {
#pragma unroll
        for (int ns = 1; ns * 8 <= n; ns *= 8) {  // radix-8 passes
            const int k = j & (ns - 1);
            if (ns > 1) {
#pragma unroll
                for (int r = 1; r < 8; r++) v[r] = cmul(v[r], tw[r * k * (n / (ns * 8))]);
            }
            fft8(v);
            if (ns * 8 == n) return;  // the last pass
            __syncthreads();  // the reads of the pass before are done
            const int b = (j - k) * 8 + k;
#pragma unroll
            for (int r = 0; r < 8; r++) S[(b + r * ns) * LS + l] = v[r];
            __syncthreads();
            if (ns * 64 <= n) {
#pragma unroll
                for (int r = 0; r < 8; r++) v[r] = S[(j + r * (n / 8)) * LS + l];
            }
        }
        if constexpr (R == 4) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const int jj = j + h * (n / 8);
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    v[4 * h + r] = S[(jj + r * NsL) * LS + l];
                    if (r > 0) v[4 * h + r] = cmul(v[4 * h + r], tw[r * jj]);
                }
                fft4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
            }
        } else if constexpr (R == 2) {
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int jj = j + h * (n / 8);
                v[2 * h] = S[jj * LS + l];
                v[2 * h + 1] = cmul(S[(jj + NsL) * LS + l], tw[jj]);
                fft2(v[2 * h], v[2 * h + 1]);
            }
        }
    }
};

// tw[i] = exp(-2 pi i / n)
__device__ __forceinline__ void twiddle_table(float2 *tw, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        float sn, cs;
        sincospif(-2.0f * (float)i / (float)n, &sn, &cs);
        tw[i] = make_float2(cs, sn);
    }
}

// lines along x of field blockIdx.y (0: u_x + i u_y, 1: u_z), the velocity
// times pre (a power of two); L consecutive lines per block, through shared
// memory with one column of padding
template <int LOGN>
__global__ void __launch_bounds__(fft_threads(LOGN)) fft_x_kernel(const double *u, float2 *d, long long N, float pre) {
    constexpr int n = 1 << LOGN, L = fft_lines(LOGN), LS = L + 1, TB = fft_threads(LOGN);
    extern __shared__ float2 sm[];
    float2 *S = sm, *tw = sm + n * LS;
    const int f = blockIdx.y;
    const long long first = (long long)blockIdx.x * L * n;
    twiddle_table(tw, n);
    const double *p = u + (f ? 2 * N : 0) + first;
    for (int e = threadIdx.x; e < L * n; e += TB)
        S[(e & (n - 1)) * LS + (e >> LOGN)] = make_float2(pre * (float)p[e], f ? 0.0f : pre * (float)p[N + e]);
    __syncthreads();
    const int l = threadIdx.x % L, j = threadIdx.x / L;
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 8; r++) v[r] = S[(j + r * (n / 8)) * LS + l];
    LineFft<LOGN>::run(v, S, LS, tw, j, l);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; r++) S[LineFft<LOGN>::out(j, r) * LS + l] = v[r];
    __syncthreads();
    float2 *o = d + f * N + first;
    for (int e = threadIdx.x; e < L * n; e += TB) o[e] = S[(e & (n - 1)) * LS + (e >> LOGN)];
}

// lines along y, in place: L consecutive x of one z per block
template <int LOGN>
__global__ void __launch_bounds__(fft_threads(LOGN)) fft_y_kernel(float2 *d, long long N) {
    constexpr int n = 1 << LOGN, L = fft_lines(LOGN) < n ? fft_lines(LOGN) : n;
    extern __shared__ float2 sm[];
    float2 *S = sm, *tw = sm + n * L;
    twiddle_table(tw, n);
    __syncthreads();
    const int l = threadIdx.x % L, j = threadIdx.x / L;
    const long long z = blockIdx.x / (n / L), x = (blockIdx.x % (n / L)) * L + l;
    float2 *p = d + blockIdx.y * N + z * n * n + x;
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 8; r++) v[r] = p[(long long)(j + r * (n / 8)) * n];
    LineFft<LOGN>::run(v, S, L, tw, j, l);
#pragma unroll
    for (int r = 0; r < 8; r++) p[(long long)LineFft<LOGN>::out(j, r) * n] = v[r];
}

// shell K = round(|k|) of an integer squared norm k2, decided in integers:
// K^2 - K + 1 <= k2 <= K^2 + K
__device__ __forceinline__ int shell_of(int k2) {
    int K = (int)sqrtf((float)k2);
    while (K * K + K < k2) K++;
    while (K > 0 && K * K - K + 1 > k2) K--;
    return K;
}

// |z|^2 as an unevaluated FP32 sum
__device__ __forceinline__ float2 norm_pair(float2 z) { return pair_add(pair_mul(z.x, z.x), pair_mul(z.y, z.y)); }

// lines along z of both fields and the shell sums: per block in turn H lines
// k_x = i and the H lines of their opposites (i = 0 is paired with n/2: both
// are their own opposites) at one k_y
template <int LOGN>
__global__ void __launch_bounds__(fft_threads(LOGN)) fft_z_bins_kernel(const float2 *d, long long N, double scale,
                                                                      double dfac, int nbins, double *part) {
    constexpr int n = 1 << LOGN, L = fft_lines(LOGN) < n ? fft_lines(LOGN) : n, H = L / 2, TB = (L * n) / 8;
    constexpr int groups = n / 2 / H;
    extern __shared__ float2 sm[];
    float2 *S = sm, *tw = sm + n * L;
    double *sb = (double *)(tw + n);  // E[nbins], D[nbins]
    twiddle_table(tw, n);
    for (int i = threadIdx.x; i < 2 * nbins; i += TB) sb[i] = 0.0;
    __syncthreads();
    const int l = threadIdx.x % L, j = threadIdx.x / L;
    for (int g = blockIdx.x; g < groups * n; g += gridDim.x) {
        const int iy = g / groups, i0 = (g % groups) * H;
        const int iu = i0 + l % H;  // this thread's line: iu or its opposite
        const int ix = l < H ? iu : (iu == 0 ? n / 2 : n - iu);
        float2 e[8];
#pragma unroll
        for (int f = 0; f < 2; f++) {
            const float2 *p = d + f * N + (long long)iy * n + ix;
            float2 v[8];
#pragma unroll
            for (int r = 0; r < 8; r++) v[r] = p[(long long)(j + r * (n / 8)) * n * n];
            LineFft<LOGN>::run(v, S, L, tw, j, l);
#pragma unroll
            for (int r = 0; r < 8; r++) e[r] = f == 0 ? norm_pair(v[r]) : pair_add(e[r], norm_pair(v[r]));
            __syncthreads();  // S is free for the next field
        }
#pragma unroll
        for (int r = 0; r < 8; r++) S[LineFft<LOGN>::out(j, r) * L + l] = e[r];
        __syncthreads();
        // (k_x, k_z >= 0) with k_z = 0 .. n/2: add the opposite lines and -k_z
        const int ky = iy < n / 2 ? iy : iy - n;
        for (int t = threadIdx.x; t < H * (n / 2 + 1); t += TB) {
            const int a = t % H, kz = t / H, zo = (n - kz) & (n - 1);
            float2 s0 = S[kz * L + a], s1 = S[kz * L + a + H];
            if (zo != kz) {
                s0 = pair_add(s0, S[zo * L + a]);
                s1 = pair_add(s1, S[zo * L + a + H]);
            }
            const int kx = i0 + a;
            const int ka = ky * ky + kz * kz;
            auto put = [&](float2 s, int k2) {
                const int K = shell_of(k2);
                if (K >= nbins) return;
                const double q = pair_value(s);
                atomicAdd(&sb[K], q);
                atomicAdd(&sb[nbins + K], (double)k2 * q);
            };
            if (kx == 0) {
                put(s0, ka);
                put(s1, ka + (n / 2) * (n / 2));
            } else {
                put(pair_add(s0, s1), ka + kx * kx);
            }
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < nbins; k += TB) {
        part[(size_t)blockIdx.x * 2 * nbins + k] = scale * sb[k];
        part[(size_t)blockIdx.x * 2 * nbins + nbins + k] = scale * dfac * sb[nbins + k];
    }
}

template <int LOGN>
static cudaError_t spectrum_t(Ctx &c, int nbins, float2 *field, double *part, double scale, double dfac, float pre,
                              int &blocks) {
    constexpr int n = 1 << LOGN, Lx = fft_lines(LOGN), L = Lx < n ? Lx : n, TB = fft_threads(LOGN), TZ = L * n / 8;
    const size_t smx = sizeof(float2) * (size_t)(n * (Lx + 1) + n), smy = sizeof(float2) * (size_t)(n * L + n),
                 smz = smy + sizeof(double) * 2 * (size_t)nbins,
                 // the attribute is the process's: what the most bins need,
                 // so that no other thread's call sets it below this one's
                 smz_most = smy + sizeof(double) * 2 * LBM_SPECTRUM_MAX_BINS;
    cudaError_t e;
    if ((e = cudaFuncSetAttribute(fft_x_kernel<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smx)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(fft_y_kernel<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smy)) != cudaSuccess ||
        (e = cudaFuncSetAttribute(fft_z_bins_kernel<LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smz_most)) != cudaSuccess)
        return e;
    int per_sm = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fft_z_bins_kernel<LOGN>, TZ, smz);
    blocks = spectrum_blocks((size_t)c.q * (size_t)c.N * storage_bytes(c.storage), c.N, n, L / 2, nbins,
                             (per_sm > 0 ? per_sm : 1) * (sms > 0 ? sms : 1));
    if (blocks < 1) return cudaErrorInvalidValue;  // refused by the caller already
    count_launch(c, G_STATS, 3);
    fft_x_kernel<LOGN><<<dim3((unsigned)(n * n / Lx), 2), TB, smx, c.stream>>>(c.u_f, field, c.N, pre);
    fft_y_kernel<LOGN><<<dim3((unsigned)(n * n / L), 2), TZ, smy, c.stream>>>(field, c.N);
    fft_z_bins_kernel<LOGN><<<(unsigned)blocks, TZ, smz, c.stream>>>(field, c.N, scale, dfac, nbins, part);
    return cudaGetLastError();
}

cudaError_t run_spectrum(Ctx &c, int flags, int nbins, double *E, double *D) {
    cudaError_t e;
    const int n = c.nx;
    int logn = 0;
    while ((1 << logn) < n) logn++;
    const long long N = c.N;
    float2 *field = (float2 *)c.fB;
    double *part = (double *)((char *)c.fB + spectrum_bins_offset(N));
    if ((e = launch_macro(c)) != cudaSuccess) return e;
    const int ibm = c.armed_bc == LBM_BC_IBM_U || c.armed_bc == LBM_BC_IBM_B;
    if (!(ibm && (flags & LBM_STATS_UNMASK)))
        if ((e = launch_mask(c)) != cudaSuccess) return e;
    const double nu = (c.tau - 0.5) / 3.0;
    const double scale = 0.5 / ((double)N * (double)N);
    const double two_pi_n = 2.0 * 3.141592653589793 / n;
    const double dfac = 2.0 * nu * two_pi_n * two_pi_n;
    std::vector<double> hp;
    auto sums = [&](float pre) -> cudaError_t {  // E and D of the velocity times pre; their sum of |Z|^2 in total
        int blocks = 0;
        const double sc = scale / ((double)pre * (double)pre);
        switch (logn) {
#define SP(K) case K: e = spectrum_t<K>(c, nbins, field, part, sc, dfac, pre, blocks); break
            SP(3); SP(4); SP(5); SP(6); SP(7); SP(8); SP(9); SP(10);
#undef SP
        default: return cudaErrorInvalidValue;  // refused by the caller already
        }
        if (e != cudaSuccess) return e;
        hp.resize((size_t)2 * nbins * blocks);
        if ((e = cudaMemcpyAsync(hp.data(), part, sizeof(double) * hp.size(), cudaMemcpyDeviceToHost, c.stream)) !=
            cudaSuccess)
            return e;
        if ((e = cudaStreamSynchronize(c.stream)) != cudaSuccess) return e;
        for (int k = 0; k < nbins; k++) {
            double se = 0.0, sd = 0.0;
            for (int b = 0; b < blocks; b++) {  // fixed block order
                se += hp[(size_t)b * 2 * nbins + k];
                sd += hp[(size_t)b * 2 * nbins + nbins + k];
            }
            E[k] = se;
            D[k] = sd;
        }
        return cudaSuccess;
    };
    if ((e = sums(1.0f)) != cudaSuccess) return e;
    // |Z|^2 is formed in FP32. Where its mean over the wave vectors is below
    // 2^-72, the transform's own rounding (2^-24 of Z) has squares that
    // underflow; the velocity goes in again times 2^80 (|Z| < 2^59 then).
    // Beyond FP32's range (an unstable state), times 2^-64.
    double total = 0.0;
    for (int k = 0; k < nbins; k++) total += E[k];
    if (!std::isfinite(total)) return sums(0x1p-64f);
    if (total < 0x1p-72 * scale * (double)N) return sums(0x1p80f);
    return cudaSuccess;
}

}  // namespace lbmgb
