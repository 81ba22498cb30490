// The pipe sweep on the column layout (columns.cuh): fused pull-stream +
// collide of the fluid columns with the wall's interpolated bounce-back
// (Sec. 2.1), one launch per step.
//
// What bounds it: HBM. Each fluid cell reads and writes its populations
// once (2 x 19 values), in whole sectors: on the benchmark pipe
// (148 x 148 x 438, R = 73) FP32 takes 0.1766 ms per step, 6.32 TB/s of
// algorithmic bytes.
//
// Why columns: with x fastest the pipe's rows are runs of up to 146 cells
// that start anywhere, the wall cells sit at the ends of every run, and a
// warp that holds one spends a third more instructions on moving values
// between its lanes. With z fastest the wall is uniform over a warp: a wall
// column (one in 28 on the benchmark pipe) takes a uniform branch with
// weights loaded once per warp, the others carry nothing for it, and no
// work list, ghost array or partial value survives a step. The sweep over
// x-fast fluid runs with the wall's values exchanged between the lanes
// took 0.2275 ms (FP32) and, with two cells per lane, 0.178 ms (FP16)
// against 0.1766 and 0.125 ms here.
#include "columns.cuh"

#include <type_traits>

namespace lbmgb {

template <typename R>
struct ColumnCoef {
    R k1, k2;
};

__device__ __forceinline__ ColumnCoef<float> ld_coef(const ColumnCoef<float> *p) {
    const float2 v = __ldg((const float2 *)p);
    return ColumnCoef<float>{v.x, v.y};
}
__device__ __forceinline__ ColumnCoef<double> ld_coef(const ColumnCoef<double> *p) {
    const double2 v = __ldg((const double2 *)p);
    return ColumnCoef<double>{v.x, v.y};
}

struct ColumnArgs {
    const void *A;      // shifted as the pointers of the pulls
    const int2 *cols;   // fluid columns: x + nx y, index of the column's wall record (-1: no wall link)
    const uint4 *wall;  // per wall column: direction masks of its links (x), of those with q >= 1/2 (y), single-node (z)
    const void *coef;   // per wall column 19 pairs of weights (arithmetic type of the storage)
    ColumnItems items;
    ColumnPtrs p;
    long long Np;
    unsigned *status;
    PairK pk;
    Rates rt;
    double F[3];
    float Fs[3];
};

// Resident blocks of 256 per SM the registers are sized for. The sweep lives
// on loads in flight: FP32 on the benchmark pipe took 0.190 ms at 3 and 4
// blocks, 0.180 at 5, 0.1766 at 6 (40 registers, no spills), 0.192 at 7 (32,
// spills); FP16 0.143, 0.131, 0.125, 0.139. Blocks of 64, 128 or 512 threads
// at the same registers were no faster, a persistent grid with the next
// column's record loaded one round ahead slower (0.192). The MRT collision
// fits 4 blocks without spilling, FP64 3 (BGK, 4 bytes spilled) and 2.
// The flat walk's small sections live on the latency of the wall's loads
// instead: 64 registers for six links' values at once (148 x 148 x 4, FP32:
// 8.2 us per step with the links one by one, 6.2 so).
constexpr int column_min_blocks(int S, bool SRT, bool FLAT) {
    return S == LBM_F64 ? (SRT ? 3 : 2) : (SRT && !FLAT ? 6 : 4);
}

// v as it reads back from storage: what the wall adds to a population is a
// stored number like the populations themselves (SCALED: v is g * 2^10)
template <int S, bool SCALED, typename R>
__device__ __forceinline__ R stored(R v) {
    if constexpr (S == LBM_F16S) {
        constexpr float f = SCALED ? 1.0f : F16_SCALE;
        return __half2float(__float2half_rn(v * f)) * (1.0f / f);
    } else if constexpr (S == LBM_BF16S) {
        return __bfloat162float(__float2bfloat16_rn(v));
    } else {
        return v;
    }
}

// One thread per cell of the fluid columns. SN: the wall has single-node
// links. WRAP: fluid columns touch an x or y face of the box,
// so that pulls wrap in x and y too.
template <int S, bool FORCE, bool SRT, bool SN, bool WRAP, bool FLAT>
__global__ void __launch_bounds__(256, column_min_blocks(S, SRT, FLAT)) sweep_columns(ColumnArgs a) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    // BGK on FP16 runs on the stored numbers g * 2^10 (the scale is a power
    // of two: the arithmetic rounds as on g itself)
    constexpr bool pairs = SRT && sizeof(R) == 4;
    constexpr bool scaled = S == LBM_F16S && pairs;
    auto ld = [](const T *p) -> R {
        if constexpr (scaled) return Store<LBM_F16S>::ld_scaled(p);
        else return Store<S>::ld(p);
    };
    unsigned ci;
    int z;
    if (!a.items.cell<FLAT>(ci, z)) return;
    const int2 col = __ldg(a.cols + ci);
    if (z >= a.p.nz) return;
    const int e = column_element<FLAT>(a.p, col.x, z);
    R g[19];
    uint4 w;
    if constexpr (FLAT) w = col.y >= 0 ? __ldg(a.wall + col.y) : make_uint4(0u, 0u, 0u, 0u);  // on its way with the pulls
    column_pull<T, WRAP, FLAT>(g, a.p, col.x, z, ld);
    if (col.y >= 0) {  // uniform over a warp of one column
        // the populations that come back from the wall (linear interpolated
        // bounce-back, or the single-node scheme): f_ibar(x_f, t+1) =
        //   k1 f*_l(x_f) + k2 f*_l(x_f - c_l)   q < 1/2, the pull of direction l
        //   k1 f*_l(x_f) + k2 f*_ibar(x_f)      q >= 1/2
        //   f*_l(x_f) + k2 (d_l + d_ibar)       single-node
        if constexpr (!FLAT) w = __ldg(a.wall + col.y);
        const ColumnCoef<R> *kc = (const ColumnCoef<R> *)a.coef + 19 * (size_t)col.y;
        const T *Ae = (const T *)a.A + e;  // the cell's own populations
        auto bounce = [&](int l, R k1, R k2, R fl, auto own) {  // own(): f*_ibar(x_f)
            if (SN && ((w.z >> l) & 1u)) {
                const R d = single_node_pair<S>(Ae, (size_t)a.Np, l, body_force<R>(a, 0), body_force<R>(a, 1),
                                                body_force<R>(a, 2), a.rt);
                g[opp(l)] = stored<S, scaled>(fma(scaled ? k2 * R(F16_SCALE) : k2, d, fl));
            } else if ((w.y >> l) & 1u) {
                g[opp(l)] = stored<S, scaled>(fma(k1, fl, k2 * own()));
            } else {
                g[opp(l)] = fma(k2, g[l], stored<S, scaled>(k1 * fl));
            }
        };
        if constexpr (FLAT) {
            // the lanes' columns have different links and a small section has
            // no other warps to hide their loads: six directions (three
            // opposite pairs) at a time, the loads of a group in flight together
#pragma unroll
            for (int l0 = 1; l0 < 19; l0 += 6) {
                if (((w.x >> l0) & 63u) == 0u) continue;
                R f[6];
                ColumnCoef<R> k[6];
#pragma unroll
                for (int j = 0; j < 6; j++) {
                    const int l = l0 + j, o = opp(l);
                    f[j] = ((w.x >> l) | (w.y >> o)) & 1u ? ld(Ae + l * a.Np) : R(0);
                    k[j] = (w.x >> l) & 1u ? ld_coef(kc + l) : ColumnCoef<R>{R(0), R(0)};
                }
#pragma unroll
                for (int j = 0; j < 6; j++)
                    if ((w.x >> (l0 + j)) & 1u) bounce(l0 + j, k[j].k1, k[j].k2, f[j], [&]() { return f[opp(l0 + j) - l0]; });
            }
        } else {
#pragma unroll
            for (int l = 1; l < 19; l++) {
                if (!((w.x >> l) & 1u)) continue;
                const R k1 = __ldg(&kc[l].k1), k2 = __ldg(&kc[l].k2);
                bounce(l, k1, k2, ld(Ae + l * a.Np), [&]() { return ld(Ae + opp(l) * a.Np); });
            }
        }
    }
    if constexpr (pairs) {
        float rho, u2;
        collide_pairs<FORCE, scaled ? 10 : 0>(g, a.pk, rho, u2);
        if (!(rho > 0.5f && rho < 2.0f && u2 < 0.09f)) atomicOr(a.status, 1u);
    } else {
        R rho, ux, uy, uz;
        collide<R, FORCE, SRT>(g, body_force<R>(a, 0), body_force<R>(a, 1), body_force<R>(a, 2), a.rt, rho, ux, uy, uz);
        watchdog(rho, ux, uy, uz, a.status);
    }
#pragma unroll
    for (int i = 0; i < 19; i++) {
        if constexpr (scaled) Store<LBM_F16S>::st_scaled((T *)a.p.Bp[i] + e, g[i]);
        else Store<S>::st((T *)a.p.Bp[i] + e, g[i]);
    }
}

template <int S, bool FORCE, bool SRT>
static cudaError_t launch_columns_t(Ctx &c) {
    ColumnArgs a{};
    a.cols = c.col_list;
    a.wall = c.col_wall;
    a.coef = c.col_coef;
    a.items = column_items(c, c.ncols);
    const bool sn = c.static_single > 0, wrap = !c.pipe_nowrap || (c.col_flat && sn);
    column_ptrs(c, a.p);
    a.A = (const char *)c.fA + (long long)storage_bytes(c.storage) * a.p.shift;
    a.Np = c.Np;
    a.status = c.d_status;
    a.pk = make_pair_k(c.rt.d_nu, c.F);
    a.rt = c.rt;
    for (int d = 0; d < 3; d++) {
        a.F[d] = c.F[d];
        a.Fs[d] = (float)c.F[d];
    }
    const unsigned nb = column_item_blocks(c, a.items);
    count_launch(c, G_BULK);
    if (nb == 0) return cudaSuccess;
    if (c.col_flat) {
        if (wrap) sweep_columns<S, FORCE, SRT, true, true, true><<<nb, 256, 0, c.stream>>>(a);
        else sweep_columns<S, FORCE, SRT, false, false, true><<<nb, 256, 0, c.stream>>>(a);
    } else if (wrap) {
        sweep_columns<S, FORCE, SRT, true, true, false><<<nb, 256, 0, c.stream>>>(a);
    } else {
        if (sn) sweep_columns<S, FORCE, SRT, true, false, false><<<nb, 256, 0, c.stream>>>(a);
        else sweep_columns<S, FORCE, SRT, false, false, false><<<nb, 256, 0, c.stream>>>(a);
    }
    return cudaGetLastError();
}

template <int S>
static cudaError_t launch_columns_s(Ctx &c) {
    const bool force = c.F[0] != 0.0 || c.F[1] != 0.0 || c.F[2] != 0.0;
    if (c.rates == LBM_RATES_SRT) return force ? launch_columns_t<S, true, true>(c) : launch_columns_t<S, false, true>(c);
    return force ? launch_columns_t<S, true, false>(c) : launch_columns_t<S, false, false>(c);
}

cudaError_t launch_column_sweep(Ctx &c) {
    switch (c.storage) {
    case LBM_F64: return launch_columns_s<LBM_F64>(c);
    case LBM_F32: return launch_columns_s<LBM_F32>(c);
    case LBM_F16S: return launch_columns_s<LBM_F16S>(c);
    default: return launch_columns_s<LBM_BF16S>(c);
    }
}

}  // namespace lbmgb
