// Conversions between the column layout of the pipe (columns.cuh) and the
// x-fast order of everything outside its sweeps: the whole state (when the
// wall is first used, in checkpoints), single planes (populations in and
// out), and the macroscopic fields.
#include "columns.cuh"

namespace lbmgb {

// q planes of the state: x fastest -> columns (TOX false) or back
template <typename T, bool TOX>
__global__ void __launch_bounds__(256) convert_kernel(const void *src, void *dst, int q, int nx, int ny, int nz, int zp,
                                                      long long N, long long Np, const uint8_t *solid) {
    __shared__ T sh[COL_TILE][COL_TILE + 1];
    for (int y = blockIdx.y; y < ny; y += gridDim.y)
    for (int i = 0; i < q; i++) {
        const T *s = (const T *)src + i * (TOX ? Np : N);
        T *d = (T *)dst + i * (TOX ? N : Np);
        auto at_x = [&](int x, int z) { return x + (long long)nx * (y + (long long)ny * z); };
        auto at_z = [&](int x, int z) { return z + (long long)zp * (x + (long long)nx * y); };
        column_exchange<T, TOX>(
            sh, nx, nz, [&](int x, int z) {
                if (solid && (solid[x + (long long)nx * y] & FL_SOLID)) return T(0);
                return s[TOX ? at_z(x, z) : at_x(x, z)];
            },
            [&](int x, int z, T v) { d[TOX ? at_x(x, z) : at_z(x, z)] = v; });
    }
}

template <typename T>
static cudaError_t convert_t(Ctx &c, const void *src, void *dst, bool to_x, const uint8_t *solid) {
    if (to_x) convert_kernel<T, true><<<column_tiles(c), 256, 0, c.stream>>>(src, dst, c.q, c.nx, c.ny, c.nz, c.zp, c.N, c.Np,
                                                                                    solid);
    else convert_kernel<T, false><<<column_tiles(c), 256, 0, c.stream>>>(src, dst, c.q, c.nx, c.ny, c.nz, c.zp, c.N, c.Np,
                                                                                solid);
    return cudaGetLastError();
}

// zero_solid: solid columns (flags of plane 0) are stored as zeros
cudaError_t convert_columns(Ctx &c, const void *src, void *dst, bool to_x, bool zero_solid) {
    const uint8_t *solid = zero_solid ? c.flags : nullptr;
    const size_t sb = storage_bytes(c.storage);
    return sb == 8 ? convert_t<double>(c, src, dst, to_x, solid)
                   : (sb == 4 ? convert_t<float>(c, src, dst, to_x, solid) : convert_t<unsigned short>(c, src, dst, to_x, solid));
}

// one population plane to or from the FP64 field v (x fastest, unshifted:
// f = g + w)
template <int S, bool TOX>
__global__ void __launch_bounds__(256) plane_kernel(void *plane, double *v, double w, int nx, int ny, int nz, int zp) {
    typedef typename Store<S>::T T;
    typedef typename Store<S>::R R;
    __shared__ double sh[COL_TILE][COL_TILE + 1];
    T *p = (T *)plane;
    for (int y = blockIdx.y; y < ny; y += gridDim.y) {
    auto at_x = [&](int x, int z) { return x + (long long)nx * (y + (long long)ny * z); };
    auto at_z = [&](int x, int z) { return z + (long long)zp * (x + (long long)nx * y); };
    column_exchange<double, TOX>(
        sh, nx, nz, [&](int x, int z) { return TOX ? (double)Store<S>::ld(p + at_z(x, z)) + w : v[at_x(x, z)]; },
        [&](int x, int z, double f) {
            if (TOX) v[at_x(x, z)] = f;
            else Store<S>::st(p + at_z(x, z), R(f - w));
        });
    }
}

template <int S>
static cudaError_t plane_t(Ctx &c, int i, double w, bool to_f64) {
    void *p = (typename Store<S>::T *)c.fA + i * c.Np;
    if (to_f64) plane_kernel<S, true><<<column_tiles(c), 256, 0, c.stream>>>(p, c.rho_f, w, c.nx, c.ny, c.nz, c.zp);
    else plane_kernel<S, false><<<column_tiles(c), 256, 0, c.stream>>>(p, c.rho_f, w, c.nx, c.ny, c.nz, c.zp);
    return cudaGetLastError();
}

cudaError_t column_plane_copy(Ctx &c, int i, double w, bool to_f64) {
    switch (c.storage) {
    case LBM_F64: return plane_t<LBM_F64>(c, i, w, to_f64);
    case LBM_F32: return plane_t<LBM_F32>(c, i, w, to_f64);
    case LBM_F16S: return plane_t<LBM_F16S>(c, i, w, to_f64);
    default: return plane_t<LBM_BF16S>(c, i, w, to_f64);
    }
}

// rho and u of the post-collision state (macro_kernel's arithmetic), read
// along z and written along x as FP64. IBM (info not null): the total force
// of the last collision is the body force on fluid columns plus the IBM
// force planes sF of the support columns.
template <int S>
__global__ void __launch_bounds__(256) column_macro_kernel(const void *A, const uint8_t *flags, const int *info,
                                                           const void *sFv, long long SF, float4 *rec, double *rho_o, double *u_o,
                                                           int nx, int ny, int nz, int zp, long long N, long long Np,
                                                           double F0, double F1, double F2) {
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
            const int col = x + nx * y;
            const bool solid = flags[col] & FL_SOLID;  // plane 0 tells
            if (solid && !info) return V{R(0), R(0), R(0), R(0)};
            const T *P = (const T *)A + (size_t)col * zp + z;
            R r = R(0), j0 = R(0), j1 = R(0), j2 = R(0);
#pragma unroll
            for (int i = 0; i < 19; i++) {
                const R g = Store<S>::ld(P + i * Np);
                r += g;
                j0 += g * R(cx(i));
                j1 += g * R(cy(i));
                j2 += g * R(cz(i));
            }
            R Fx = solid ? R(0) : R(F0), Fy = solid ? R(0) : R(F1), Fz = solid ? R(0) : R(F2);
            const int k = info ? (info[col] >> 1) - 1 : -1;
            if (k >= 0) {
                const R *sF = (const R *)sFv + (size_t)k * nz + z;
                Fx += sF[0];
                Fy += sF[SF];
                Fz += sF[2 * SF];
            }
            const R rho = R(1) + r, ir = R(1) / rho;
            return V{rho, (j0 - R(0.5) * Fx) * ir, (j1 - R(0.5) * Fy) * ir, (j2 - R(0.5) * Fz) * ir};
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

cudaError_t launch_column_macro(Ctx &c, float4 *rec) {
    count_launch(c, G_STATS);
    const int *info = c.armed_bc == LBM_BC_IBB ? nullptr : c.col_ibm;
    const long long SF = (long long)c.pipe_sp * c.nz;
    switch (c.storage) {
#define MK(S) column_macro_kernel<S><<<column_tiles(c), 256, 0, c.stream>>>(c.fA, c.flags, info, c.sup_F, SF, rec, c.rho_f, c.u_f, c.nx, c.ny, \
                                                                           c.nz, c.zp, c.N, c.Np, c.F[0], c.F[1], c.F[2])
    case LBM_F64: MK(LBM_F64); break;
    case LBM_F32: MK(LBM_F32); break;
    case LBM_F16S: MK(LBM_F16S); break;
    default: MK(LBM_BF16S); break;
#undef MK
    }
    return cudaGetLastError();
}

}  // namespace lbmgb
