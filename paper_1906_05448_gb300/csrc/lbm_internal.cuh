// Internal definitions of the GB300 lattice Boltzmann library: the context
// that the C ABI hands out, profiling groups and the launcher prototypes.
// Device-side definitions are in lbm_device.cuh.
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <vector>

#include "lbm.h"
#include "lbm_device.cuh"

namespace lbmgb {

// ------------------------------------------------------------ context -----
struct Ctx {
    lbm_grid g;
    int nx, ny, nz;
    long long N;
    double tau, F[3];
    int storage, rates;
    int q = 19;  // velocity set: 19 (every path) or 27 (periodic box or pipe with IBB, BGK)
    unsigned *q27_colmask;  // D3Q27 pipe: per (x, y) column, the directions whose column is solid
    unsigned *q27_hmask;    // D3Q27 pipe: per column, the wall directions with q >= 1/2 or the halfway fallback
    void *q27_coef;         // D3Q27 pipe: per column and direction, the two wall weights
    Rates rt;
    cudaStream_t stream;
    char *ws;
    size_t ws_bytes;
    // fields
    void *fA, *fB;
    uint8_t *flags;
    int *owner, *aux;
    // compact sites (IBB boundary cells or IBM support cells)
    long long max_sites;
    int *site_cell, *site_first;
    unsigned *site_mask;
    // IBM per site: (rho, u*) as 4 values, accumulated force, force of the
    // current pass, in the storage's arithmetic type (double for FP64, else float)
    void *sup_ru, *sup_F, *sup_Fp;
    // links
    long long max_links;
    int *link_cell, *link_pid;
    int8_t *link_dir, *link_scheme;
    double *link_q;
    void *link_dP, *link_dT;  // per-link momentum exchange and torque (arithmetic type of the storage)
    // column layout of the pipe (columns.cuh), in use once zlay is set
    int zlay, zp;      // zp: elements from a column to the next (>= nz)
    int col_flat;      // the sweeps walk the cells across the ends of the columns (zp = nz)
    long long Np;      // elements of a population plane in that layout
    int2 *col_list;    // fluid columns: x + nx y, index of the column's wall record or -1 (IBB, D3Q27)
    long long ncols, max_wall;
    uint4 *col_wall;   // per wall column: direction masks of its links, of those with q >= 1/2, of single-node ones
    void *col_coef;    // per wall column 19 pairs of weights (arithmetic type of the storage)
    int *col_ibm;      // IBM: per column (support index + 1) << 1 | solid (in the place of col_list)
    int markers_stale; // IBM on columns: the marker forces of the last step are not in mFacc yet
    long long static_single;  // single-node (scheme 2) links of a plane of the wall
    int pipe_nowrap;   // no fluid cell on an x or y face: pulls wrap only in z
    // compaction scratch
    int nblk;
    long long *blk_sites, *blk_links;
    long long *d_counts;  // [0] sites, [1] links, [2] refill nodes, [3] closure samples, [4] single-node links
    int *sn_list;         // links of the single-node scheme (link indices), d_counts[4] of them
    int *refill_list, *refill_pid;
    long long max_refill;
    long long nsites, nlinks;   // host copies (valid after a sync)
    long long nsites_hint;      // launch sizing: a bound on the device count
    long long nlinks_hint;
    // particles (FP64)
    int max_np, np, fixed;
    double dens;
    double *X, *Xold, *U, *W, *R, *mass, *inertia, *Fh, *Th, *Fprev, *Tprev, *Fc, *Iu, *Ir;
    int *has_prev;
    float4 *Xf;  // FP32 centre and radius (contact search)
    // markers
    long long max_markers, nm;
    double *mX, *mUnit, *mdV, *mFacc;
    void *mUd, *mFaccR;  // desired marker velocity, pass force sum (arithmetic type of the storage)
    void *mFr;  // marker forces of the pass in the arithmetic type (spreading)
    int *mB;    // per marker: first stencil node floor(X) - 1 (3 ints, wrapped)
    void *mE;   // per marker: X - floor(X) in the arithmetic type (3 values)
    int *mpid, *m_first;
    double rd;  // marker retraction (IBM-B: 0.4)
    double max_radius;
    bool same_radius;  // every particle has max_radius
    // pipe IBM: ring markers per plane and, per (x, y) column, the ring
    // markers whose 4x4 footprint covers it with their x-y weights
    int pipe_nc;
    double pipe_dV;
    int *pipe_xy_start, *pipe_xy_j;
    void *pipe_xy_w;  // x-y weights in the storage's arithmetic type
    long long pipe_max_xy;
    // pipe interpolation: per ring marker, 16 (support site in a plane, x-y
    // weight) entries; pipe_sp = support sites per z plane
    int *pipe_it_k;
    void *pipe_it_w;  // arithmetic type of the storage
    int pipe_sp, pipe_max_ring;
    // statistics scratch
    double *rho_f, *u_f, *partials;  // u_f begins where rho_f ends (up to the alignment of the workspace's arrays)
    unsigned long long *near_key;  // nearest particle surface per cell (diag.cu)
    // status
    unsigned *d_status;
    unsigned *h_status;  // pinned: [0] status word, [2..5] d_counts[0..1]
    cudaEvent_t ev_status;
    bool status_pending;
    double wait_limit_s;  // bound of the host waits on the stream (lbm_set_wait_limit)
    // geometry
    int has_pipe;
    double pipe_R, pipe_cx, pipe_cy;
    int armed_bc;
    long long step;
    bool broken;
    bool initialised_pops;
    char err[256];
    // learned closure: weights, scales and sample buffers
    float *cl_w, *cl_X, *cl_Y, *cl_eps;
    int *cl_cells;
    void *cl_pk;
    long long max_cl, cl_last_n;
    double cl_uscale, cl_gscale;
    int cl_ready;
    // profiling
    long long launches;                 // every kernel launched
    long long group_launches[LBM_NGROUPS];
    int prof_on;
    void *prof;                         // host-side event records (lbm_api.cu)
};

// every launcher calls this once per kernel it launches
inline void count_launch(Ctx &c, int group, int n = 1) {
    c.launches += n;
    c.group_launches[group] += n;
}
enum { G_BULK = 0, G_BND = 1, G_IBM = 2, G_IBMCOL = 3, G_PART = 4, G_GEOM = 5, G_STATS = 6, G_OTHER = 7, G_CLOSURE = 8 };

}  // namespace lbmgb

struct lbm_ctx {
    lbmgb::Ctx c;
};

// ------------------------------------------------ cross-file launchers ----
namespace lbmgb {
cudaError_t launch_init_equilibrium(Ctx &c, const double *u_dev, double rho0);
cudaError_t launch_stream_collide(Ctx &c, int bc);
cudaError_t launch_column_sweep(Ctx &c);  // sweep_columns.cu: the pipe's IBB step
// columns.cu: the state between the two layouts, one plane to or from
// c.rho_f, the macroscopic fields
cudaError_t convert_columns(Ctx &c, const void *src, void *dst, bool to_x, bool zero_solid);
cudaError_t column_plane_copy(Ctx &c, int i, double w, bool to_f64);
cudaError_t launch_column_macro(Ctx &c, float4 *rec);  // rec: FP32 records instead of c.rho_f, c.u_f
// ibm_columns.cu: the pipe's IBM step, and its forces in the order of the ABI
cudaError_t launch_ibm_columns_sweep(Ctx &c);
cudaError_t launch_ibm_columns_passes(Ctx &c);
cudaError_t launch_ibm_columns_collide(Ctx &c);
cudaError_t refresh_markers(Ctx &c);
cudaError_t copy_site_force(Ctx &c, void *list, bool out);
cudaError_t launch_ibb_links(Ctx &c);
cudaEvent_t prof_event(Ctx &c);  // profiling event on the stream (null when off)
void prof_span(Ctx &c, int g, cudaEvent_t a, cudaEvent_t b);  // time from a to b into group g
cudaError_t launch_ibm_collide(Ctx &c);
cudaError_t launch_pipe_flags(Ctx &c);
cudaError_t launch_sphere_mark(Ctx &c, bool clear_old);
cudaError_t launch_refill(Ctx &c);
cudaError_t launch_finish_geometry(Ctx &c);
cudaError_t build_sites(Ctx &c, int mode);  // mode 1: IBB links, 2: IBM support
cudaError_t launch_gimem(Ctx &c);
cudaError_t launch_release(Ctx &c);
cudaError_t launch_particle_update(Ctx &c);
cudaError_t launch_markers_place(Ctx &c);
cudaError_t launch_marker_offsets(Ctx &c);
cudaError_t launch_support_mark(Ctx &c);
cudaError_t launch_ibm_passes(Ctx &c);
cudaError_t launch_ibm_particle_sums(Ctx &c, bool init_only);
cudaError_t launch_ibm_rigid_overwrite(Ctx &c);
// rho and u into c.rho_f and c.u_f (FP64); u32, if not null, receives FP32
// records (ux, uy, uz, rho) per cell, alone with rec_only (32- and 16-bit storage)
cudaError_t launch_macro(Ctx &c, float *u32 = nullptr, bool rec_only = false);
cudaError_t launch_mask(Ctx &c);  // statistics velocity: solid cells take the rigid-body velocity
cudaError_t run_spectrum(Ctx &c, int flags, int nbins, double *E, double *D);
cudaError_t run_pipe_profiles(Ctx &c, int flags, int nbins, double *out);
size_t pipe_profile_scratch_bytes(int nbins);
cudaError_t run_tke_budget(Ctx &c, int flags, int nbins, double *out);
// D3Q27 periodic box (q27.cu)
cudaError_t launch_q27_step(Ctx &c);
cudaError_t launch_q27_init(Ctx &c, const double *u_dev, double rho0);
cudaError_t q27_plane_copy(Ctx &c, int i, bool to_f64);
cudaError_t launch_q27_macro(Ctx &c, float4 *rec);
void q27_pipe_colmask(const Ctx &c, std::vector<unsigned> &mask);
cudaError_t launch_q27_coef(Ctx &c);
size_t tke_budget_scratch_bytes(int nbins);
cudaError_t run_stats(Ctx &c, int flags, lbm_stats_t *out);
cudaError_t closure_samples(Ctx &c, double u_scale, float *X, int *cells, long long cap, long long *n_out);
cudaError_t closure_targets(Ctx &c, const int *cells, long long n, double g_scale, float *T);
size_t mlp_pack_bytes();
cudaError_t mlp_pack_device(const float *w, void *pk, cudaStream_t s);
// tensor-core (tcgen05) closure inference, closure_tc.cu
cudaError_t mlp_forward_tc(const float *X, long long n, const float *w, const void *pk, float *Y, int *err,
                           cudaStream_t s);
cudaError_t mlp_train_tc(const float *X, const float *T, long long s0, long long s1, const float *w, const void *pk,
                         float *gpart, float *lpart, int max_blocks, int *err, cudaStream_t s, int *nblk_out);
cudaError_t closure_eps_tc(const Ctx &c, const float *u32, const int *cells, const int *pid, const long long *count,
                           long long cap, const void *pk, float *eps_o, int *err);
}  // namespace lbmgb
