// Internal launch interface between api.cu and the kernels' files (form.cu, form_tile.cu,
// pcg.cu, pcg_reg.cu, pcg_split.cu, pcg_cta.cu).
#pragma once

#include "common.cuh"

namespace mpcg {

template <typename T>
struct SchurArgs {
    int nx, nu;
    BatchView bv;
    int Kgrid;  // host-side upper bound on the total knots (grid size only)
    const T *A, *B, *Qd, *Rd, *q, *r, *c;
    const T *Qf, *Rf;  // dense SPD cost blocks (nullptr: diagonal Qd, Rd)
    T *Sd, *So, *gamma;
    unsigned *info;
};

template <typename T>
struct PcgParams {
    int nx;
    BatchView bv;
    const T *Sd, *So, *Pd, *Po;
    const T *rhs;  // b = rhs_sign * rhs
    T rhs_sign;
    T *lam;
    const unsigned *info;
    mpcg_stats *stats;
    int *queue;       // instance counters, one per group level (nullptr: static round robin)
    int pick;         // pcg_reg_kernel: 1 / -1: this launch serves batches of more / at most `work`;
                      // pcg_tile_kernel: batches that clusters / one CTA each serve faster
    int pick_C, pick_m, pick_n;  // pcg_tile_kernel, with pick: CTAs per cluster, clusters and CTAs at a time
    int pick_packed;             // ... does the form with one CTA stream packed blocks?
    long long work;
    int n_above, n_upto;  // pcg_reg_kernel: the horizons this launch takes, (n_above, n_upto]
    int split;        // pcg_reg_kernel: clusters split into groups for shorter horizons;
                      // pcg_tile_kernel: instances by quarters of n_long, long ones first
    int n_long;       // the longest horizon of the launch (pcg_tile_kernel; with pick)
    const int *inst_list;  // tickets -> instances (nullptr: ticket t is instance t)
    int n_tickets;         // instances to solve (B, or the list's length)
    double tol;
    int tol_mode;
    int max_iter;     // <= 0: 10 N nx
    int precon;       // 0: symmetric stair Phi^-1 (Pd, Po); 1: block Jacobi (Pd only)
    int kpc_max;      // knot slots per CTA (blockDim.x / LPK)
    int stage_smem;   // pcg_cluster_kernel: stage blocks in shared memory
    int vs;           // shared vector stride (elements per knot)
    int depth;        // pcg_tile_kernel: steps each knot stream copies ahead
    const T *Sdp, *Pdp;  // pcg_tile_kernel: packed diagonal blocks (nullptr: full Sd, Pd)
    int npk;             // entries per packed diagonal block
};

// Instance counters of one launch (int each): a level per group size
constexpr int QUEUE_LEVELS = 8;

struct PcgLaunch {
    int cta_mode;  // 0: cluster per instance (pcg_reg_kernel when reg, else
                   // pcg_cluster_kernel); 1: one CTA per instance, blocks from L2
                   // (pcg_cta_kernel); 2: one CTA per instance, blocks streamed as
                   // TMA tiles (pcg_tile_kernel)
    int C;         // CTAs per cluster
    int clusters;  // clusters in the grid
    int threads;   // threads per CTA
    int lpk, rpt, stage, vs, kpc_max;
    int reg;       // cluster form with resident operators (float32, nx = 14): 1 both in
                   // registers, 2 Phi^-1 in shared memory, two CTAs per SM
    int split_rows; // cluster form with rows split over lanes (pcg_split.cu): its variant, 0 none
    // reg == 2: the form in registers too, and the work from which the batch is
    // not its own (clusters > 0: the device chooses, see pcg_reg.cu)
    struct {
        int C, clusters, n_mid, n_low, split, kpc_max, threads;
        size_t smem;
        long long work;
    } light;
    int n_mid, n_low;  // reg: clusters of the later stages, 3/4 and 1/2 of the full
                   // size (0: one launch; see pcg_reg.cu)
    int no_queue;  // instances that need no queue in another form of the launch, and so
                   // no workspace in this one either (they are dealt out in turn)
    int n_cta;     // tiled: instances that one CTA each takes at a time
    // tiled with C > 1: the form with one CTA per instance, where the device chooses
    // by the horizons (clusters > 0), and the clusters at a time of this one
    struct {
        int clusters, kpc_max, threads, depth, pk, m;
        size_t smem;
    } one;
    int split;     // reg: one counter per group level, clusters split (see pcg_reg.cu);
                   // tiled: long horizons first (one counter per quarter of n_long)
    int n_long;    // tiled, reg with light: the longest horizon the launch is sized for
    int vw;        // pcg_tile_kernel: elements per shared-memory row load (2 or 4)
    int depth;     // pcg_tile_kernel: steps each knot stream copies ahead (1..4)
    int nxc;       // pcg_tile_kernel: nx fixed at compile time (14, 36), else 0
    int pk;        // pcg_tile_kernel: streams the packed diagonal blocks (nx = 36)
    int dot;       // float32 only: 1 accumulates the dot products in float64 (AccF64)
    size_t smem;
};

template <typename T> cudaError_t launch_form_schur(const SchurArgs<T> &, cudaStream_t);
template <typename T>
cudaError_t launch_form_precon(int nx, BatchView bv, int Kgrid, const T *Sd, const T *So, T *Pd,
                               T *Po, cudaStream_t s);
template <typename T>
cudaError_t launch_recover(int nx, int nu, BatchView bv, int Kgrid, const T *A, const T *B,
                           const T *Qd, const T *Rd, const T *hx, const T *hu, const T *v, T *zx,
                           T *zu, cudaStream_t s);
template <typename T>
cudaError_t launch_recover_dense(int nx, int nu, BatchView bv, int Kgrid, const T *A, const T *B,
                                 const T *Qf, const T *Rf, const T *hx, const T *hu, const T *v,
                                 T *zx, T *zu, cudaStream_t s);
// the same for float32 nx = 14, nu = 7 (form_tile.cu)
cudaError_t launch_recover_dense_14(BatchView bv, int Kgrid, const float *A, const float *B, const float *Qf,
                                    const float *Rf, const float *hx, const float *hu, const float *v, float *zx,
                                    float *zu, cudaStream_t s);
template <typename T>
cudaError_t launch_cgh(int nx, int nu, BatchView bv, int Kgrid, const T *A, const T *B,
                       const T *Qd, const T *Rd, const T *hx, const T *hu, const T *w, T *out,
                       cudaStream_t s);
template <typename T>
cudaError_t launch_grad(int nx, int nu, BatchView bv, int Kgrid, const T *lam, const T *mu,
                        const T *dx, const T *du, const T *gq, const T *gr, T *gA, T *gB, T *gQd,
                        T *gRd, T *gc, cudaStream_t s);
template <typename T>
cudaError_t launch_resid(int nx, int nu, BatchView bv, int Kgrid, const T *A, const T *B, const T *Qd,
                         const T *Rd, const T *q, const T *r, const T *c, T csign, const T *lam,
                         T *out, cudaStream_t s);
template <typename T>
cudaError_t launch_axpy(int nx, BatchView bv, int Kgrid, const T *d, T *lam, cudaStream_t s);
template <typename T>
cudaError_t launch_zero(int nx, BatchView bv, int Kgrid, T *v, cudaStream_t s);
template <typename T>
cudaError_t launch_pack_diag(int nx, int npk, BatchView bv, int Kgrid, const T *D, T *Dp, cudaStream_t s);
// entries per packed diagonal block: nx(nx+1)/2 rounded up to 4 (16 bytes)
__host__ __device__ __forceinline__ int packed_len(int nx) { return (nx * (nx + 1) / 2 + 3) / 4 * 4; }
template <typename T> cudaError_t pcg_launch(const PcgLaunch &, const PcgParams<T> &, cudaStream_t);
template <typename T> int pcg_max_clusters(const PcgLaunch &);
cudaError_t pcg_prepare(int smem_optin);
cudaError_t pcg_reg_launch(const PcgLaunch &, const PcgParams<float> &, cudaStream_t);
int pcg_reg_max_clusters(const PcgLaunch &);
size_t pcg_reg_smem_bytes(const PcgLaunch &);
cudaError_t pcg_reg_prepare(int smem_optin);
// sets L to pcg_split.cu's shape for C CTAs; co-resident clusters (0: not its shape)
template <typename T> int pcg_split_shape(int nx, int N, int C, PcgLaunch &L);
template <typename T> cudaError_t pcg_split_launch(const PcgLaunch &, const PcgParams<T> &, cudaStream_t);
cudaError_t pcg_split_prepare(int smem_optin);
cudaError_t pcg_cta_prepare(int smem_optin);
cudaError_t pcg_tile_prepare(int smem_optin);
template <typename T>
size_t pcg_tile_smem_bytes(int nmax, int vs, int W, int NS, int nx, int depth, int npk, bool cluster);
template <typename T> cudaError_t pcg_tile_launch(const PcgLaunch &, const PcgParams<T> &, cudaStream_t);
template <typename T> int pcg_tile_max_clusters(const PcgLaunch &, int sms);
// nx = 36, B instances of N knots each: clusters of C CTAs, m at a time, rather than one
// CTA each, n at a time?
bool tile_clusters_pay_when_equal(int N, int B, int C, int m, int n, bool packed);
template <typename T> size_t pcg_cta_smem_bytes(int nmax, int vs, int W);
template <typename T> cudaError_t pcg_cta_launch(const PcgLaunch &, const PcgParams<T> &, cudaStream_t);
template <typename T> int pcg_cta_max_blocks(const PcgLaunch &);
cudaError_t form_prepare(int smem_optin);
template <typename T> size_t pcg_smem_bytes(int kpc_max, int vs, int C, int W, int nx, int stage, int dot);

}  // namespace mpcg
