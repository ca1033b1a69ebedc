// batch.cuh -- argument blocks of the kernels and their batched (many slabs, one launch)
// entry points.
//
// Every kernel has a device body that takes its argument block and explicit block
// coordinates.  The single-slab kernel passes blockIdx; the batched kernel walks a work
// list: an op's metadata in device memory is
//     meta = [n, pre[0..N], gx[0..N), sid[0..N)]      (ints, N = slabs the batch holds)
// where participant j (of n <= N) is slab sid[j] (argument block xs[sid[j]]), owns blocks
// pre[j] .. pre[j+1]-1, and its block l has coordinates (l % gx[j], l / gx[j]).  The
// batched grid is fixed (by the largest work list any step can have) and strides over
// the list, so a CUDA graph of the launches stays valid while the participant set shrinks
// as slabs converge; blocks past pre[n] leave at once.
#pragma once
#include <algorithm>
#include "common.cuh"
#include "pair.cuh"
#include "tri_layout.cuh"

namespace trt {

// ---- argument blocks ----
struct OpacityArgs {
    int nx, G;
    const double *T, *edges;
    double s;
    double *sigE, *emis, *sigR;
    float *sig32, *emis32;   // FP32 sweep inputs (sigma_E + 1/(c dt)) h/2, h e/2, or null
    float *kap32;            // FP32 sweep input h/(2 c dt) per cell, or null
    const double *h;
    double icdt;
    const double *otab;      // Problem::otab (sigma_E, sigma_R series scaled by 27 s)
    double kE;               // 27 s C_B: the emission factor of the tabulated path
    const double *Erad;      // radiation energy per cell: sigma_E, sigma_R at T_r, or null
    const int *gate;         // Problem::gate (single-slab kernel only)
    double *cterm;           // Problem::cterm: per-cell terms (single-slab kernel only)
    // the pair form (TRT_LO_PAIR), when otabp is non-null: Problem::otabp and ::cpair (the
    // latter single-slab only), and 1/(c dt) split into two floats on the host
    const fpair *otabp;
    fpair *cpair;
    float icdt_h, icdt_l;
    // for evaluations outside physics.cu: the integrals' tables on the device, and texp's
    const SeriesTables *ser;
    const double *e2;
    ExpConsts ec;
};

struct SweepArgs {
    int nx, N, G, ldG, D;
    double icdt;
    const double *h, *mu, *w, *Iin0, *IinX;
    const void *sigE, *emis;   // [G][nx], SR-typed
    const void *I_old;
    void *I_new;
    void *part;       // [n_dt][2][G][nx], R-typed
    void *psi_exit;   // [M][ldG], R-typed
    double *f, *fb0, *fbX, *C0, *CX;
    const float *kap32;   // h/(2 c dt) per cell in FP32 (with the FP32 inputs), or null
    const float *dir32;   // [M][4] |mu|, |mu|/2, w/2, w mu^2/2 in FP32
    int ntile;            // partial-moment tiles of the finalize
    double *ts;           // paired FP64 sweep: t, s, sum per (|mu|, cell, group), or null
    double *hand;         // paired FP64 sweep: psi of split jobs, then their flags, or null
    int *hand_flag;       // (set by its launcher, with the launch's number)
    int hand_epoch;
    double *tab64;        // paired FP64 sweep: its pre-scaled inputs (2 nx ldG + nx), or null
};

struct FinalizeArgs {
    int nx, N, G, ldG, ntile, nb_cell;
    const void *part, *psi_exit;   // R-typed
    const double *mu, *w, *Iin0, *IinX;
    double *f, *fb0, *fbX, *C0, *CX;
};

struct LoCtx {
    int nx;
    double dt, icdt, idt;   // dt, 1/(c dt), 1/dt
    const double *h, *ihf, *hf;
    const double *hc, *h2, *fwl, *fwr, *hidt, *dxicdt;   // Problem's LO row constants
    const int *lo_slot;
    const fpair *pc;   // Problem::lopc (the pair form's row constants), or null
    Level L;
    const double *a_cell, *s_cell;   // grey: explicit absorption / source per cell
    const int *gate;                 // Problem::gate (single-slab kernels only)
};

struct RestrictCtx {
    int nx, r, n_to;         // r = members per coarse group
    int mode, nt, kc, nchunk;   // RestrictPlan
    const double *h, *ihf;
    Level S;                 // source level (coefficients + solution)
    Level T;                 // target level (written)
    const int *gate;
    int *ticket;             // [n_to][nt + 1], zero between launches (nchunk > 1)
    double *bpart, *part;    // [n_to][nchunk][16] and [n_to][nchunk][12][32 nt]
    // the grey visit's per-cell Newton terms, formed with the cell means when newton != 0
    // (single slab, target = the grey level): into pre [3][nx], with the visit's arguments
    int newton;
    GreyArgs ga;
    double *pre;
    // the target's Eold and Fold sums already hold this step's values (they change only
    // between steps): neither loaded nor summed
    int skip_old;
    int fixed;     // sums kept between the visits of a cycle: 1 store them in fix, 2 take them
    double *fix;   // [n_to][4][32 nt]
};

// How one restriction is split (lo.cu): mode 0, a warp per coarse group; mode 1, a CTA per
// kc members of one, nchunk of them; nt position tiles (and one block of boundary means)
// by gy rows of CTAs.
struct RestrictPlan {
    int mode, nt, kc, nchunk, gy;
};

struct GreyCtx {
    LoCtx lo;
    GreyArgs a;
};

struct CopyArgs {
    double *dst;
    const double *src;
    long n;
};

struct GroupSumArgs {
    int n, nx;
    const double *X;
    double *out;
};

// ---- work-list decoding ----
inline size_t bmeta_ints(int N) { return (size_t)3 * N + 2; }

__device__ inline bool bdecode(const int *__restrict__ meta, int N, int b, int &s, int &bx,
                               int &by)
{
    const int n = meta[0];
    const int *pre = meta + 1;
    const int *gx = meta + 2 + N;
    if (n <= 0 || b >= pre[n]) return false;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pre[mid] <= b)
            lo = mid;
        else
            hi = mid - 1;
    }
    const int l = b - pre[lo];
    bx = l % gx[lo];
    by = l / gx[lo];
    s = meta[2 + 2 * N + lo];
    return true;
}

// ---- host-side argument builders (the single-slab launchers use the same) ----
OpacityArgs make_opacity_args(const Problem &p, const double *T, double *sigE, double *emis,
                              double *sigR, float *sig32, float *emis32, double dt,
                              const double *Erad = nullptr);
cudaError_t launch_cell_terms(const Problem &p, const OpacityArgs &a);   // k_cell_terms
int opacity_blocks(const Problem &p);
int opacity_gx(const Problem &p);   // blocks along the cells (32 cells x 8 groups each)
SweepArgs make_sweep_args(const Problem &p, double dt, const void *sigE, const void *emis,
                          const void *I_old, void *I_new, double *part, double *psi_exit,
                          double *f, double *fb0, double *fbX, double *C0, double *CX, int D);
FinalizeArgs make_finalize_args(const Problem &p, const SweepArgs &a);
int finalize_blocks(const Problem &p);
int pick_D(const Problem &p);   // directions per CTA of the single-slab sweep
LoCtx make_lo_ctx(const Problem &p, double dt, const Level &L);
RestrictPlan restrict_plan(const Problem &p, int n_from, int n_to);
RestrictCtx make_restrict_ctx(const Problem &p, const Level &src, const Level &dst);
GreyCtx make_grey_ctx(const Problem &p, const Level &g, const GreyArgs &a);

// ---- batched launchers (grid: CTAs of the fixed grid; stream: the batch's stream) ----
cudaError_t launch_opacity_b(const int *meta, int N, const OpacityArgs *xs, int grid,
                             cudaStream_t st);
// sweep and its finalize: every participant uses the same R/SR types, D and shape
cudaError_t launch_sweep_b(int precision, bool sigma_fp32, int D, int shape, const int *meta,
                           int N, const SweepArgs *xs, int grid, cudaStream_t st);
cudaError_t launch_finalize_b(int precision, const int *meta, int N, const FinalizeArgs *xs,
                              int grid, cudaStream_t st);
cudaError_t launch_lo_solve_b(int precision, const BatchSmem &bs, const int *meta, int N,
                              const LoCtx *xs, int grid, cudaStream_t st);
cudaError_t launch_restrict_b(const int *meta, int N, const RestrictCtx *xs, int grid,
                              cudaStream_t st);
cudaError_t launch_grey_b(const BatchSmem &bs, const int *meta, int N, const GreyCtx *xs, int grid,
                          cudaStream_t st);
cudaError_t launch_group_sum_b(const int *meta, int N, const GroupSumArgs *xs, int grid,
                               cudaStream_t st);
cudaError_t launch_copy_b(const int *meta, int N, const CopyArgs *xs, int grid, cudaStream_t st);

}  // namespace trt
