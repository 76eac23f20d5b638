// Internal declarations of the GB300 boundary-integral JFNK library.
// Everything here is private to libbfs; the public ABI is include/bfs.h.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "bfs.h"

namespace bfs {

// Per-source record (16 values, FP64 or FP32).  Lengths are in units of dx,
// measured from the mesh centre, so that horizontal offsets between nodes
// and half points are exact in FP32 when dx == dy.
//   0 xs   1 ys   2 zeta/dx   3 (beta+1)/dx
//   4 zeta_x  5 zeta_y  6 beta_x  7 beta_y
//   8 w1 f   9 w2 zeta_x   10 w1 g   11 w2 sigma beta_x
//   12 w1    13 w2   14,15 unused
// with f = phi - x, g = psi - x, w the trapezoid weight, w1 = w/dx^2 (double
// layer, K1 scales as 1/dx^2) and w2 = w/dx (single layer and S2).
constexpr int REC = 16;

// Per-target record (16 values) for the half point (k, l):
//   0 xt  1 yt  2 zeta*/dx  3 (beta*+1)/dx  4 zeta_x*  5 zeta_y*  6 f*  7 g*
//   8 A  9 B  10 C   (S2 coefficients of the free surface at the target)
//   11 zeta*/dx + 1/dx   12 (beta*+1)/dx - 1/dx   13 phi_x*  14 phi_y*  15 unused
constexpr int TREC = 16;

// Double-float records of the df64 pair kernel (hi/lo float pairs from index 2
// on; lengths in mesh units as above).  A source has DSRC floats, sources in
// interleaved pairs:
//   0 column  1 row (mesh units, exact)  2 zeta/dx  4 (beta+1)/dx
//   6 zeta_x  8 zeta_y dy/dx  10 beta_x  12 beta_y dy/dx
//   14 c f  16 c g  18 c dx zeta_x  20 c dx sigma beta_x  22 c  23 unused
// with c = cx cy the trapezoid weight without dx dy.  A target has DTGT floats:
//   0 column  1 row  2 zeta*/dx  4 zeta*/dx + 1/dx  6 (beta*+1)/dx - 1/dx
//   8 (beta*+1)/dx  10 f*  12 g*  14 zeta_x*  16 zeta_y* dy/dx  18,19 unused
constexpr int DSRC = 24, DTGT = 20;
// Heights of either sheet, in mesh cells, up to which the df64 pair kernel takes the
// differences of two of them as they come (pairs_df64.cu); k_records raises d_flag[1]
// where a node of the residual at hand is higher.  DF_EXACT: vertical distances, in
// cells, up to which its form for dx == dy is exact; d_flag[2] where one may be larger.
constexpr float DF_HIGH = 16.f, DF_EXACT = 1447.f;

// Accumulators written by the pair kernels, per split and target:
//   0  double and single layers at top targets (top and bottom sheets)
//   1  sum of w S2 at top targets
//   2  double layers (both sheets) and single layer of the top sheet at bottom targets
constexpr int NACC = 3;

// One instance of a batched sweep as the persistent pair kernel sees it.
struct BatchInst {
    const float *src;
    const float *tgt;
    double *part;
    int *flag;  // the instance's status word (bit 2: a wait timed out)
    int Nt, per_split;
};

struct BatchVariant {
    int tpb, tpt;
};

// One step of the FP32 preconditioner sweeps (apply.cu): the slice k whose
// rows it finishes and the stored blocks (k, m[p]) it multiplies.
//   out 0: y_k = r_k - sum_p B(k, m_p) v_p;  out 1: z_k = sum_p +-B(k, m_p) v_p
//   vec[p] bit 0: v_p is z_{m_p} (else y_{m_p}); bit 1: sign + (else -);
//          bits 2-3: where a thread finds its columns of v_p (SW_EARLY, SW_WIN,
//          SW_CRIT); bits 4-5: the register-window index (SW_WIN)
//   uid[p]: the task that wrote v_p (tasks are numbered group 0 first)
constexpr int SW_BMAX = 7;  // blocks per task: half bands up to 6
constexpr int SW_HW = 2;  // register window: the last SW_HW critical vectors
enum { SW_EARLY = 0, SW_WIN = 1, SW_CRIT = 2 };
struct SweepTask {
    int k, out, nblk;
    int m[SW_BMAX], vec[SW_BMAX], uid[SW_BMAX];
};

// A task as the kernel reads it, in 16-byte words: head {k, out, nblk, order} and
// per block {m, word offset of its vector from y, uid, 0}, blocks in the order
// SW_WIN (newest first), SW_EARLY, SW_CRIT.  order: bits 0-1 the register-window
// entries used, bit 2 a critical block, bit 4 + p the sign of block p (1: plus).
struct SweepDev {
    int4 head;
    int4 blk[SW_BMAX];
};

struct SweepPlan {
    int twist = -1;          // first middle slice of the two-ended order, or -1
    int groups = 1;          // chains run side by side (CTA groups)
    int ntask[2] = {0, 0};   // tasks per group
    std::vector<SweepTask> tasks;
};

struct PairPlan {
    int tpb;        // threads per CTA
    int tpt;        // targets per thread
    int chunk;      // sources staged per shared-memory chunk
    int splits;     // source splits (grid.y)
    int per_split;  // sources per split (multiple of chunk)
    int tiles;      // target tiles (grid.x)
};

}  // namespace bfs

struct bfs_ctx {
    // problem
    int N, M, half;
    double x1, y1, dx, dy, F;
    double beta_max;  // highest bottom node; a valid F keeps it below F^2/2
    bfs_options opt;
    int n, Nt, NM, Ns, Ns_cap;
    double xc, yc;  // centre of the mesh (physical)
    int device;

    // residual buffers
    double *d_beta, *d_bx, *d_by;  // NM each
    double *d_nodal;               // 8 NM: zeta, zx, zy, phi, phx, phy, psi, psx
    double *d_src64;               // Ns_cap * REC
    float *d_src32;                // Ns_cap * REC
    double *d_tgt64;               // Nt * TREC
    float *d_tgt32;                // Nt * TREC
    double *d_part;                // max splits * NACC * Nt
    double *d_constB;              // Nt: bottom-only single-layer part at bottom targets
    double *d_psurf;               // NM applied surface pressure, or nullptr
    int *d_flag;                   // [0] non-finite and timeout flags; [1] DF_HIGH, [2] DF_EXACT exceeded
    float *d_srcdf;                // Ns_cap * DSRC double-float source records
    float *d_tgtdf;                // Nt * DTGT double-float target records
    bfs::PairPlan plan64, plan32, plandf;
    size_t part_cap;

    // Jacobian-vector product scratch
    double *d_up, *d_Fp;  // n each
    double *d_scal;       // 16 scalars

    // Newton / GMRES workspace
    int stop_at_tol;  // bfs_set_stop_at_tol
    int m_alloc;
    double *d_V;      // (m+1) n Krylov basis
    double *d_Z;      // m n preconditioned basis vectors z_j = P^-1 v_j
    double *d_H;      // Hessenberg, column j at d_H + j (m+1)
    double *d_giv;    // cs[m], sn[m], g[m+1], y[m], h[m+1], h2[m+1]
    double *d_red;    // reduction partials
    unsigned int *d_tailbar;  // grid barrier of the fused Arnoldi tail
    int tail_grid;            // its grid (0: the kernels one by one)
    double *d_sbase;  // one allocation holding the n-vectors below
    double *d_F, *d_du, *d_ut, *d_Ft, *d_w, *d_F32, *d_uio;  // n each
    double *h_pin;    // pinned host scalars

    // preconditioner
    int pc_ready, pc_h, nb, apply_grid;
    double *d_pc;      // M * (2h+1) * nb * nb  block-banded factors
    float *d_pc32;     // FP32 copy of d_pc (precond_precision FP32C)
    unsigned long long *d_flow;  // tagged y and z of the FP32 sweeps, 2 M nb, then the tag word
    unsigned long long flow_count;  // FP32 sweep launches since the tags were reset
    int capturing;               // a CUDA graph is being captured on the solver stream
    int pc_twist;                // two-ended factor order: first middle slice; -1: one-ended
    bfs::SweepDev *d_tasks;      // task table of the FP32 sweeps
    std::vector<bfs::SweepDev> h_tasks;
    int sweep_table;             // 1: the task-table kernel runs the FP32 sweeps
    int sweep_groups, sweep_ntask[2], sweep_ntags, sweep_nslot;
    int sweep_gg, sweep_sw, sweep_wpt, sweep_nq, sweep_rows, sweep_bm;  // shape of the task-table kernel
    int flow_vs;                 // words of a slice of the tagged vectors
    size_t sweep_dyn;
    int dbg_stall_task;          // test hook: task whose first wait is made unsatisfiable, or -1
    int dbg_stall_skip;          // sweep launches before that one

    // Arnoldi steps of bfs_solve replayed as CUDA graphs, one per (Krylov
    // index j, base residual buffer); cleared whenever a captured argument
    // could change (factor, F, topography, surface pressure, u buffer)
    std::vector<cudaGraphExec_t> gm_exec;
    std::vector<unsigned long long> gm_nlaunch, gm_nflow;
    // gm_iscond[key]: the step sits in a conditional node behind a guard that
    // reads the device-side end-of-cycle flag, so the next step can be queued
    // before this one's scalars reach the host; gm_cond: 1 while such graphs
    // instantiate, -1 once one failed (plain step graphs from then on)
    std::vector<char> gm_iscond;
    int gm_cond;
    cudaEvent_t gm_ev;
    // solves handed the legacy default stream run here (graph capture needs a
    // stream of its own), joined to the caller's stream by join_ev
    cudaStream_t own_stream;
    cudaEvent_t join_ev;
    const double *gm_u;
    int gm_warm, gm_disabled;
    int ldp32;                   // padded row length of d_pc32
    int flow_checked;
    double *d_gj;      // Gauss-Jordan work matrices and GEMM scratch
    void *d_slices;    // operand slices of sg_gemm, while factoring
    void *d_gjscr;     // dataflow Gauss-Jordan: candidate slots, perm / pinv
    double *d_gjdata;  // dataflow Gauss-Jordan: candidate rows
    double *d_rowsum5; // Nt
    // condensed slice blocks (condense.cu): phi_x eliminated, nb = 2 (N+1) + 1
    int pc_cond;
    double pc_F;       // Froude number the preconditioner was factored for
    double *d_ktab;    // tables of K5, K7, K6, then scratch and K6 in float pairs
    double *d_rc, *d_zc;  // reduced right-hand side and solution, M nb each
    int *d_pivflag;
    double *d_perm_a, *d_perm_b;  // n each

    // profiling: launch counter and CUDA-event timing of the pair kernels
    unsigned long long launches;
    int prof_on;
    std::vector<cudaEvent_t> ev_pool;
    std::vector<int> ev_kind;  // per recorded pair: 0 FP64, 1 FP32C
    size_t ev_used;

    std::string err;
};

namespace bfs {

// residual.cu
int residual_launch(bfs_ctx *c, const double *u, double *Fu, int precision, cudaStream_t s);
// which: record copies to write, bit 0 FP64, bit 1 FP32, bit 2 double-float
int unpack_launch(bfs_ctx *c, const double *u, cudaStream_t s, int which = 3);
int constB_launch(bfs_ctx *c, cudaStream_t s);
PairPlan make_plan(int Nt, int Ns, int tpb, int tpt, int chunk, int splits_req, int sms);
PairPlan fine_plan(int Nt, int Ns, int tpb, int unit, int per_sm, int splits_req, int sms);
PairPlan plan64_fine(int Nt, int Ns, int splits_req, int sms);
void plans_for(int Nt, int Ns, int splits_req, int sms, PairPlan *p64, PairPlan *p32);

int finish_launch(bfs_ctx *c, double *Fu, int precision, cudaStream_t s);

// apply.cu
int precond_make_f32(bfs_ctx *c, cudaStream_t s);
int apply_flow_launch(bfs_ctx *c, const double *r, double *z, cudaStream_t s);
int flow_wrap_check(bfs_ctx *c, cudaStream_t s);
int flow_reset(bfs_ctx *c, cudaStream_t s);
int sweep_plan(int M, int h, int twisted, SweepPlan &P);
int sweep_twist_ok(bfs_ctx *c, int h);
extern const BatchVariant kBatchVariants[];
extern const int kNumBatchVariants;
int batch_pairs_occupancy(int v, int *blocks_per_sm);
void batch_pairs_launch(int v, int grid, const BatchInst *inst, const int4 *items, int n_items,
                        unsigned int *counter, const unsigned char *mask, cudaStream_t s);

// slice_gemm.cu
void sg_alloc(bfs_ctx *c);
int sg_gemm(bfs_ctx *c, const std::vector<const double *> &A, const std::vector<const double *> &B,
            const std::vector<double *> &C, double alpha, double beta, cudaStream_t s);

// condense.cu
int cond_ok(const bfs_ctx *c);
int cond_fits(const bfs_ctx *c, int h);
int cond_tables(bfs_ctx *c, cudaStream_t s);
int cond_form(bfs_ctx *c, cudaStream_t s);
int cond_pre(bfs_ctx *c, const double *r, cudaStream_t s);
int cond_post(bfs_ctx *c, const double *r, double *z, bool pairs, cudaStream_t s);

// pairs_df64.cu
PairPlan plan_df(int Nt, int Ns, int splits_req, int sms);
int pairs_df_launch(bfs_ctx *c, cudaStream_t s);

// solver.cu
// GMRES state of one instance between device phases (see solver.cu).
struct Gm {
    enum State { BEGIN, ARNOLDI, CYCLE_END, RESTART, DONE };
    const double *u, *F, *Fbase;
    double target, res;
    int maxit, its, j, status, precs, jvs;
    State state;
};
double gm_last_eta(const bfs_ctx *c, double finf, double eta);
constexpr double GM_EXTRA_ETA = 0.2;
constexpr int GM_EXTRA_ITS = 12;
bool gm_extra_step(const bfs_ctx *c, int k, double finf);
int gm_extra_drop(bfs_ctx *c, cudaStream_t s);
void gm_start(bfs_ctx *c, Gm &g, const double *u, const double *F, const double *Fbase,
              double fnorm2, double eta, int maxit, cudaStream_t s);
void gm_cycle_begin(bfs_ctx *c, Gm &g, double beta, cudaStream_t s);
int gm_arnoldi_pre(bfs_ctx *c, Gm &g, cudaStream_t s);
int gm_arnoldi_sweep(bfs_ctx *c, Gm &g, cudaStream_t s);
// several instances' Arnoldi steps at once (up to GM_BMAX per launch)
constexpr int GM_BMAX = 64;
int gm_multi_pre(bfs_ctx *const *cs, Gm *const *gs, int cnt, cudaStream_t s);
int gm_multi_post(bfs_ctx *const *cs, Gm *const *gs, int cnt, cudaStream_t s);
int gm_arnoldi_post(bfs_ctx *c, Gm &g, cudaStream_t s);
void gm_arnoldi_host(bfs_ctx *c, Gm &g, double hn, double res);
int gm_cycle_end(bfs_ctx *c, Gm &g, cudaStream_t s);
int gm_restart_post(bfs_ctx *c, Gm &g, cudaStream_t s);
int jv_prep(bfs_ctx *c, const double *u, const double *z, double h, int precision, cudaStream_t s,
            bool unorm_ready);
int jv_post(bfs_ctx *c, const double *Fu, double *Jz, cudaStream_t s);
void solver_axpby(bfs_ctx *c, double *y, const double *x, const double *z, double a, double b,
                  cudaStream_t s);
int jvp_launch(bfs_ctx *c, const double *u, const double *Fu, const double *z, double *Jz,
               double h, int precision, cudaStream_t s, bool unorm_ready = false);
int solve_device(bfs_ctx *c, double *u, bfs_stats *st, cudaStream_t s);
void gm_graphs_clear(bfs_ctx *c);
int alloc_solver(bfs_ctx *c);
void free_solver(bfs_ctx *c);
void norms_launch(bfs_ctx *c, const double *v, int n, double *d_out2, double *d_outinf, cudaStream_t s);

// precond.cu
int precond_factor(bfs_ctx *c, int half_band, cudaStream_t s);
int precond_apply(bfs_ctx *c, const double *r, double *z, cudaStream_t s);
void precond_free(bfs_ctx *c);

int num_sms(int device);
// records an event pair around a pair-kernel launch when profiling is on
cudaEvent_t prof_event(bfs_ctx *c);
// Packed FP32x2 arithmetic of sm_100-class GPUs: one instruction applies the
// same operation to two values (low and high half of a 64-bit register pair).
struct f2 {
    unsigned long long v;
};
__device__ __forceinline__ f2 f2_pack(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 x, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;" : "=l"(d.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return d;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b)
{
    f2 d;
    asm("sub.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.ftz.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
// sign flip of both halves: integer operations, off the FMA pipe
__device__ __forceinline__ f2 f2_neg(f2 a) { return f2{a.v ^ 0x8000000080000000ull}; }
__device__ __forceinline__ f2 f2_both(float a) { return f2_pack(a, a); }
__device__ __forceinline__ f2 f2_rsq(f2 x)
{
    float a, b;
    f2_unpack(x, a, b);
    return f2_pack(rsqrtf(a), rsqrtf(b));
}

}  // namespace bfs

// An allocation: no memory is BFS_ENOMEM, and not an error that the next launch would find.
#define BFS_ALLOC_TRY(ctx, call)                                                     \
    do {                                                                             \
        cudaError_t e_ = (call);                                                     \
        if (e_ != cudaSuccess) {                                                     \
            cudaGetLastError();                                                      \
            (ctx)->err = std::string(#call) + ": " + cudaGetErrorString(e_);         \
            return e_ == cudaErrorMemoryAllocation ? BFS_ENOMEM : BFS_ECUDA;         \
        }                                                                            \
    } while (0)

#define BFS_CUDA_TRY(ctx, call)                                                      \
    do {                                                                             \
        cudaError_t e_ = (call);                                                     \
        if (e_ != cudaSuccess) {                                                     \
            (ctx)->err = std::string(#call) + ": " + cudaGetErrorString(e_);         \
            return BFS_ECUDA;                                                        \
        }                                                                            \
    } while (0)
