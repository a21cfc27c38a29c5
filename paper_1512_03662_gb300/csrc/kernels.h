// Host-side launch interface between the solver engine and the kernels.
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "common.cuh"

namespace jfnk {

// number of kernels launched through the launchers below (profiling aid)
extern long long g_launch_count;

// kModeJvD: the Jacobian-free product times delta, L^-1 (G(X + delta R w) - G(X));
// GMRES takes the 1/delta into its Hessenberg column instead
enum { kModeG = 0, kModeBn = 1, kModeRes = 2, kModeNewton = 3, kModeJv = 4, kModeJvD = 5 };

// device scalar slots (double array `scal` in the workspace)
enum {
    kSlotXhatNorm = 0,   // ||R^-1 X||_2
    kSlotDelta = 1,      // perturbation delta of the current Jv
    kSlotBeta = 2,       // ||b||_2 of the current GMRES cycle
    kSlotRes = 3,        // GMRES residual estimate |g_{j+1}|
    kSlotDxInf = 4,      // ||dxhat||_inf
    kSlotZnorm = 5,      // ||z||_2 of the last preconditioned vector
    kSlotMaxSpeed = 6,   // max |u| + c_s
    kSlotTmp = 7,
    kSlotBeta0 = 8,
    kSlotInvDelta = 9,   // 1/delta of the current Jv (one division, not one per thread)
    kSlotInnerB = 10,    // ||b||_2 of the finest-level SI system of the current preconditioner apply
    kSlotInnerR = 11,    // ||b - A x||_2 after its V-cycles
    kSlotWnorm0 = 12,    // ||w||_2 of the new Arnoldi vector before Gram-Schmidt (selective second pass)
    kNumSlots = 16
};
// counters of finished blocks of the kernels that end in their last block
enum { kCounterZ = 0, kCounterGs = 1, kNumCounters = 2 };

// residual.cu
// p, T and, when the grid has conduction, chi = K0 T^exp per cell
void launch_eos(const Grid& G, const double* X, double* p, double* T, double* chi, cudaStream_t s);
template <typename TZ>
void launch_perturb(const Grid& G, const double* X, const TZ* z, const double* R, const double* scal, int slot,
                    double* Xp, cudaStream_t s);
void launch_face_fluxes(const Grid& G, const double* X, const double* p, const double* T, const double* chi,
                        double* Fm, double* FE, cudaStream_t s);
void launch_mom_fluxes(const Grid& G, const double* X, const double* Fm, double* Psi, cudaStream_t s);
void launch_fluxes(const Grid& G, const double* X, const double* p, const double* T, const double* chi, double* Fm,
                   double* FE, double* Psi, cudaStream_t s);
template <int MODE, typename TO>
void launch_assemble(const Grid& G, const double* X, const double* p, const double* Fm, const double* FE,
                     const double* Psi, const double* bn, const double* G0, const double* Linv, const double* scal,
                     double dt, double* outd, TO* outb, cudaStream_t s);
// also sets the kNumCounters counters to zero
void launch_scaling(const Grid& G, const double* X, double a1, double a2, double* L, double* R, double* Linv,
                    double* Rinv, double* partials, unsigned* counters, cudaStream_t s);
void launch_signal_speed(const Grid& G, const double* X, double* partials, cudaStream_t s);
unsigned cell_blocks(const Grid& G);

// krylov.cu
// finalize: scal[slot] = op(partials[0..n)) with op 0 = sqrt(sum), 1 = sum, 2 = max
// (partials is scratch: a first stage reduces in place)
void launch_finalize(double* partials, int n, double* scal, int slot, int op, cudaStream_t s);
// What the preconditioner's last kernel does with its partial sums of |z|^2: its
// last block sets scal[kSlotZnorm] and, with lambda > 0, the perturbation size
// of pert 0 (launch_delta)
struct ZFinish {
    double* partials;
    unsigned* counter;
    double* scal;
    double lambda;
};
#if defined(__CUDACC__)
__device__ __forceinline__ void set_delta(double* scal, double zn, double lambda) {
    const double d = lambda * (lambda + scal[kSlotXhatNorm] / zn);
    scal[kSlotDelta] = d;
    scal[kSlotInvDelta] = 1.0 / d;
}
// end of a kernel of 128-thread blocks that summed squares: one wave of blocks
// leaves at most kMaxRedBlocks partial sums, which its last block adds
__device__ __forceinline__ void finish_znorm(double sum, double* sh, const ZFinish& Z) {
    const double t = block_sum<128>(sum, sh);
    if (thread_linear() == 0) Z.partials[blockIdx.x] = t;
    if (!last_block(Z.counter, gridDim.x)) return;
    double a = 0.0;
    for (int i = thread_linear(); i < (int)gridDim.x; i += 128) a += __ldcg(Z.partials + i);
    a = block_sum<128>(a, sh);
    if (thread_linear() == 0) {
        const double zn = sqrt(a);
        Z.scal[kSlotZnorm] = zn;
        if (Z.lambda > 0.0) set_delta(Z.scal, zn, Z.lambda);
    }
}
#endif
// delta = lambda (lambda + xhat / ||z||) (pert 0) or the pert_new rule (pert 1,
// uses scal[kSlotTmp] = xhat . z and scal[kSlotZnorm])
void launch_delta(double* scal, double lambda, int pert, cudaStream_t s);
template <typename T>
void launch_norm2_partials(const T* x, long long n, double* partials, cudaStream_t s);
template <typename T>
void launch_dot_partials(const double* a, const double* ainv_scale, const T* b, long long n, double* partials,
                         cudaStream_t s);
// Device scalars of the Gram-Schmidt step that its kernels' last blocks write.
struct GsState {
    double* partials;
    unsigned* counter;       // of blocks done, zero between launches
    double* scal;
    double* vscale;          // lazy scales of the basis vectors
    double *H, *cs, *sn, *g; // Hessenberg columns (leading dimension ldh), rotations, right-hand side
    int ldh;
};
// hcol[i] = vscale[i] <v_i, w>, i < nv
template <typename T>
void launch_multidot(const T* V, long long ld, int nv, const T* w, long long n, const GsState& S, double* hcol,
                     cudaStream_t s);
// w -= sum_i hcol[i] vscale[i] v_i and scal[kSlotTmp] = ||w||.  With column >= 0
// this ends the iteration: hcol is column `column` of H (plus, where given, the
// second pass' coefficients `more`), its subdiagonal entry and the lazy scale
// of the new vector are set, the column is multiplied by
// scal[col_scale_slot] (col_scale_slot >= 0: w was formed as delta J^ z), rotated,
// and scal[kSlotRes] is the residual estimate.
template <typename T>
void launch_axpy_norm(T* w, const T* V, long long ld, int nv, const double* hcol, long long n, const GsState& S,
                      int column, const double* more, int col_scale_slot, cudaStream_t s);
// the end of the iteration alone, ||w|| in scal[kSlotTmp]
void launch_gs_end(const GsState& S, int column, const double* hcol, int col_scale_slot, cudaStream_t s);
void launch_backsolve(const double* H, int ldh, int k, const double* g, double* y, cudaStream_t s);
template <typename T>
void launch_update(double* x, const T* Z, long long ld, int k, const double* y, long long n, cudaStream_t s);
template <typename TS, typename TD>
void launch_scale_copy(const TS* src, double alpha, const double* scal, int slot, int invert, TD* dst, long long n,
                       cudaStream_t s);
void launch_newton_update(double* X, const double* R, const double* dxh, long long n, double* partials,
                          cudaStream_t s);
template <typename T>
void launch_zero(T* x, long long n, cudaStream_t s);
template <typename T>
void launch_restart_residual(T* r, const double* G0, const double* bn, const double* Linv, long long n,
                             cudaStream_t s);
void launch_init_cycle(double* scal, double* g, double* vscale, int m, cudaStream_t s);
// coefficients of the Jacobian-free product for one linearisation:
// P = L^-1 / dt, Q = theta L^-1, C = L^-1 G(X)
void launch_jv_coeffs(const double* Linv, const double* G0, double dt, double theta, double* P, double* Q, double* C,
                      long long n, long long u_begin, cudaStream_t s);

// precond.cu
struct MGLevel {
    int n[3];
    long long ncell;
    void* M;     // nf*nf fields: cell matrix
    void* K;     // nf*ndim fields: coefficient on the lower face over the squared cell width of the level
    void* D;     // nf*nf fields: inverse of the diagonal block (M plus the face coefficients around the cell)
    void* x;     // nf fields
    void* rhs;   // nf fields
    void* r;     // nf fields: residual scratch for the restriction
};

// per-cell coefficient fields of the preconditioner transforms
// PcQ0..PcQ5: FP64 mode: B^-1 entries (b00, b01, b10, b11) applied to
// (r_p, r_e) as the oracle does; FP32 mode: the same map folded with the
// transform, rhs_p = Q0 r_rho + Q1 r_E - Q2 <u.r_u>, rhs_e = Q3 r_rho + Q4 r_E
// - Q5 <u.r_u>, coefficients formed in double so no FP32 cancellation occurs.
enum {
    PcLr = 0, PcLE, PcInvRho, PcE, PcDpdrho, PcDpde, PcInvDpdrho, PcCde,
    PcQ0, PcQ1, PcQ2, PcQ3, PcQ4, PcQ5, PcPr, PcPE, PcRinvR, PcRinvE,
    PcLu, PcU = PcLu + 3, PcInvRhof = PcU + 3, PcThf = PcInvRhof + 3, PcRinvU = PcThf + 3,
    PcNumFields = PcRinvU + 3
};

// Tg, chi: those of k_eos at X
template <typename T>
void launch_pc_setup(const Grid& G, const double* X, const double* Tg, const double* chi, const double* L,
                     const double* Rinv, double dt, int nf, T* C, MGLevel& L0, cudaStream_t s);
// renew only the scaling fields (L and R^-1) of the coefficient array C
template <typename T>
void launch_pc_rescale(const Grid& G, const double* L, const double* Rinv, T* C, cudaStream_t s);
// The transform in also starts the level-0 multigrid unknowns: with nu1 > 0 it
// runs the first red half sweep of the zero start (x = D rhs on the red
// cells; no neighbour counts), otherwise it zeroes x
template <typename T>
void launch_precond_in(const Grid& G, const T* C, const T* v, const double* vscale, int vslot, int nf, T* rp, T* re,
                       T* ru, MGLevel& L0, cudaStream_t s, int nu1);
template <typename T>
void launch_precond_out(const Grid& G, const T* C, double dt, int nf, const T* rp, const T* re, const T* ru,
                        const MGLevel& L0, T* z, const ZFinish& Z, cudaStream_t s);

// multigrid.cu
// D of a level from its M and K
template <typename T>
void launch_block_inverse(const Grid& G, int nf, MGLevel& L, cudaStream_t s);
// M, K and D of level C from those of the finer level F
template <typename T>
void launch_coarsen(const Grid& G, int nf, const MGLevel& F, MGLevel& C, cudaStream_t s);
// half sweep of one colour (0 red, 1 black); tr = 1: the transposed system
// (cell matrices transposed), here and below
template <typename T>
void launch_smooth(const Grid& G, int nf, MGLevel& Lv, int colour, cudaStream_t s, int tr);
// Residual of F to the right-hand side of C.  pre_smoothed: a black half
// sweep was the last on F (the residual is zero on black cells, so red cells
// only are read) and x of C gets the red half sweep of its zero start
// (the solution itself on a single-cell level); otherwise x of C is zeroed
template <typename T>
void launch_restrict(const Grid& G, int nf, MGLevel& F, MGLevel& C, cudaStream_t s, int tr, int pre_smoothed);
template <typename T>
void launch_mg_residual(const Grid& G, int nf, MGLevel& F, cudaStream_t s);
// x_F += P x_C; red_only when a black half sweep follows (it overwrites the
// black cells without reading them)
template <typename T>
void launch_prolong(const Grid& G, int nf, MGLevel& F, MGLevel& C, cudaStream_t s, int red_only);
template <typename T>
void launch_coarsest(int nf, MGLevel& C, cudaStream_t s, int tr);
// Each side of a 2D level in one launch, for levels that tiled_level accepts:
// pre-smoothing (from the second half sweep on where `started`), residual and
// restriction, x left in F.r; prolongation and post-smoothing from F.r to F.x
template <typename T>
bool tiled_level(const Grid& G, int nf, const MGLevel& F, const MGLevel& C, int nu1, int nu2);
template <typename T>
void launch_pre2d(int nf, MGLevel& F, MGLevel& C, int nu1, int started, cudaStream_t s);
template <typename T>
void launch_post2d(const Grid& G, int nf, MGLevel& F, MGLevel& C, int nu2, cudaStream_t s);

// vcycle_cluster.cu
// blocks of the cluster that runs the coarse end of a V-cycle on the current
// device (0: none)
template <typename T>
int vcycle_cluster_ctas(int nf, int nd);
// first level that it takes (levels.size(): none)
template <typename T>
size_t vcycle_cluster_top(int nf, int nd, const std::vector<MGLevel>& levels, int ctas);
// `cycles` V-cycles on the levels levels[0 .. nlev-1], the last one the
// single-cell level; started: the kernel that wrote the right-hand side of
// levels[0] has run the first red half sweep of its zero start
template <typename T>
void launch_vcycle_cluster(const Grid& G, int nf, const MGLevel* levels, int nlev, int nu1, int nu2, int cycles,
                           int started, int ctas, cudaStream_t s, int tr);

// precond_f32.cu: the float transforms of the internal energy form, with L and
// R of the state of the coefficients and an x extent that four divides; C holds
// at most 16 fields of its own, z the velocity rows between in and out, q (one
// field) what the one-field scheme keeps
void launch_pcf_setup(const Grid& G, const double* X, const double* Tg, const double* chi, const double* L,
                      const double* Rinv, double dt, int nf, float* C, MGLevel& L0, cudaStream_t s);
void launch_pcf_in(const Grid& G, const float* C, const float* v, const double* vscale, int vslot, double dt, int nf,
                   float* z, float* q, MGLevel& L0, cudaStream_t s, int nu1);
void launch_pcf_out(const Grid& G, const float* C, int nf, const float* q, const MGLevel& L0, float* z,
                    const ZFinish& Z, cudaStream_t s);

// adjoint.cu
// y = (a dU/dX + b dR/dX)^T w at X (p, T, chi and mass fluxes of X precomputed);
// adj: vjp_scratch_doubles(G) doubles of scratch
void launch_vjp(const Grid& G, const double* X, const double* p, const double* T, const double* chi, const double* Fmh,
                const double* w, double a_u, double b_r, double* adj, double* Xb, cudaStream_t s);
long long vjp_scratch_doubles(const Grid& G);
// partial sums of w_E . (conduction divergence / K0) (T of the state given)
void launch_dRdK0_dot(const Grid& G, const double* T, const double* w, double* partials, cudaStream_t s);
void launch_precondT_out(const Grid& G, const double* C, double dt, int nf, const double* y, double* rub, double* reb,
                         double* rpb, MGLevel& L0, cudaStream_t s, int nu1);
void launch_precondT_in(const Grid& G, const double* C, int nf, const MGLevel& L0, const double* rub,
                        const double* reb, const double* rpb, double* z, cudaStream_t s);
void launch_mul(const double* x, const double* y, double* out, long long n, cudaStream_t s);
void launch_sub(const double* a, const double* b, double* out, long long n, cudaStream_t s);
void launch_mask_walls(const Grid& G, double* v, cudaStream_t s);

}  // namespace jfnk
