// Finite-volume right-hand side R_U(X) of the paper's Sect. 2 on the
// staggered grid, and the residual-type operators built from it:
//   G(X)  = U(X)/dt - theta R_U(X)                 (Jv, Newton set-up)
//   b^n   = U(X^n)/dt + (1-theta) R_U(X^n)          (Eq. crank_nicholson)
//   F_U   = G(X) - b^n
//   Jv    = L^-1 [G(X + delta R v) - G(X)] / delta   (Eqs. jacobian_free, pert_old)
//
// The evaluation is split so that every van Leer slope and every flux is
// computed once per slot (the FP64 rate of sm_103a, about 0.6 TFMA/s, binds
// these kernels, not HBM).  The flux kernels form their products and limited
// slopes on the integer pipes (emu64.cuh: one rounding each, checked once per
// evaluation, redone on the FP64 pipe where an operand left the range) and
// address neighbours by constant offsets away from the ends of the grid
// (NbIn, common.cuh), so the FP64 pipe keeps the sums only:
//   k_eos          p, T per cell (perturbed state written first by k_perturb)
//   k_face_fluxes  mass flux Fm_d and energy flux FE_d (advective part minus
//                  conduction) on the lower face of every cell, per direction
//   k_mom_fluxes   momentum fluxes Psi_cd: for c == d at cell centres, for
//                  c != d on the edges between faces; stored doubled (carried
//                  by the sum of two mass fluxes, not their mean: exact, and
//                  the assemble takes the 1/2 into 1/(2 dx))
//   k_assemble     divergences, sources, U(X) and the requested combination
//
// Reconstruction (van Leer 1974): slope 2ab/(a+b) if ab > 0 else 0; the
// upwind face value is q_L + s_L/2 when the upwinding speed is >= 0, else
// q_R - s_R/2.  Only the slope on the upwind side is evaluated.
#include "common.cuh"
#include "kernels.h"

namespace jfnk {

long long g_launch_count = 0;

template <typename TZ>
__global__ void k_perturb(Grid G, const double* X, const TZ* z,
                          const double* R, const double* scal, int delta_slot,
                          double* Xp, long long nvec) {
    pdl_wait();
    long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= nvec) return;
    const double delta = scal[delta_slot];
    // R_rho = rho and R_e = e (Eq. jacobian_system_norm; k_scaling stores
    // them as copies of X): the density and energy rows take R from X
    // instead of reading it again
    const double x = X[k];
    const double r = k < 2 * G.ncell ? x : R[k];
    Xp[k] = x + delta * (r * to_f64(z[k]));
}

__device__ __forceinline__ double conductivity(const Grid& G, double T) {
    return G.chi3 ? G.K0 * (T * T * T) : G.K0 * pow(T, G.chi_exp);
}

// p, T and (with conduction) chi = K0 T^exp per cell, each formed once for
// all the faces that use it.  This kernel stays on the FP64 pipe: it is
// bound by memory latency, and its six products on the integer pipes made
// it slower (0.20 -> 0.23 ms at 256^3, the ALU pipe 74 % busy).
template <int ND>
__global__ void k_eos(Grid G, const double* X, double* p, double* T,
                      double* chi) {
    pdl_wait();
    Idx3 P;
    long long c;
    if (!cell_pos(G.n, P, c)) return;
    const long long nc = G.ncell;
    double rho = X[c];
    double e = X[nc + c];
    if (G.energy_form == 1) {
        double ke = 0.0;
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const double* u = X + (2 + d) * nc + c;
            const double ul = normal_along(G, u, P, d, 0);
            const double uu = normal_along(G, u, P, d, 1);
            ke = ke + 0.25 * (ul * ul + uu * uu);
        }
        e = e - ke;
    }
    p[c] = G.gm1 * rho * e;
    const double Tc = G.gm1 * e;
    T[c] = Tc;
    if (G.has_cond) chi[c] = conductivity(G, Tc);
}

// Mass and energy flux of the lower face of direction d of one cell (its
// own reciprocal batch of two); with checked Ops nothing is written unless
// every operation was in range.
template <int ND, int EF, class O, class N>
__device__ __forceinline__ bool face_flux_dir(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                              const double* __restrict__ p, const double* __restrict__ T,
                                              const double* __restrict__ chi, double* __restrict__ Fm,
                                              double* __restrict__ FE, int d, long long c) {
    const long long nc = G.ncell;
    const double* rho = X + c;
    const double* E = X + nc + c;
    const double u = nb.along(X + (2 + d) * nc + c, d, 0);
    const int om2 = nb.off(d, -2), om1 = nb.off(d, -1), op1 = nb.off(d, 1);
    const double r0 = *rho, e0 = *E;
    const double r2 = rho[om2], e2 = E[om2];
    const double r1 = rho[om1], e1 = E[om1];
    const double r3 = rho[op1], e3 = E[op1];
    // upwind side: cell i-1 for u >= 0 (ties to the lower side), else cell i
    const bool left = nonneg(u);
    const Stencil st[2] = {{left ? r1 : r0, left ? r2 : r3, left ? r0 : r1},
                           {left ? e1 : e0, left ? e2 : e3, left ? e0 : e1}};
    double up[2];
    upwind_values<2>(st, up, ops);
    const double fm = ops.mul(u, up[0]);
    double fe = ops.mul(fm, up[1]);
    if constexpr (EF == 1) {
        const double pl = p[c + om1];
        fe = fe + 0.5 * (pl + p[c]) * u;
    }
    if (G.has_cond) {
        // q = chi_f (T_c - T_l) / dx with chi_f the mean of the two cells
        const double Tl = T[c + om1];
        const double chil = chi[c + om1];
        const double sq = ops.mul(chil + chi[c], G.hidx[d]);
        fe = fma(-sq, T[c] - Tl, fe);
    }
    if (!ops.valid()) return false;
    Fm[d * nc + c] = fm;                  // mass flux (every consumer takes half the sum of two)
    FE[d * nc + c] = fe;
    return true;
}

// products of the face fluxes on the integer pipes, sums on the FP64 pipe
using FaceOps = IntOps;

// the FP64-pipe redo of one direction, out of line: inlined, the compiler
// predicates part of it into the fast path, where its FP64 instructions
// still occupy the FP64 pipe with every lane switched off
template <int ND, int EF>
__device__ __noinline__ void face_flux_dir_fp64(const Grid G, const double* __restrict__ X,
                                                const double* __restrict__ p, const double* __restrict__ T,
                                                const double* __restrict__ chi, double* __restrict__ Fm,
                                                double* __restrict__ FE, int d, const Idx3 P, long long c) {
    face_flux_dir<ND, EF>(FpOps(), NbGen(G, P), G, X, p, T, chi, Fm, FE, d, c);
}

template <int ND, int EF, class N>
__device__ __forceinline__ void face_fluxes_cell(const N& nb, const Grid& G, const double* __restrict__ X,
                                                 const double* __restrict__ p, const double* __restrict__ T,
                                                 const double* __restrict__ chi, double* __restrict__ Fm,
                                                 double* __restrict__ FE, const Idx3& P, long long c) {
#pragma unroll 1
    for (int d = 0; d < ND; ++d)
        if (!face_flux_dir<ND, EF>(FaceOps(), nb, G, X, p, T, chi, Fm, FE, d, c))
            face_flux_dir_fp64<ND, EF>(G, X, p, T, chi, Fm, FE, d, P, c);
}

// One direction at a time in a loop that is not unrolled, at least 10 blocks of
// 128 threads per SM (48 registers): 124 us at 128^3, against 146 us unrolled
// with 6 blocks (latency: 35 % of the warps resident) and 176 us with the
// products and a batched reciprocal in place of harm_mid and one neighbour
// form.  The FP64 pipe (27 instructions per cell) is 76 % busy, the ALU pipe
// 72 %.  The energy form EF (0: internal, 1: total) is a template parameter: as
// a runtime test its pressure-work term was predicated, and its FP64
// instructions occupied the FP64 pipe with every lane off.
template <int ND, int EF>
__global__ void __launch_bounds__(128, 10) k_face_fluxes(Grid G, const double* X, const double* p,
                              const double* T, const double* chi, double* Fm,
                              double* FE) {
    pdl_wait();
    Idx3 P;
    long long c;
    if (!cell_pos(G.n, P, c)) return;
    if (inner_block<ND>(G)) face_fluxes_cell<ND, EF>(NbIn(G, P), G, X, p, T, chi, Fm, FE, P, c);
    else face_fluxes_cell<ND, EF>(NbGen(G, P), G, X, p, T, chi, Fm, FE, P, c);
}

// Momentum flux Psi_cd of one cell; with checked Ops nothing is written unless
// every operation was in range.
template <int ND, class O, class N>
__device__ __forceinline__ bool mom_flux(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                         const double* __restrict__ Fm, double* __restrict__ Psi, int c, int d,
                                         long long cc) {
    const long long nc = G.ncell;
    const double* uc = X + (2 + c) * nc + cc;         // pointers at the thread's own slot
    const double* fmd = Fm + d * nc + cc;
    double m, q0, q1, q2, q3;                         // q0..q3 along d, the flux between q1 and q2
    if (c == d) {
        // flux at the cell centre between faces i and i+1 along c, carried
        // by the mean of the two mass fluxes (here their sum: Psi doubled)
        m = *fmd + nb.up(fmd, c);
        q0 = nb.along(uc, c, -1);
        q1 = nb.along(uc, c, 0);
        q2 = nb.along(uc, c, 1);
        q3 = nb.along(uc, c, 2);
    } else {
        // flux on the edge between c-face i_c and d-face i_d
        m = fmd[nb.off(c, -1)] + *fmd;
        q0 = nb.across(uc, c, d, -2);
        q1 = nb.across(uc, c, d, -1);
        q2 = nb.across(uc, c, d, 0);
        q3 = nb.across(uc, c, d, 1);
    }
    const bool left = nonneg(m);
    const Stencil st[1] = {{left ? q1 : q2, left ? q0 : q3, left ? q2 : q1}};
    double up[1];
    upwind_values<1>(st, up, ops);
    const double psi = ops.mul(m, up[0]);
    if (!ops.valid()) return false;
    Psi[(c * ND + d) * nc + cc] = psi;
    return true;
}

// products of the momentum fluxes on the integer pipes, sums on the FP64 pipe
using MomOps = IntOps;

// the FP64-pipe redo of one flux, out of line (see face_flux_dir_fp64)
template <int ND>
__device__ __noinline__ void mom_flux_fp64(const Grid G, const double* __restrict__ X, const double* __restrict__ Fm,
                                           double* __restrict__ Psi, int c, int d, const Idx3 P, long long cc) {
    mom_flux<ND>(FpOps(), NbGen(G, P), G, X, Fm, Psi, c, d, cc);
}

// The components run as a loop that is not unrolled, which keeps the
// straight-line code, and the instruction-cache misses of its warps, three
// times smaller; one flux at a time, at least 14 blocks of 128 threads per SM
// (32 registers): 165 us at 128^3 (168 us with 10 or 12 blocks; 229 us with the
// products and batched reciprocals of a component's three fluxes and one
// neighbour form).  The FP64 pipe (36 instructions per cell) is 76 % busy, the
// ALU pipe 69 %.
template <int ND, class N>
__device__ __forceinline__ void mom_fluxes_cell(const N& nb, const Grid& G, const double* __restrict__ X,
                                                const double* __restrict__ Fm, double* __restrict__ Psi, const Idx3& P,
                                                long long cc) {
#pragma unroll 1
    for (int c = 0; c < ND; ++c)
#pragma unroll
        for (int d = 0; d < ND; ++d)
            if (!mom_flux<ND>(MomOps(), nb, G, X, Fm, Psi, c, d, cc)) mom_flux_fp64<ND>(G, X, Fm, Psi, c, d, P, cc);
}

template <int ND>
__global__ void __launch_bounds__(128, 14) k_mom_fluxes(Grid G, const double* X,
                                                        const double* Fm, double* Psi) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    if (inner_block<ND>(G)) mom_fluxes_cell<ND>(NbIn(G, P), G, X, Fm, Psi, P, cc);
    else mom_fluxes_cell<ND>(NbGen(G, P), G, X, Fm, Psi, P, cc);
}

// Divergences and sources Rv and conserved variables Uv of one cell.  With
// checked Ops (false, nothing valid, where an operand was out of range) the
// products and twelve differences of fluxes (those of the mass and energy fluxes
// and of the momentum fluxes across) are formed on the integer pipes, which this
// kernel left at 20 %; the FP64 pipe keeps 44 of 56 instructions per cell.  Both
// give the same bits, so the share is a matter of balance alone.  G / float
// product at 128^3, in us: all fifteen flux differences 196 / 222 (ALU pipe 79 %
// busy), without those of the mass fluxes 191 / 219, without the diagonal
// momentum fluxes 186 / 210, without both 197 / 216; none 228 / 246.
template <int ND, class O, class N>
__device__ __forceinline__ bool assemble_terms(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                               const double* __restrict__ p, const double* __restrict__ Fm,
                                               const double* __restrict__ FE, const double* __restrict__ Psi,
                                               long long cc, double (&Uv)[2 + ND], double (&Rv)[2 + ND]) {
    const long long nc = G.ncell;
    constexpr int nd = ND;
    double Rr = 0.0, RE = 0.0, divu = 0.0;
#pragma unroll
    for (int d = 0; d < nd; ++d) {
        const double* fmd = Fm + d * nc + cc;              // pointers at the thread's own cell
        const double* fed = FE + d * nc + cc;
        const double fm0 = *fmd, fm1 = nb.up(fmd, d);
        const double fe0 = *fed, fe1 = nb.up(fed, d);
        Rr = Rr - ops.isub(fm1, fm0) * G.idx[d];
        RE = RE - ops.isub(fe1, fe0) * G.idx[d];
        if (G.energy_form == 0) {
            const double* ud = X + (2 + d) * nc + cc;
            const double u0 = nb.along(ud, d, 0);
            const double u1 = nb.along(ud, d, 1);
            divu = divu + (u1 - u0) * G.idx[d];
        } else if ((G.gmask >> d) & 1) {
            RE = RE + G.hg[d] * (fm0 + fm1);
        }
    }
    const double pc = p[cc];
    if (G.energy_form == 0) RE = RE - pc * divu;

    const double rho = X[cc];
    Uv[0] = rho;            Rv[0] = Rr;
    Uv[1] = ops.mul(rho, X[nc + cc]); Rv[1] = RE;
#pragma unroll
    for (int c = 0; c < nd; ++c) {
        // every thread evaluates (wall slots read mirrored, in-range cells)
        // and wall slots select zero, so no branch splits the warp
        const int om1 = nb.off(c, -1);
        const double pl = p[cc + om1];
        const double rl = X[cc + om1];
        // rs = rl + rho = 2 rho_f: the 1/2 of the face mean is carried by
        // g/2 here and by the halved 1/dt factors of the momentum rows below
        // (exact powers of two: the results are those of rho_f itself)
        const double rs = rl + rho;
        double Rc = ops.mul(pl - pc, G.idx[c]);
        if ((G.gmask >> c) & 1) Rc = fma(rs, G.hg[c], Rc);
#pragma unroll
        for (int d = 0; d < nd; ++d) {
            const double* ps = Psi + (c * nd + d) * nc + cc;
            double a, b;
            if (c == d) {
                b = *ps;
                a = ps[om1];                          // centre i-1 along c
                Rc = Rc - (b - a) * G.hidx[c];                // Psi stored doubled
            } else {
                a = *ps;
                b = nb.up(ps, d);
                Rc = Rc - ops.isub(b, a) * G.hidx[d];
            }
        }
        const bool wall = nb.wall(c);
        Uv[2 + c] = wall ? 0.0 : ops.mul(rs, X[(2 + c) * nc + cc]);        // 2 rho_f u
        Rv[2 + c] = wall ? 0.0 : Rc;
    }
    return ops.valid();
}

template <int ND> struct AsmTerms { double U[2 + ND], R[2 + ND]; };

// the FP64-pipe redo, out of line (see face_flux_dir_fp64); the terms come
// back by value so that the caller's arrays stay in registers
template <int ND>
__device__ __noinline__ AsmTerms<ND> assemble_terms_fp64(const Grid G, const double* __restrict__ X,
                                                         const double* __restrict__ p, const double* __restrict__ Fm,
                                                         const double* __restrict__ FE,
                                                         const double* __restrict__ Psi, const Idx3 P, long long cc) {
    AsmTerms<ND> t;
    assemble_terms<ND>(FpOps(), NbGen(G, P), G, X, p, Fm, FE, Psi, cc, t.U, t.R);
    return t;
}

template <int ND, int MODE, typename TO, class N>
__device__ __forceinline__ void assemble_cell(const N& nb, const Grid& G, const double* __restrict__ X,
                                              const double* __restrict__ p, const double* __restrict__ Fm,
                                              const double* __restrict__ FE, const double* __restrict__ Psi,
                                              const double* __restrict__ bn, const double* __restrict__ G0,
                                              const double* __restrict__ Linv, const double* __restrict__ scal,
                                              double dt_inv, double dt_inv_h, double* __restrict__ outd,
                                              TO* __restrict__ outb, const Idx3& P, long long cc) {
    const long long nc = G.ncell;
    constexpr int nd = ND;
    const double th = G.theta;
    double inv_delta = 0.0;
    if (MODE == kModeJv) inv_delta = scal[kSlotInvDelta];

    double Uv[2 + ND], Rv[2 + ND];
    if (!assemble_terms<ND>(IntOps(), nb, G, X, p, Fm, FE, Psi, cc, Uv, Rv)) {
        const AsmTerms<ND> t = assemble_terms_fp64<ND>(G, X, p, Fm, FE, Psi, P, cc);
#pragma unroll
        for (int k = 0; k < 2 + ND; ++k) {
            Uv[k] = t.U[k];
            Rv[k] = t.R[k];
        }
    }
#pragma unroll
    for (int k = 0; k < 2 + nd; ++k) {
        const long long j = k * nc + cc;
        const bool wall = (k >= 2) && nb.wall(k - 2);
        const double di = k >= 2 ? dt_inv_h : dt_inv;      // momentum rows hold 2 rho_f u
        if (MODE == kModeG) {
            outd[j] = Uv[k] * di - th * Rv[k];
        } else if (MODE == kModeBn) {
            outd[j] = Uv[k] * di + (1.0 - th) * Rv[k];
        } else if (MODE == kModeRes) {
            outd[j] = Uv[k] * di - th * Rv[k] - bn[j];
        } else if (MODE == kModeNewton) {
            double g = Uv[k] * di - th * Rv[k];
            outd[j] = g;
            outb[j] = wall ? (TO)0 : from_f64<TO>(-((g - bn[j]) * Linv[j]));
        } else {
            // kModeJv: L^-1 (G(X+dw) - G(X)) / delta with bn, G0, Linv holding
            // Q = theta L^-1, C = L^-1 G(X) and P = L^-1/dt, halved on the
            // momentum rows (launch_jv_coeffs):
            // (U P - R Q - C) / delta, two FMAs and a product per unknown;
            // kModeJvD leaves out the 1/delta (GMRES applies it to its
            // Hessenberg column): two FMAs per unknown
            const double q = fma(Rv[k], bn[j], G0[j]);
            const double d = fma(Uv[k], Linv[j], -q);
            outb[j] = wall ? (TO)0 : from_f64<TO>(MODE == kModeJv ? d * inv_delta : d);
        }
    }
}

// At least 12 blocks of 128 threads per SM (40 registers).  At 128^3: 186 us (G),
// 210 us (float product); with all differences on the FP64 pipe (84 % busy) 228
// and 246 us, and with 8 blocks 17 us more.
template <int ND, int MODE, typename TO>
__global__ void __launch_bounds__(128, 12) k_assemble(Grid G, const double* X, const double* p,
                           const double* Fm, const double* FE,
                           const double* Psi, const double* bn,
                           const double* G0, const double* Linv,
                           const double* scal, double dt_inv, double dt_inv_h,
                           double* outd, TO* outb) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    if (inner_block<ND>(G))
        assemble_cell<ND, MODE, TO>(NbIn(G, P), G, X, p, Fm, FE, Psi, bn, G0, Linv, scal, dt_inv, dt_inv_h, outd, outb, P, cc);
    else
        assemble_cell<ND, MODE, TO>(NbGen(G, P), G, X, p, Fm, FE, Psi, bn, G0, Linv, scal, dt_inv, dt_inv_h, outd, outb, P, cc);
}

// --------------------------------------------------------------------------
// scaling L, R (Eq. jacobian_system_norm) and ||R^-1 X||^2 partial sums
// --------------------------------------------------------------------------

__device__ __forceinline__ double internal_e(const Grid& G, const double* X, const Idx3& P, int o0, int o1, int o2) {
    const long long nc = G.ncell;
    double E = load_cell(G, X + nc, P, o0, o1, o2);
    if (G.energy_form == 0) return E;
    Idx3 Q;
    Q.i[0] = cell_map(P.i[0] + o0, G.n[0], G.bc[0]);
    Q.i[1] = cell_map(P.i[1] + o1, G.n[1], G.bc[1]);
    Q.i[2] = cell_map(P.i[2] + o2, G.n[2], G.bc[2]);
    double ke = 0.0;
    for (int d = 0; d < G.ndim; ++d) {
        const double* u = X + (2 + d) * nc;
        int o[3] = {0, 0, 0};
        o[d] = 1;
        double ul = load_normal(G, u, d, Q, 0, 0, 0);
        double uu = load_normal(G, u, d, Q, o[0], o[1], o[2]);
        ke = ke + 0.25 * (ul * ul + uu * uu);
    }
    return E - ke;
}

// L, R, their inverses and the squares of x_hat = R^-1 X of one cell.  With
// checked Ops the roots, reciprocals and products are formed on the integer
// pipes (false, nothing written, where one was out of range); the FP64 pipe
// keeps the two sums per face and the squares.  x_hat is one where R is X
// itself (density, energy) and in range; the redo with FpOps forms it, so that
// a NaN, an infinity or a zero there reaches the norm.
template <int ND, class O, class N>
__device__ __forceinline__ bool scaling_cell(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                             double alpha1_h, double alpha2_h, double* __restrict__ L,
                                             double* __restrict__ R, double* __restrict__ Linv,
                                             double* __restrict__ Rinv, const Idx3& P, long long cc, double& acc) {
    const long long nc = G.ncell;
    const double rho = X[cc], E = X[nc + cc];
    double den[2 * (2 + ND)], inv[2 * (2 + ND)];      // L, then R
    den[0] = den[2 + ND] = rho;
    den[1] = ops.mul(rho, E);
    den[3 + ND] = E;
    const double cs0 = ops.root(ops.mul(G.ggm1, G.energy_form == 0 ? E : internal_e(G, X, P, 0, 0, 0)));
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const int o = nb.off(c, -1);
        double el;
        if (G.energy_form == 0) el = X[nc + cc + o];
        else el = internal_e(G, X, P, c == 0 ? -1 : 0, c == 1 ? -1 : 0, c == 2 ? -1 : 0);
        const double rho_f = ops.half(X[cc + o] + rho);
        const double css = ops.root(ops.mul(G.ggm1, el)) + cs0;         // 2 c_s on the face: the alphas are halved
        const double au = fabs(X[(2 + c) * nc + cc]);
        const bool wall = nb.wall(c);
        den[2 + c] = wall ? 1.0 : ops.mul(rho_f, ops.larger(au, ops.mul(alpha1_h, css)));
        den[4 + ND + c] = wall ? 1.0 : ops.larger(au, ops.mul(alpha2_h, css));
    }
    if constexpr (O::checked) {
#pragma unroll
        for (int k = 0; k < 2 * (2 + ND); ++k) inv[k] = k == 2 + ND ? inv[0] : ops.recip(den[k]);
    } else {
        recip_all<2 * (2 + ND)>(den, inv);
    }
    double xh[ND];
#pragma unroll
    for (int c = 0; c < ND; ++c) xh[c] = nb.wall(c) ? 0.0 : ops.mul(X[(2 + c) * nc + cc], inv[4 + ND + c]);
    if (!ops.valid()) return false;
    double a = 2.0;
    if constexpr (!O::checked) {                      // a density or energy without a finite inverse counts as it is
        const double xr = rho * inv[2 + ND], xe = E * inv[3 + ND];
        a = xr * xr + xe * xe;
    }
#pragma unroll
    for (int c = 0; c < ND; ++c) a = fma(xh[c], xh[c], a);
#pragma unroll
    for (int k = 0; k < 2 + ND; ++k) {
        const long long j = k * nc + cc;
        L[j] = den[k];
        R[j] = den[2 + ND + k];
        Linv[j] = inv[k];
        Rinv[j] = inv[2 + ND + k];
    }
    acc = a;
    return true;
}

template <int ND>
__device__ __noinline__ double scaling_cell_fp64(const Grid G, const double* __restrict__ X, double alpha1_h,
                                                 double alpha2_h, double* __restrict__ L, double* __restrict__ R,
                                                 double* __restrict__ Linv, double* __restrict__ Rinv, const Idx3 P,
                                                 long long cc) {
    double acc = 0.0;
    scaling_cell<ND>(FpOps(), NbGen(G, P), G, X, alpha1_h, alpha2_h, L, R, Linv, Rinv, P, cc, acc);
    return acc;
}

// at least 5 blocks of 128 threads per SM (80 registers): 155 us at 128^3, against
// 168 us with 64 registers; with the roots, maxima and most
// products on the FP64 pipe and a batched inversion it took 323 us and 2.54 ms.
// The ALU pipe is 71 % busy.
template <int ND>
__global__ void __launch_bounds__(128, 5) k_scaling(Grid G, const double* X, double alpha1_h,
                          double alpha2_h, double* L, double* R, double* Linv,
                          double* Rinv, double* partials, unsigned* counters) {
    pdl_wait();
    __shared__ double sh[32];
    Idx3 P;
    long long cc;
    double acc = 0.0;
    if (cell_pos(G.n, P, cc)) {
        if (!scaling_cell<ND>(IntOps(), NbGen(G, P), G, X, alpha1_h, alpha2_h, L, R, Linv, Rinv, P, cc,
                              acc))
            acc = scaling_cell_fp64<ND>(G, X, alpha1_h, alpha2_h, L, R, Linv, Rinv, P, cc);
    }
    double s = block_sum<128>(acc, sh);
    if (thread_linear() == 0) partials[block_linear()] = s;
    // last, so that no load waits behind it (159 us with the store first)
    if (block_linear() == 0 && thread_linear() < kNumCounters) counters[thread_linear()] = 0u;
}

// max over cells of |u_cell| + c_s (Sect. 1, CFL_hydro)
template <int ND>
__global__ void k_signal_speed(Grid G, const double* X, double* partials) {
    pdl_wait();
    __shared__ double sh[32];
    Idx3 P;
    long long cc;
    double v = 0.0;
    if (cell_pos(G.n, P, cc)) {
        const long long nc = G.ncell;
        double s = 0.0;
        for (int c = 0; c < ND; ++c) {
            int o[3] = {0, 0, 0};
            o[c] = 1;
            double u0 = load_normal(G, X + (2 + c) * nc, c, P, 0, 0, 0);
            double u1 = load_normal(G, X + (2 + c) * nc, c, P, o[0], o[1], o[2]);
            double ub = 0.5 * (u0 + u1);
            s = s + ub * ub;
        }
        double e = internal_e(G, X, P, 0, 0, 0);
        v = sqrt(s) + sqrt(G.gamma * G.gm1 * e);
        if (!(v == v)) v = __longlong_as_double(0x7ff8000000000000ULL);
    }
    double m = block_max<128>(v, sh);
    if (thread_linear() == 0) partials[block_linear()] = m;
}

// --------------------------------------------------------------------------
// launchers
// --------------------------------------------------------------------------

static inline unsigned nblk(long long n) { return (unsigned)((n + kBlock - 1) / kBlock); }

#define CELL_LAUNCH(KERNEL, ...)                                                          \
    do {                                                                                  \
        CellLaunch cl_ = cell_launch(G.n);                                                \
        ++g_launch_count;                                                                 \
        if (G.ndim == 3) launch_k(KERNEL<3>, cl_.grid, cl_.block, 0, s, __VA_ARGS__);           \
        else launch_k(KERNEL<2>, cl_.grid, cl_.block, 0, s, __VA_ARGS__);                       \
    } while (0)

void launch_eos(const Grid& G, const double* X, double* p, double* T, double* chi, cudaStream_t s) {
    CELL_LAUNCH(k_eos, G, X, p, T, chi);
}

template <typename TZ>
void launch_perturb(const Grid& G, const double* X, const TZ* z, const double* R, const double* scal, int slot,
                    double* Xp, cudaStream_t s) {
    long long nvec = (2 + G.ndim) * G.ncell;
    ++g_launch_count;
    launch_k(k_perturb<TZ>, nblk(nvec), kBlock, 0, s, G, X, z, R, scal, slot, Xp, nvec);
}
template void launch_perturb<double>(const Grid&, const double*, const double*, const double*, const double*, int,
                                     double*, cudaStream_t);
template void launch_perturb<float>(const Grid&, const double*, const float*, const double*, const double*, int,
                                    double*, cudaStream_t);

void launch_face_fluxes(const Grid& G, const double* X, const double* p, const double* T, const double* chi,
                        double* Fm, double* FE, cudaStream_t s) {
    const CellLaunch cl = cell_launch(G.n);
    ++g_launch_count;
    if (G.ndim == 3) {
        if (G.energy_form == 1) launch_k(k_face_fluxes<3, 1>, cl.grid, cl.block, 0, s, G, X, p, T, chi, Fm, FE);
        else launch_k(k_face_fluxes<3, 0>, cl.grid, cl.block, 0, s, G, X, p, T, chi, Fm, FE);
    } else {
        if (G.energy_form == 1) launch_k(k_face_fluxes<2, 1>, cl.grid, cl.block, 0, s, G, X, p, T, chi, Fm, FE);
        else launch_k(k_face_fluxes<2, 0>, cl.grid, cl.block, 0, s, G, X, p, T, chi, Fm, FE);
    }
}

void launch_mom_fluxes(const Grid& G, const double* X, const double* Fm, double* Psi, cudaStream_t s) {
    CELL_LAUNCH(k_mom_fluxes, G, X, Fm, Psi);
}

void launch_fluxes(const Grid& G, const double* X, const double* p, const double* T, const double* chi, double* Fm,
                   double* FE, double* Psi, cudaStream_t s) {
    launch_face_fluxes(G, X, p, T, chi, Fm, FE, s);
    launch_mom_fluxes(G, X, Fm, Psi, s);
}

template <int MODE, typename TO>
void launch_assemble(const Grid& G, const double* X, const double* p, const double* Fm, const double* FE,
                     const double* Psi, const double* bn, const double* G0, const double* Linv, const double* scal,
                     double dt, double* outd, TO* outb, cudaStream_t s) {
    CellLaunch cl = cell_launch(G.n);
    ++g_launch_count;
    if (G.ndim == 3)
        launch_k(k_assemble<3, MODE, TO>, cl.grid, cl.block, 0, s, G, X, p, Fm, FE, Psi, bn, G0, Linv, scal, 1.0 / dt,
                 0.5 / dt, outd, outb);
    else
        launch_k(k_assemble<2, MODE, TO>, cl.grid, cl.block, 0, s, G, X, p, Fm, FE, Psi, bn, G0, Linv, scal, 1.0 / dt,
                 0.5 / dt, outd, outb);
}
#define INST(M, T)                                                                                             \
    template void launch_assemble<M, T>(const Grid&, const double*, const double*, const double*, const double*, \
                                        const double*, const double*, const double*, const double*,           \
                                        const double*, double, double*, T*, cudaStream_t);
INST(kModeG, double)
INST(kModeBn, double)
INST(kModeRes, double)
INST(kModeNewton, double)
INST(kModeNewton, float)
INST(kModeJv, double)
INST(kModeJv, float)
INST(kModeJvD, double)
INST(kModeJvD, float)
#undef INST

void launch_scaling(const Grid& G, const double* X, double a1, double a2, double* L, double* R, double* Linv,
                    double* Rinv, double* partials, unsigned* counters, cudaStream_t s) {
    CELL_LAUNCH(k_scaling, G, X, 0.5 * a1, 0.5 * a2, L, R, Linv, Rinv, partials, counters);
}

void launch_signal_speed(const Grid& G, const double* X, double* partials, cudaStream_t s) {
    CELL_LAUNCH(k_signal_speed, G, X, partials);
}

unsigned cell_blocks(const Grid& G) {
    CellLaunch cl = cell_launch(G.n);
    return cl.grid.x * cl.grid.y * cl.grid.z;
}

}  // namespace jfnk
