// Adjoint kernels: vector-Jacobian products of the residual and the transpose
// of the physics-based preconditioner.
//
// y = (a dU/dX + b dR_U/dX)^T w at a state X, with (a, b) = (1/dt, -theta)
// for G = U/dt - theta R_U and (1/dt, 1 - theta) for b^n.  Each forward
// kernel of residual.cu has a reverse kernel here that recomputes its local
// forward values and scatters the adjoints of its inputs with atomic adds, in
// the reverse order of the forward pass:
//   k_vjp_assemble   adjoints of the half mass fluxes, energy fluxes,
//                    momentum fluxes and p, plus the direct terms (U, gravity,
//                    p div u); gathers and stores, the others scatter
//   k_vjp_mom        momentum fluxes -> velocities and half mass fluxes
//   k_vjp_face       face fluxes -> rho, e or eps_t, velocities, T, chi (and p)
//   k_vjp_eos        p, T, chi -> rho, e (and the kinetic energy for eps_t)
// The derivative of the van Leer face value q_near + ab/(a+b) is
// d/dq_near = 2b/(a+b), d/dq_far = -b^2/(a+b)^2, d/dq_other = a^2/(a+b)^2 where
// ab > 0 (1, 0, 0 otherwise: the derivative of q_near alone); the
// upwind switch contributes nothing (piecewise derivative).  Atomic
// accumulation makes the sums order-dependent at round-off level.
//
// The transposed preconditioner applies the transposes of the pointwise
// transforms and back substitutions exactly, and solves the transposed
// multigrid system with the same V-cycle on the transposed cell matrices.
#include "common.cuh"
#include "kernels.h"

namespace jfnk {


// storage slot and sign of the velocity normal to direction c at position
// (pos + off); false for a wall face (a constant zero, no adjoint).
__device__ __forceinline__ bool normal_slot(const Grid& G, int c, const Idx3& P, int o0, int o1, int o2,
                                            long long& j, double& sgn) {
    int k[3] = {P.i[0] + o0, P.i[1] + o1, P.i[2] + o2};
    sgn = 1.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (d == c && G.bc[d] == 1) {
            int n = G.n[d];
            int kk = k[d];
            if (kk == 0 || kk == n) return false;
            if (kk < 0) { kk = -kk; sgn = -sgn; }
            else if (kk > n) { kk = 2 * n - kk; sgn = -sgn; }
            k[d] = kk;
        } else {
            k[d] = cell_map(k[d], G.n[d], G.bc[d]);
        }
    }
    j = flat(G, k[0], k[1], k[2]);
    return true;
}

__device__ __forceinline__ long long cell_slot(const Grid& G, const Idx3& P, int o0, int o1, int o2) {
    return flat(G, cell_map(P.i[0] + o0, G.n[0], G.bc[0]), cell_map(P.i[1] + o1, G.n[1], G.bc[1]),
                cell_map(P.i[2] + o2, G.n[2], G.bc[2]));
}

// slot of the face above cell P along d (false at an upper wall)
__device__ __forceinline__ bool up_slot(const Grid& G, int d, const Idx3& P, long long& j) {
    if (G.bc[d] == 1 && P.i[d] + 1 == G.n[d]) return false;
    int o[3] = {0, 0, 0};
    o[d] = 1;
    j = cell_slot(G, P, o[0], o[1], o[2]);
    return true;
}

// van Leer face value and its partial derivatives.  With ai = a/(a+b), bi =
// b/(a+b) (they add to one): v = near + a bi, dv/dnear = 1 + bi^2 - ai^2 = 2 bi,
// dv/dfar = -bi^2, dv/dother = ai^2 where the limiter is on; v = near, 1, 0, 0
// where it is off.
struct UpwindD {
    double v, ai, bi;
    bool on;
};

// The adjoint kernels were bound by the FP64 pipe (about 30 instructions per
// face value, ten of them a division): their products and reciprocals run on
// the integer pipes like those of the forward kernels, and the FP64 pipe keeps
// the differences and sums.  Values are formed first and scattered after the
// range check; where it fails the thread redoes the face with FpOps.
template <class O>
__device__ __forceinline__ UpwindD upwind_d(O& ops, double q_near, double q_far, double q_other) {
    const double a = q_near - q_far, b = q_other - q_near;
    UpwindD r;
    if constexpr (O::checked) {
        const uint32_t ah = emu::hi_word(a), bh = emu::hi_word(b);
        r.on = ((ah ^ bh) >> 31) == 0u && ((ah & 0x7fffffffu) | emu::lo_word(a)) != 0u &&
               ((bh & 0x7fffffffu) | emu::lo_word(b)) != 0u;
    } else {
        r.on = positive(a * b);
    }
    const double inv = ops.recip(r.on ? a + b : 1.0);
    r.ai = ops.mul(a, inv);
    r.bi = ops.mul(b, inv);
    const double h = ops.mul(a, r.bi);
    r.v = q_near + (r.on ? h : 0.0);
    return r;
}

// adjoints of the three values of a face whose value's adjoint is vb
struct FaceAdj {
    double near, far, other;
};
template <class O>
__device__ __forceinline__ FaceAdj face_adjoint(O& ops, const UpwindD& u, double vb) {
    const double t = ops.mul(vb, u.bi), r = ops.mul(vb, u.ai);
    FaceAdj f;
    f.near = u.on ? t + t : vb;
    f.far = u.on ? emu::neg(ops.mul(t, u.bi)) : 0.0;
    f.other = u.on ? ops.mul(r, u.ai) : 0.0;
    return f;
}

__device__ __forceinline__ double cond_dchi(const Grid& G, double T) {
    return G.chi3 ? 3.0 * G.K0 * (T * T) : G.K0 * G.chi_exp * pow(T, G.chi_exp - 1.0);
}

struct AdjBufs {
    double* Fmhb;   // nd fields
    double* FEb;    // nd fields
    double* Psib;   // nd*nd fields
    double* pb;
    double* Tb;
    double* chib;
    double* Xb;     // packed
};

// --------------------------------------------------------------------------
// reverse of k_assemble
// --------------------------------------------------------------------------
// Every adjoint here is the sum of what the cell itself and one neighbour
// contribute, so each thread gathers both and stores the values of its own
// slots: no atomic adds, no zeroing of the 24 fields before, and the rest of
// the reverse pass adds to what is stored here.  Products with checked Ops on
// the integer pipes; a thread for which one was out of range stores again.
template <int ND, class O, class N>
__device__ __forceinline__ bool vjp_assemble_cell(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                                  const double* __restrict__ p, const double* __restrict__ w,
                                                  double a_u, double b_r, const AdjBufs& A, long long cc) {
    const long long nc = G.ncell;
    const double w0 = w[cc], wE = w[nc + cc], rho = X[cc], E = X[nc + cc];
    double divu = 0.0, ub[ND];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const bool low = nb.has_low(d);
        const int o = low ? nb.off(d, -1) : 0;
        const double w0l = low ? w[cc + o] : 0.0, wEl = low ? w[nc + cc + o] : 0.0;
        double fm = ops.mul(w0 - w0l, b_r * G.tidx[d]);
        if (G.energy_form == 1 && ((G.gmask >> d) & 1)) fm = fm + ops.mul(wE + wEl, b_r * G.g[d]);
        A.Fmhb[d * nc + cc] = fm;
        A.FEb[d * nc + cc] = ops.mul(wE - wEl, b_r * G.idx[d]);
        ub[d] = 0.0;
        if (G.energy_form == 0) {
            const double* ud = X + (2 + d) * nc + cc;
            divu = fma(nb.along(ud, d, 1) - nb.along(ud, d, 0), G.idx[d], divu);
            if (low) ub[d] = ops.mul(ops.mul(wE, p[cc]) - ops.mul(wEl, p[cc + o]), b_r * G.idx[d]);
        }
    }
    double pb = G.energy_form == 0 ? -(ops.mul(b_r, wE) * divu) : 0.0;
    double rfs = 0.0;                                    // adjoints of rho_f on the faces below and above
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const double* wc = w + (2 + c) * nc + cc;
        const double* uc = X + (2 + c) * nc + cc;
        const bool wall = nb.wall(c), up = nb.has_up(c);
        const int ou = up ? nb.off(c, 1) : 0;
        const double v = wall ? 0.0 : wc[0], vu = up ? wc[ou] : 0.0;
        const double t = ops.mul(vu - v, b_r * G.idx[c]);
        pb = pb + t;
        const double bg = b_r * G.g[c];
        rfs = rfs + (ops.mul(v, fma(a_u, wall ? 0.0 : uc[0], bg)) + ops.mul(vu, fma(a_u, uc[ou], bg)));
        const double rho2 = X[cc + nb.off(c, -1)] + rho;
        A.Xb[(2 + c) * nc + cc] = wall ? 0.0 : fma(ops.mul(v, 0.5 * a_u), rho2, ub[c]);
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            double psi = t;                              // c == d: the flux at the cell centre
            if (c != d) {
                const bool low = nb.has_low(d);
                const double vl = low && !wall ? wc[low ? nb.off(d, -1) : 0] : 0.0;
                psi = ops.mul(v - vl, b_r * G.idx[d]);
            }
            A.Psib[(c * ND + d) * nc + cc] = psi;
        }
    }
    A.pb[cc] = pb;
    A.Tb[cc] = 0.0;
    A.chib[cc] = 0.0;
    A.Xb[cc] = fma(0.5, rfs, ops.mul(a_u, fma(wE, E, w0)));
    A.Xb[nc + cc] = ops.mul(ops.mul(a_u, wE), rho);
    return ops.valid();
}

template <int ND>
__device__ __noinline__ void vjp_assemble_cell_fp64(const Grid G, const double* __restrict__ X,
                                                    const double* __restrict__ p, const double* __restrict__ w,
                                                    double a_u, double b_r, const AdjBufs A, const Idx3 P,
                                                    long long cc) {
    vjp_assemble_cell<ND>(FpOps(), NbGen(G, P), G, X, p, w, a_u, b_r, A, cc);
}

// 259 us at 128^3; as a scatter 363 us, after 60 us to zero the fields
template <int ND>
__global__ void __launch_bounds__(128, 8) k_vjp_assemble(Grid G, const double* X,
                                                         const double* p, const double* w,
                                                         double a_u, double b_r, AdjBufs A) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const bool ok = inner_block<ND>(G)
                        ? vjp_assemble_cell<ND>(IntOps(), NbIn(G, P), G, X, p, w, a_u, b_r, A, cc)
                        : vjp_assemble_cell<ND>(IntOps(), NbGen(G, P), G, X, p, w, a_u, b_r, A, cc);
    if (!ok) vjp_assemble_cell_fp64<ND>(G, X, p, w, a_u, b_r, A, P, cc);
}

// --------------------------------------------------------------------------
// reverse of k_mom_fluxes (Fm: the forward mass fluxes; m is the carrying
// mean of two of them, which the adjoint buffers below differentiate as the
// sum of two half fluxes)
// --------------------------------------------------------------------------
template <int ND, class O, class N>
__device__ __forceinline__ bool vjp_mom_face(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                             const double* __restrict__ Fm, const AdjBufs& A, int c, int d,
                                             long long cc, double psib) {
    const long long nc = G.ncell;
    const double* uc = X + (2 + c) * nc + cc;           // pointers at the thread's own slot
    const double* fmd = Fm + d * nc + cc;
    double* ub = A.Xb + (2 + c) * nc + cc;
    double* fb = A.Fmhb + d * nc + cc;
    // the four velocities along d as in mom_flux, the flux between 1 and 2
    int o[4], om;
    bool flip[4], ok[4], hasm;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        ok[k] = c == d ? nb.slot_along(c, k - 1, o[k], flip[k]) : nb.slot_across(c, d, k - 2, o[k], flip[k]);
    // the second of the two mass fluxes that carry it
    if (c == d) {
        hasm = nb.has_up(c);
        om = hasm ? nb.off(c, 1) : 0;
    } else {
        hasm = true;
        om = nb.off(c, -1);
    }
    const double m2 = fmd[0] + (hasm ? fmd[om] : 0.0);  // twice the carrying mean
    const bool left = nonneg(m2);
    double q[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const double v = uc[o[k]];
        q[k] = ok[k] ? (flip[k] ? emu::neg(v) : v) : 0.0;
    }
    const UpwindD U = upwind_d(ops, left ? q[1] : q[2], left ? q[0] : q[3], left ? q[2] : q[1]);
    const double mb = ops.mul(psib, U.v);
    const FaceAdj f = face_adjoint(ops, U, ops.mul(0.5 * psib, m2));
    if (!ops.valid()) return false;
    atomicAdd(fb, mb);
    if (hasm) atomicAdd(fb + om, mb);
    // (a wall face reads zero and has no adjoint; signs flip on the integer pipe)
    auto put = [&](int k, double v) {
        if (ok[k]) atomicAdd(ub + o[k], flip[k] ? emu::neg(v) : v);
    };
    put(1, left ? f.near : f.other);
    put(2, left ? f.other : f.near);
    if (U.on) {
        if (left) put(0, f.far);
        else put(3, f.far);
    }
    return true;
}

// plain operators with a division, for the redo
struct AdjFp : FpOps {
    __device__ __forceinline__ double recip(double d) { return 1.0 / d; }
};

template <int ND>
__device__ __noinline__ void vjp_mom_face_fp64(const Grid G, const double* __restrict__ X,
                                               const double* __restrict__ Fm, const AdjBufs A, int c, int d,
                                               const Idx3 P, long long cc, double psib) {
    vjp_mom_face<ND>(AdjFp(), NbGen(G, P), G, X, Fm, A, c, d, cc, psib);
}

template <int ND, class N>
__device__ __forceinline__ void vjp_mom_cell(const N& nb, const Grid& G, const double* __restrict__ X,
                                             const double* __restrict__ Fm, const AdjBufs& A, const Idx3& P,
                                             long long cc) {
#pragma unroll 1
    for (int c = 0; c < ND; ++c)
#pragma unroll 1
        for (int d = 0; d < ND; ++d) {
            const double psib = A.Psib[(c * ND + d) * G.ncell + cc];
            if (is_zero(psib)) continue;
            if (!vjp_mom_face<ND>(IntOps(), nb, G, X, Fm, A, c, d, cc, psib))
                vjp_mom_face_fp64<ND>(G, X, Fm, A, c, d, P, cc, psib);
        }
}

// Bound by the ALU pipe (77 % busy): 467 us at 128^3 with at least 8 blocks of 128
// threads per SM; with divisions and products on the FP64 pipe 1,139 us, with them
// on the integer pipes but slots recomputed by the general mapping 668 us.
template <int ND>
__global__ void __launch_bounds__(128, 8) k_vjp_mom(Grid G, const double* X,
                                                    const double* Fm, AdjBufs A) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    if (inner_block<ND>(G)) vjp_mom_cell<ND>(NbIn(G, P), G, X, Fm, A, P, cc);
    else vjp_mom_cell<ND>(NbGen(G, P), G, X, Fm, A, P, cc);
}

// --------------------------------------------------------------------------
// reverse of k_face_fluxes
// --------------------------------------------------------------------------
template <int ND, class O, class N>
__device__ __forceinline__ bool vjp_face_dir(O ops, const N& nb, const Grid& G, const double* __restrict__ X,
                                             const double* __restrict__ p, const double* __restrict__ T,
                                             const double* __restrict__ chi, const AdjBufs& A, int d, long long c,
                                             double fmhb, double feb) {
    const long long nc = G.ncell;
    const double* rho = X;
    const double* E = X + nc;
    const bool wall = nb.wall(d);
    const double u = wall ? 0.0 : X[(2 + d) * nc + c];
    const bool left = nonneg(u);
    const long long jl = c + nb.off(d, -1), jn = left ? jl : c, jo = left ? c : jl;
    const long long jf = c + (left ? nb.off(d, -2) : nb.off(d, 1));
    const UpwindD Ur = upwind_d(ops, rho[jn], rho[jf], rho[jo]);
    const UpwindD Ue = upwind_d(ops, E[jn], E[jf], E[jo]);
    const double fm = ops.mul(u, Ur.v);
    const double fmb = 0.5 * fmhb + ops.mul(feb, Ue.v);
    double ubar = ops.mul(fmb, Ur.v);
    const FaceAdj fr = face_adjoint(ops, Ur, ops.mul(fmb, u));
    const FaceAdj fe = face_adjoint(ops, Ue, ops.mul(feb, fm));
    double pq = 0.0, qa = 0.0, qb = 0.0;
    if (G.energy_form == 1) {
        ubar += 0.5 * ops.mul(feb, p[jl] + p[c]);
        pq = 0.5 * ops.mul(feb, u);
    }
    if (G.has_cond) {
        // FE contains -q, q = (chi_L + chi_R)/2 (T_R - T_L) / dx
        const double qh = ops.mul(feb, -G.hidx[d]);
        qa = ops.mul(qh, T[c] - T[jl]);
        qb = ops.mul(qh, chi[jl] + chi[c]);             // chi of the forward k_eos
    }
    if (!ops.valid()) return false;
    if (!wall) {
        atomicAdd(A.Xb + (2 + d) * nc + c, ubar);
        atomicAdd(A.Xb + jn, fr.near);
        if (Ur.on) {
            atomicAdd(A.Xb + jf, fr.far);
            atomicAdd(A.Xb + jo, fr.other);
        }
        atomicAdd(A.Xb + nc + jn, fe.near);
        if (Ue.on) {
            atomicAdd(A.Xb + nc + jf, fe.far);
            atomicAdd(A.Xb + nc + jo, fe.other);
        }
        if (G.energy_form == 1) {
            atomicAdd(A.pb + jl, pq);
            atomicAdd(A.pb + c, pq);
        }
    }
    if (G.has_cond) {
        atomicAdd(A.chib + jl, qa);
        atomicAdd(A.chib + c, qa);
        atomicAdd(A.Tb + c, qb);
        atomicAdd(A.Tb + jl, -qb);
    }
    return true;
}

template <int ND>
__device__ __noinline__ void vjp_face_dir_fp64(const Grid G, const double* __restrict__ X,
                                               const double* __restrict__ p, const double* __restrict__ T,
                                               const double* __restrict__ chi, const AdjBufs A, int d, const Idx3 P,
                                               long long c, double fmhb, double feb) {
    vjp_face_dir<ND>(AdjFp(), NbGen(G, P), G, X, p, T, chi, A, d, c, fmhb, feb);
}

template <int ND, class N>
__device__ __forceinline__ void vjp_face_cell(const N& nb, const Grid& G, const double* __restrict__ X,
                                              const double* __restrict__ p, const double* __restrict__ T,
                                              const double* __restrict__ chi, const AdjBufs& A, const Idx3& P,
                                              long long c) {
#pragma unroll 1
    for (int d = 0; d < ND; ++d) {
        const double fmhb = A.Fmhb[d * G.ncell + c], feb = A.FEb[d * G.ncell + c];
        if (is_zero(fmhb) && is_zero(feb)) continue;
        if (!vjp_face_dir<ND>(IntOps(), nb, G, X, p, T, chi, A, d, c, fmhb, feb))
            vjp_face_dir_fp64<ND>(G, X, p, T, chi, A, d, P, c, fmhb, feb);
    }
}

// 330 us at 128^3, 716 us with divisions and products on the FP64 pipe
template <int ND>
__global__ void __launch_bounds__(128, 8) k_vjp_face(Grid G, const double* X,
                                                     const double* p, const double* T,
                                                     const double* chi, AdjBufs A) {
    pdl_wait();
    Idx3 P;
    long long c;
    if (!cell_pos(G.n, P, c)) return;
    if (inner_block<ND>(G)) vjp_face_cell<ND>(NbIn(G, P), G, X, p, T, chi, A, P, c);
    else vjp_face_cell<ND>(NbGen(G, P), G, X, p, T, chi, A, P, c);
}

// --------------------------------------------------------------------------
// reverse of k_eos; finishes Xb (wall slots cleared)
// --------------------------------------------------------------------------
template <int ND>
__global__ void k_vjp_eos(Grid G, const double* X, const double* T, AdjBufs A) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const long long nc = G.ncell;
    const double rho = X[cc];
    const double Tc = T[cc];
    const double e = Tc / G.gm1;
    double Tbt = A.Tb[cc];
    if (G.has_cond) Tbt += A.chib[cc] * cond_dchi(G, Tc);
    const double pbv = A.pb[cc];
    const double eb = pbv * G.gm1 * rho + Tbt * G.gm1;
    atomicAdd(A.Xb + cc, pbv * G.gm1 * e);
    atomicAdd(A.Xb + nc + cc, eb);
    if (G.energy_form == 1) {
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const double* ud = X + (2 + d) * nc;
            long long j;
            double sg;
            if (!is_wall_slot(G, d, P)) atomicAdd(A.Xb + (2 + d) * nc + cc, -eb * 0.5 * ud[cc]);
            int o[3] = {0, 0, 0};
            o[d] = 1;
            if (normal_slot(G, d, P, o[0], o[1], o[2], j, sg))
                atomicAdd(A.Xb + (2 + d) * nc + j, -eb * 0.5 * ud[j]);
        }
    }
}

// w . dR_U/dK0: the conduction divergence without K0, dotted with w_E
template <int ND>
__global__ void k_dRdK0_dot(Grid G, const double* T, const double* w,
                            double* partials) {
    pdl_wait();
    __shared__ double sh[32];
    Idx3 P;
    long long cc;
    double acc = 0.0;
    if (cell_pos(G.n, P, cc)) {
        const long long nc = G.ncell;
        double div = 0.0;
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            int o[3] = {0, 0, 0};
            o[d] = -1;
            const long long jl = cell_slot(G, P, o[0], o[1], o[2]);
            const double Tl = T[jl], Tc = T[cc];
            const double kl = G.chi3 ? Tl * Tl * Tl : pow(Tl, G.chi_exp);
            const double kc = G.chi3 ? Tc * Tc * Tc : pow(Tc, G.chi_exp);
            const double q0 = 0.5 * (kl + kc) * (Tc - Tl) * G.idx[d];
            double q1 = 0.0;
            long long ju;
            if (up_slot(G, d, P, ju)) {
                const double Tu = T[ju];
                const double ku = G.chi3 ? Tu * Tu * Tu : pow(Tu, G.chi_exp);
                q1 = 0.5 * (kc + ku) * (Tu - Tc) * G.idx[d];
            }
            div = div + (q1 - q0) * G.idx[d];
        }
        acc = w[nc + cc] * div;
    }
    double s = block_sum<128>(acc, sh);
    if (thread_linear() == 0) partials[block_linear()] = s;
}

#define CELL_LAUNCH_A(KERNEL, ...)                                                        \
    do {                                                                                  \
        CellLaunch cl_ = cell_launch(G.n);                                                \
        ++g_launch_count;                                                                 \
        if (G.ndim == 3) launch_k(KERNEL<3>, cl_.grid, cl_.block, 0, s, __VA_ARGS__);           \
        else launch_k(KERNEL<2>, cl_.grid, cl_.block, 0, s, __VA_ARGS__);                       \
    } while (0)

void launch_vjp(const Grid& G, const double* X, const double* p, const double* T, const double* chi, const double* Fm,
                const double* w, double a_u, double b_r, double* adj, double* Xb, cudaStream_t s) {
    const long long nc = G.ncell, nd = G.ndim;
    AdjBufs A;
    A.Fmhb = adj;
    A.FEb = A.Fmhb + nd * nc;
    A.Psib = A.FEb + nd * nc;
    A.pb = A.Psib + nd * nd * nc;
    A.Tb = A.pb + nc;
    A.chib = A.Tb + nc;
    A.Xb = Xb;
    CELL_LAUNCH_A(k_vjp_assemble, G, X, p, w, a_u, b_r, A);
    CELL_LAUNCH_A(k_vjp_mom, G, X, Fm, A);
    CELL_LAUNCH_A(k_vjp_face, G, X, p, T, chi, A);
    CELL_LAUNCH_A(k_vjp_eos, G, X, T, A);
}

long long vjp_scratch_doubles(const Grid& G) {
    const long long nc = G.ncell, nd = G.ndim;
    return (2 * nd + nd * nd + 3) * nc;
}

void launch_dRdK0_dot(const Grid& G, const double* T, const double* w, double* partials, cudaStream_t s) {
    CELL_LAUNCH_A(k_dRdK0_dot, G, T, w, partials);
}

// --------------------------------------------------------------------------
// transposed preconditioner (FP64)
// --------------------------------------------------------------------------

__device__ __forceinline__ long long mg0_index(const Grid& G, const Idx3& P) {
    return rb_index(G.n[0], G.n[1], G.ncell, P.i[0], P.i[1], P.i[2]);
}

// Stage 1: y -> adjoints of (dp, de, du) through R^-1, dX/dV and the back
// substitution; writes the multigrid right-hand side (transposed system),
// the adjoints of r_u and r_e, and the direct part of the adjoint of r_p.
template <int ND>
__global__ void k_precondT_out(Grid G, const double* C, double dt, int nf, const double* y,
                               double* rub, double* reb, double* rpb,
                               double* rhs, double* x0, const double* D,
                               int nu1) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const long long nc = G.ncell;
    // adjoint of dX = R^-1 y (diagonal), then of dX/dV
    const double drhob = y[cc] * C[PcRinvR * nc + cc];
    const double dEb = y[nc + cc] * C[PcRinvE * nc + cc];
    double dpb = drhob * C[PcInvDpdrho * nc + cc];
    double deb = dEb - C[PcDpde * nc + cc] * C[PcInvDpdrho * nc + cc] * drhob;
    // du adjoint at the faces of this cell (own slot), including the
    // eps_t = e + <u.du> term for the total energy form
    double dub[ND];
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        dub[c] = y[(2 + c) * nc + cc] * C[(PcRinvU + c) * nc + cc];
        if (G.energy_form == 1 && !is_wall_slot(G, c, P)) {
            int o[3] = {0, 0, 0};
            o[c] = -1;
            const long long jl = cell_slot(G, P, o[0], o[1], o[2]);
            const double dEbl = y[nc + jl] * C[PcRinvE * nc + jl];
            dub[c] += 0.5 * C[(PcU + c) * nc + cc] * (dEb + dEbl);
        }
    }
    // back substitution: du_c(k) = dt (r_u - thf (dp(k) - dp(k-1)))
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        rub[c * nc + cc] = dt * dub[c];
        dpb -= dt * C[(PcThf + c) * nc + cc] * dub[c];
        long long ju;
        if (up_slot(G, c, P, ju)) {
            double yu = y[(2 + c) * nc + ju] * C[(PcRinvU + c) * nc + ju];
            if (G.energy_form == 1) {
                const double dEbu = y[nc + ju] * C[PcRinvE * nc + ju];
                yu += 0.5 * C[(PcU + c) * nc + ju] * (dEbu + dEb);
            }
            dpb += dt * C[(PcThf + c) * nc + ju] * yu;
        }
    }
    const long long mi = mg0_index(G, P);
    // multigrid start as in k_precond_in, with the transposed diagonal block
    const bool red = nu1 > 0 && ((P.i[0] + P.i[1] + P.i[2]) & 1) == 0;
    if (nf == 1) {
        // de = dt (r_e + (dp/dt - r_p) cde)
        reb[cc] = dt * deb;
        rpb[cc] = -dt * C[PcCde * nc + cc] * deb;
        const double b0 = dpb + deb * C[PcCde * nc + cc];
        rhs[mi] = b0;
        x0[mi] = red ? D[mi] * b0 : 0.0;
    } else {
        reb[cc] = 0.0;
        rpb[cc] = 0.0;
        rhs[mi] = dpb;
        rhs[nc + mi] = deb;
        x0[mi] = red ? D[mi] * dpb + D[2 * nc + mi] * deb : 0.0;
        x0[nc + mi] = red ? D[nc + mi] * dpb + D[3 * nc + mi] * deb : 0.0;
    }
}

// Adjoints of r_p and r_e at a cell (slot j, multigrid index mi): the direct
// parts from stage 1 plus B^-T applied to the transposed multigrid solution.
struct RpRe {
    double rp, re;
};

__device__ __forceinline__ RpRe rp_re_bar(const double* C, long long nc, int nf, const double* xmg,
                                          const double* reb, const double* rpb, long long j, long long mi) {
    RpRe r;
    r.rp = rpb[j];
    r.re = reb[j];
    if (nf == 1) {
        r.rp += C[PcQ0 * nc + j] * xmg[mi];
    } else {
        const double y0 = xmg[mi], y1 = xmg[nc + mi];
        r.rp += C[PcQ0 * nc + j] * y0 + C[PcQ2 * nc + j] * y1;
        r.re += C[PcQ1 * nc + j] * y0 + C[PcQ3 * nc + j] * y1;
    }
    return r;
}

// total adjoint of r_e at cell Q (r_p = dpdrho r_rho + dpde r_e also uses r_e)
__device__ __forceinline__ double reb_total(const Grid& G, const double* C, int nf, const double* xmg,
                                            const double* reb, const double* rpb, const Idx3& Q) {
    const long long nc = G.ncell;
    const long long j = flat(G, Q.i[0], Q.i[1], Q.i[2]);
    RpRe r = rp_re_bar(C, nc, nf, xmg, reb, rpb, j, mg0_index(G, Q));
    return r.re + C[PcDpde * nc + j] * r.rp;
}

// total adjoint of r_u_c on the lower face of cell Q (adds, for the total
// energy form, the -<u.r_u> term of r_e of the two cells beside the face)
__device__ __forceinline__ double rub_total(const Grid& G, const double* C, int nf, const double* xmg,
                                            const double* reb, const double* rpb, const double* rub, int c,
                                            const Idx3& Q) {
    const long long nc = G.ncell;
    const long long j = flat(G, Q.i[0], Q.i[1], Q.i[2]);
    double v = rub[c * nc + j];
    if (G.energy_form == 1 && !is_wall_slot(G, c, Q)) {
        Idx3 L = Q;
        L.i[c] = cell_map(Q.i[c] - 1, G.n[c], G.bc[c]);
        v -= 0.5 * C[(PcU + c) * nc + j] *
             (reb_total(G, C, nf, xmg, reb, rpb, Q) + reb_total(G, C, nf, xmg, reb, rpb, L));
    }
    return v;
}

// Stage 2: adjoints of (r_p, r_e, r_u) -> z = L (dV/dU)^T (...), through B^-T.
template <int ND>
__global__ void k_precondT_in(Grid G, const double* C, int nf, const double* xmg,
                              const double* rub, const double* reb,
                              const double* rpb, double* z) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const long long nc = G.ncell;
    const RpRe r = rp_re_bar(C, nc, nf, xmg, reb, rpb, cc, mg0_index(G, P));
    // r_p = dpdrho r_rho + dpde r_e ; r_e = (r_E - E r_rho) invrho [- <u.r_u>]
    const double reb_t = r.re + C[PcDpde * nc + cc] * r.rp;
    double rrho_b = C[PcDpdrho * nc + cc] * r.rp - C[PcE * nc + cc] * C[PcInvRho * nc + cc] * reb_t;
    const double rE_b = C[PcInvRho * nc + cc] * reb_t;
    // r_u_c(k) = (L_u v_u - u_c rbar_rho) invrhof, rbar_rho the face mean of r_rho
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const double own = rub_total(G, C, nf, xmg, reb, rpb, rub, c, P);
        rrho_b -= 0.5 * C[(PcU + c) * nc + cc] * C[(PcInvRhof + c) * nc + cc] * own;
        long long ju;
        if (up_slot(G, c, P, ju)) {
            Idx3 U = P;
            U.i[c] = (P.i[c] + 1 == G.n[c]) ? 0 : P.i[c] + 1;
            const double up = rub_total(G, C, nf, xmg, reb, rpb, rub, c, U);
            rrho_b -= 0.5 * C[(PcU + c) * nc + ju] * C[(PcInvRhof + c) * nc + ju] * up;
        }
        z[(2 + c) * nc + cc] = C[(PcLu + c) * nc + cc] * C[(PcInvRhof + c) * nc + cc] * own;
    }
    z[cc] = C[PcLr * nc + cc] * rrho_b;
    z[nc + cc] = C[PcLE * nc + cc] * rE_b;
}

void launch_precondT_out(const Grid& G, const double* C, double dt, int nf, const double* y, double* rub, double* reb,
                         double* rpb, MGLevel& L0, cudaStream_t s, int nu1) {
    CELL_LAUNCH_A(k_precondT_out, G, C, dt, nf, y, rub, reb, rpb, (double*)L0.rhs, (double*)L0.x, (const double*)L0.D,
                  nu1);
}

void launch_precondT_in(const Grid& G, const double* C, int nf, const MGLevel& L0, const double* rub,
                        const double* reb, const double* rpb, double* z, cudaStream_t s) {
    CELL_LAUNCH_A(k_precondT_in, G, C, nf, (const double*)L0.x, rub, reb, rpb, z);
}

// out = x * y elementwise
__global__ void k_mul(const double* x, const double* y, double* out,
                      long long n) {
    pdl_wait();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        out[e] = x[e] * y[e];
}

void launch_mul(const double* x, const double* y, double* out, long long n, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_mul, kRedBlocks, kBlock, 0, s, x, y, out, n);
}

// out = a - b elementwise
__global__ void k_sub(const double* a, const double* b, double* out,
                      long long n) {
    pdl_wait();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        out[e] = a[e] - b[e];
}

void launch_sub(const double* a, const double* b, double* out, long long n, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_sub, kRedBlocks, kBlock, 0, s, a, b, out, n);
}

// zero the wall-face slots of a packed vector
template <int ND>
__global__ void k_mask_walls(Grid G, double* v) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
#pragma unroll
    for (int c = 0; c < ND; ++c)
        if (is_wall_slot(G, c, P)) v[(2 + c) * G.ncell + cc] = 0.0;
}

void launch_mask_walls(const Grid& G, double* v, cudaStream_t s) { CELL_LAUNCH_A(k_mask_walls, G, v); }

}  // namespace jfnk
