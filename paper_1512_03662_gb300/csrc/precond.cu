// Physics-based preconditioner (paper Sects. 3.2-3.4 and 4.3).
//
//   w = R^-1 dX/dV J~_V^-1 dV/dU L v
//
// k_precond_in   v -> r_V = dV/dU L v, factored as dV/dX dX/dU (App. B); the
//                velocity rows act face by face, r_u = (r_rhou - u rbar_rho)/rho_f;
//                the multigrid right-hand side is B^-1 (r_p, r_e), B the 2x2
//                matrix of the Laplacian coefficients of the p and e rows
//                (1x1, B = theta^2 dt Gamma1 p, for the sound-only scheme).
// k_pc_setup     cell matrix M = B^-1/dt and face coefficients K_p = 1/rho_f,
//                K_e = chi_f/c_v of the equivalent system
//                    M x - [div(K_p grad dp); div(K_e grad de)] = B^-1 r,
//                from the current Newton iterate (the multigrid of
//                multigrid.cu solves it; K is stored over dx^2).
// k_precond_out  de from the identity of Sect. 3.3.4 (sound scheme) or from
//                the coupled solve; du_f = dt (r_u - theta rho_f^-1 grad dp);
//                dX = dX/dV dV; z = R^-1 dX and partial sums of |z|^2.
// The multigrid and the pointwise transforms run in the basis precision T (float
// in mixed mode), on coefficients that are formed in double and rounded once.
#include "common.cuh"
#include "kernels.h"

namespace jfnk {

// index of fine-level cell P in the level-0 multigrid arrays
__device__ __forceinline__ long long mg0(const Grid& G, const Idx3& P) {
    return rb_index(G.n[0], G.n[1], G.ncell, P.i[0], P.i[1], P.i[2]);
}

// ---------------------------------------------------------------------------
// coefficients at the current iterate (once per Newton iteration)
// ---------------------------------------------------------------------------

// Per-cell coefficient fields of the transforms, in the basis precision T.
// Field order (index * ncell): see PcField.  All divisions of the
// preconditioner happen here, once per Newton iteration, and they reduce to
// reciprocals of rho, T and the face densities (one batched inversion); T and
// chi come from k_eos.  B is the 2x2 matrix of Laplacian coefficients of the
// p and e rows (sound scheme: its first entry alone).  For the ideal gas its
// determinant is theta c1 T (c1 = theta^2 dt, gamma - (gamma-1) = 1), so the
// inverse has the closed form
//     [ 1/(c1 rho T)   -(gamma-1)/(c1 T) ]
//     [ -1/theta        gamma rho/theta  ]
// and the map of the residuals to the right-hand side loses the terms that
// cancel (the factors of r_E and of the kinetic term in the p row are zero).
template <int ND, typename T>
__global__ void k_pc_setup(Grid G, const double* X, const double* Tg,
                           const double* chi, const double* L,
                           const double* Rinv, double ic1, double ith, double idt, int nf,
                           T* C, T* M, T* K) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const long long nc = G.ncell;
    const double rho = X[cc], E = X[nc + cc], Tc = Tg[cc];
    double den[2 + ND], inv[2 + ND];
    int om1[ND];
    den[0] = rho;
    den[1] = Tc;
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        om1[c] = cell_off(G, P, c, -1);
        den[2 + c] = 0.5 * (X[cc + om1[c]] + rho);           // rho_f on the lower face
    }
    recip_all<2 + ND>(den, inv);
    const double irho = inv[0], iT = inv[1], dpde = G.gm1 * rho;
    const double b00 = (nf == 2 ? ic1 : ic1 * G.igamma) * (irho * iT);
    const double b01 = -(G.gm1 * ic1) * iT, b10 = -ith, b11 = (G.gamma * ith) * rho;
    const long long mi = mg0(G, P);
    M[mi] = from_f64<T>(b00 * idt);
    if (nf == 2) {
        M[1 * nc + mi] = from_f64<T>(b01 * idt);
        M[2 * nc + mi] = from_f64<T>(b10 * idt);
        M[3 * nc + mi] = from_f64<T>(b11 * idt);
    }
    C[PcLr * nc + cc] = from_f64<T>(L[cc]);
    C[PcLE * nc + cc] = from_f64<T>(L[nc + cc]);
    C[PcInvRho * nc + cc] = from_f64<T>(irho);
    C[PcE * nc + cc] = from_f64<T>(E);
    C[PcDpdrho * nc + cc] = from_f64<T>(Tc);
    C[PcDpde * nc + cc] = from_f64<T>(dpde);
    C[PcInvDpdrho * nc + cc] = from_f64<T>(iT);
    C[PcCde * nc + cc] = from_f64<T>(G.igamma * irho);
    // r_p = Pr r_rho + PE r_E - dpde <u.r_u>: first row of dV/dU in the
    // product form printed in Sect. 3.2 (no cancellation between terms)
    const double Pr = Tc - G.gm1 * E;
    C[PcPr * nc + cc] = from_f64<T>(Pr);
    C[PcPE * nc + cc] = from_f64<T>(G.gm1);
    if (sizeof(T) == 8) {
        C[PcQ0 * nc + cc] = from_f64<T>(b00);
        if (nf == 2) {
            C[PcQ1 * nc + cc] = from_f64<T>(b01);
            C[PcQ2 * nc + cc] = from_f64<T>(b10);
            C[PcQ3 * nc + cc] = from_f64<T>(b11);
        }
    } else if (nf == 1) {
        C[PcQ0 * nc + cc] = from_f64<T>(b00 * Pr);
        C[PcQ1 * nc + cc] = from_f64<T>(b00 * G.gm1);
        C[PcQ2 * nc + cc] = from_f64<T>(b00 * dpde);
    } else {
        // rhs = B^-1 (r_p, r_e) with r_e = (r_E - E r_rho)/rho - <u.r_u>
        C[PcQ0 * nc + cc] = from_f64<T>(ic1 * irho);
        C[PcQ1 * nc + cc] = (T)0;
        C[PcQ2 * nc + cc] = (T)0;
        C[PcQ3 * nc + cc] = from_f64<T>(-ith * (Tc + E));
        C[PcQ4 * nc + cc] = from_f64<T>(ith);
        C[PcQ5 * nc + cc] = from_f64<T>(ith * rho);
    }
    C[PcRinvR * nc + cc] = from_f64<T>(Rinv[cc]);
    C[PcRinvE * nc + cc] = from_f64<T>(Rinv[nc + cc]);
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const bool wall = is_wall_slot(G, c, P);
        const double irhof = inv[2 + c];
        K[(0 * ND + c) * nc + mi] = from_f64<T>(wall ? 0.0 : irhof * G.idx2[c]);
        if (nf == 2) {
            const double chis = G.has_cond && !wall ? chi[cc + om1[c]] + chi[cc] : 0.0;
            K[(1 * ND + c) * nc + mi] = from_f64<T>(chis * (0.5 * G.gm1 * G.idx2[c]));
        }
        const double u = wall ? 0.0 : X[(2 + c) * nc + cc];
        C[(PcLu + c) * nc + cc] = from_f64<T>(L[(2 + c) * nc + cc]);
        C[(PcU + c) * nc + cc] = from_f64<T>(u);
        C[(PcInvRhof + c) * nc + cc] = from_f64<T>(wall ? 0.0 : irhof);
        C[(PcThf + c) * nc + cc] = from_f64<T>(wall ? 0.0 : G.theta * G.idx[c] * irhof);
        C[(PcRinvU + c) * nc + cc] = from_f64<T>(Rinv[(2 + c) * nc + cc]);
    }
}

#define CELL_LAUNCH_T(KERNEL, T, ...)                                                     \
    do {                                                                                  \
        CellLaunch cl_ = cell_launch(G.n);                                                \
        ++g_launch_count;                                                                 \
        if (G.ndim == 3) launch_k(KERNEL<3, T>, cl_.grid, cl_.block, 0, s, __VA_ARGS__);        \
        else launch_k(KERNEL<2, T>, cl_.grid, cl_.block, 0, s, __VA_ARGS__);                    \
    } while (0)

template <typename T>
void launch_pc_setup(const Grid& G, const double* X, const double* Tg, const double* chi, const double* L,
                     const double* Rinv, double dt, int nf, T* C, MGLevel& L0, cudaStream_t s) {
    CELL_LAUNCH_T(k_pc_setup, T, G, X, Tg, chi, L, Rinv, 1.0 / (G.theta * G.theta * dt), 1.0 / G.theta, 1.0 / dt, nf, C,
                  (T*)L0.M, (T*)L0.K);
}
template void launch_pc_setup<double>(const Grid&, const double*, const double*, const double*, const double*,
                                      const double*, double, int, double*, MGLevel&, cudaStream_t);
template void launch_pc_setup<float>(const Grid&, const double*, const double*, const double*, const double*,
                                     const double*, double, int, float*, MGLevel&, cudaStream_t);

// The scaling fields of C alone, as k_pc_setup writes them (the frozen-
// coefficient option renews only these at later Newton iterates).
template <int ND, typename T>
__global__ void k_pc_rescale(Grid G, const double* L, const double* Rinv,
                             T* C) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const long long nc = G.ncell;
    C[PcLr * nc + cc] = from_f64<T>(L[cc]);
    C[PcLE * nc + cc] = from_f64<T>(L[nc + cc]);
    C[PcRinvR * nc + cc] = from_f64<T>(Rinv[cc]);
    C[PcRinvE * nc + cc] = from_f64<T>(Rinv[nc + cc]);
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        C[(PcLu + c) * nc + cc] = from_f64<T>(L[(2 + c) * nc + cc]);
        C[(PcRinvU + c) * nc + cc] = from_f64<T>(Rinv[(2 + c) * nc + cc]);
    }
}

template <typename T>
void launch_pc_rescale(const Grid& G, const double* L, const double* Rinv, T* C, cudaStream_t s) {
    CELL_LAUNCH_T(k_pc_rescale, T, G, L, Rinv, C);
}
template void launch_pc_rescale<double>(const Grid&, const double*, const double*, double*, cudaStream_t);
template void launch_pc_rescale<float>(const Grid&, const double*, const double*, float*, cudaStream_t);

// ---------------------------------------------------------------------------
// transform in: r_V and the multigrid right-hand side
// ---------------------------------------------------------------------------

// r_rho at the cell (pos + off) with ghost mapping
template <typename T, typename TV>
__device__ __forceinline__ T rrho_at(const Grid& G, const T* C, const TV* v, T s, const Idx3& P, int o0, int o1,
                                     int o2) {
    int a = cell_map(P.i[0] + o0, G.n[0], G.bc[0]);
    int b = cell_map(P.i[1] + o1, G.n[1], G.bc[1]);
    int c = cell_map(P.i[2] + o2, G.n[2], G.bc[2]);
    long long j = flat(G, a, b, c);
    return C[PcLr * G.ncell + j] * (s * (T)v[j]);
}

// r_u on the lower face of cell Q in direction c (zero at a wall slot)
template <typename T, typename TV>
__device__ __forceinline__ T ru_at(const Grid& G, const T* C, const TV* v, T s, int c, const Idx3& Q) {
    const long long nc = G.ncell;
    const long long j = flat(G, Q.i[0], Q.i[1], Q.i[2]);
    int o[3] = {0, 0, 0};
    o[c] = -1;
    T rl = rrho_at<T, TV>(G, C, v, s, Q, o[0], o[1], o[2]);
    T r0 = C[PcLr * nc + j] * (s * (T)v[j]);
    T rb = (T)0.5 * (rl + r0);
    T ruv = C[(PcLu + c) * nc + j] * (s * (T)v[(2 + c) * nc + j]);
    return (ruv - C[(PcU + c) * nc + j] * rb) * C[(PcInvRhof + c) * nc + j];
}

template <int ND, typename T>
__global__ void k_precond_in(Grid G, const T* C, const T* v,
                             const double* vscale, int vslot, int nf, T* rp,
                             T* re, T* ru, T* rhs, T* x0,
                             const T* D, int nu1) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    const long long nc = G.ncell;
    const T s = vslot >= 0 ? (T)vscale[vslot] : (T)1;
    T r_rho = C[PcLr * nc + cc] * (s * v[cc]);
    T r_E = C[PcLE * nc + cc] * (s * v[nc + cc]);
    T r_e = (r_E - C[PcE * nc + cc] * r_rho) * C[PcInvRho * nc + cc];
    T ruv[ND];
    T dot_ur = (T)0;
#pragma unroll
    for (int c = 0; c < ND; ++c) ruv[c] = ru_at<T, T>(G, C, v, s, c, P);
    if (G.energy_form == 1) {
        T dot = (T)0;
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            Idx3 Q = P;
            T uu = (T)0, au = (T)0;
            if (!(G.bc[d] == 1 && P.i[d] + 1 == G.n[d])) {
                Q.i[d] = (P.i[d] + 1 == G.n[d]) ? 0 : P.i[d] + 1;
                uu = C[(PcU + d) * nc + flat(G, Q.i[0], Q.i[1], Q.i[2])];
                au = ru_at<T, T>(G, C, v, s, d, Q);
            }
            dot = dot + (T)0.5 * (C[(PcU + d) * nc + cc] * ruv[d] + uu * au);
        }
        r_e = r_e - dot;
        dot_ur = dot;
    }
#pragma unroll
    for (int c = 0; c < ND; ++c) ru[c * nc + cc] = ruv[c];
    // r_p and r_e are kept for the back substitution of the sound-only scheme
    if (nf == 1) re[cc] = r_e;
    const long long mi = mg0(G, P);
    T b0, b1 = (T)0;
    if (sizeof(T) == 8) {
        // double: the oracle's order, r_p = dp/drho r_rho + dp/de r_e, rhs = B^-1 (r_p, r_e)
        T r_p = C[PcDpdrho * nc + cc] * r_rho + C[PcDpde * nc + cc] * r_e;
        if (nf == 1) {
            rp[cc] = r_p;
            b0 = r_p * C[PcQ0 * nc + cc];
        } else {
            b0 = C[PcQ0 * nc + cc] * r_p + C[PcQ1 * nc + cc] * r_e;
            b1 = C[PcQ2 * nc + cc] * r_p + C[PcQ3 * nc + cc] * r_e;
        }
    } else {
        // float: folded coefficients (see PcQ*), free of cancellation
        if (nf == 1) rp[cc] = C[PcPr * nc + cc] * r_rho + C[PcPE * nc + cc] * r_E - C[PcDpde * nc + cc] * dot_ur;
        b0 = C[PcQ0 * nc + cc] * r_rho + C[PcQ1 * nc + cc] * r_E - C[PcQ2 * nc + cc] * dot_ur;
        if (nf == 2)
            b1 = C[PcQ3 * nc + cc] * r_rho + C[PcQ4 * nc + cc] * r_E - C[PcQ5 * nc + cc] * dot_ur;
    }
    rhs[mi] = b0;
    if (nf == 2) rhs[nc + mi] = b1;
    // multigrid start: the zero start's first half sweep, pointwise on the red
    // cells (the black ones are overwritten before they are read)
    if (nu1 == 0) {
        x0[mi] = (T)0;
        if (nf == 2) x0[nc + mi] = (T)0;
    } else if (((P.i[0] + P.i[1] + P.i[2]) & 1) == 0) {
        if (nf == 1) {
            x0[mi] = D[mi] * b0;
        } else {
            x0[mi] = D[mi] * b0 + D[nc + mi] * b1;
            x0[nc + mi] = D[2 * nc + mi] * b0 + D[3 * nc + mi] * b1;
        }
    }
}

template <typename T>
void launch_precond_in(const Grid& G, const T* C, const T* v, const double* vscale, int vslot, int nf, T* rp, T* re,
                       T* ru, MGLevel& L0, cudaStream_t s, int nu1) {
    CELL_LAUNCH_T(k_precond_in, T, G, C, v, vscale, vslot, nf, rp, re, ru, (T*)L0.rhs, (T*)L0.x,
                  (const T*)L0.D, nu1);
}
template void launch_precond_in<double>(const Grid&, const double*, const double*, const double*, int, int, double*,
                                        double*, double*, MGLevel&, cudaStream_t, int);
template void launch_precond_in<float>(const Grid&, const float*, const float*, const double*, int, int, float*,
                                       float*, float*, MGLevel&, cudaStream_t, int);

// ---------------------------------------------------------------------------
// back substitution and transform out
// ---------------------------------------------------------------------------

// du on the lower face of cell Q in direction c
template <typename T>
__device__ __forceinline__ T du_at(const Grid& G, const T* C, T dt, const T* ru, const T* dp, int c, const Idx3& Q) {
    const long long nc = G.ncell;
    const long long j = flat(G, Q.i[0], Q.i[1], Q.i[2]);
    int o[3] = {0, 0, 0};
    o[c] = -1;
    int a = cell_map(Q.i[0] + o[0], G.n[0], G.bc[0]);
    int b = cell_map(Q.i[1] + o[1], G.n[1], G.bc[1]);
    int cz = cell_map(Q.i[2] + o[2], G.n[2], G.bc[2]);
    Idx3 L;
    L.i[0] = a; L.i[1] = b; L.i[2] = cz;
    // dp lives in the (colour-split) multigrid array of level 0
    return dt * (ru[c * nc + j] - C[(PcThf + c) * nc + j] * (dp[mg0(G, Q)] - dp[mg0(G, L)]));
}

// One wave of blocks, each visiting cell tiles with a grid stride and
// reducing its partial |z|^2 once: with one tile per block the block-wide
// reduction (two barriers per 128 cells) cost a quarter of the kernel.
template <int ND, typename T>
__global__ void k_precond_out(Grid G, const T* C, double dt_d, double idt_d, int nf,
                              const T* rp,
                              const T* re, const T* ru, const T* x,
                              T* z, ZFinish Z, int ntiles) {
    pdl_wait();
    __shared__ double sh[32];
    // |z|^2: in double for a double z; for a float z as a compensated float
    // pair (no FP64 instruction per element), converted once per thread, or
    // redone in double from the stored z by a thread whose values are too
    // large or too small for float squares (sq_range_unsafe)
    double acc = 0.0;
    CompF accf = {0.f, 0.f};
    float mx = 0.f;
    const long long nc = G.ncell;
    const T dt = (T)dt_d, idt = (T)idt_d;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        Idx3 P;
        long long cc;
        if (!cell_pos_tile(G.n, tile, P, cc)) continue;
        const long long mi = mg0(G, P);
        const T dp = x[mi];
        T de;
        if (nf == 1) de = dt * (re[cc] + (dp * idt - rp[cc]) * C[PcCde * nc + cc]);
        else de = x[nc + mi];
        T du[ND];
#pragma unroll
        for (int c = 0; c < ND; ++c) du[c] = du_at<T>(G, C, dt, ru, x, c, P);
        T dE = de;
        if (G.energy_form == 1) {
            T dot = (T)0;
#pragma unroll
            for (int d = 0; d < ND; ++d) {
                T uu = (T)0, au = (T)0;
                if (!(G.bc[d] == 1 && P.i[d] + 1 == G.n[d])) {
                    Idx3 Q = P;
                    Q.i[d] = (P.i[d] + 1 == G.n[d]) ? 0 : P.i[d] + 1;
                    uu = C[(PcU + d) * nc + flat(G, Q.i[0], Q.i[1], Q.i[2])];
                    au = du_at<T>(G, C, dt, ru, x, d, Q);
                }
                dot = dot + (T)0.5 * (C[(PcU + d) * nc + cc] * du[d] + uu * au);
            }
            dE = de + dot;
        }
        T drho = (dp - C[PcDpde * nc + cc] * de) * C[PcInvDpdrho * nc + cc];
        T out[2 + ND];
        out[0] = drho * C[PcRinvR * nc + cc];
        out[1] = dE * C[PcRinvE * nc + cc];
#pragma unroll
        for (int c = 0; c < ND; ++c) out[2 + c] = du[c] * C[(PcRinvU + c) * nc + cc];
#pragma unroll
        for (int k = 0; k < 2 + ND; ++k) {
            z[k * nc + cc] = out[k];
            if (sizeof(T) == 8) {
                const double zd = (double)out[k];
                acc += zd * zd;
            } else {
                const float zf = (float)out[k];
                comp_fma(accf, zf, zf);
                mx = fmaxf(mx, fabsf(zf));
            }
        }
    }
    if (sizeof(T) != 8) {
        if (sq_range_unsafe(mx)) {
            for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
                Idx3 P;
                long long cc;
                if (!cell_pos_tile(G.n, tile, P, cc)) continue;
#pragma unroll
                for (int k = 0; k < 2 + ND; ++k) {
                    const double zd = (double)z[k * nc + cc];
                    acc += zd * zd;
                }
            }
        } else {
            acc = (double)accf.s + (double)accf.e;
        }
    }
    finish_znorm(acc, sh, Z);
}

// blocks of one wave of k_precond_out (occupancy query, once per kernel)
template <auto FN>
static int one_wave(int threads) {
    static const int g = [threads] {
        int dev = 0, nsm = 0, occ = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, FN, threads, 0);
        long long w = (long long)(nsm > 0 ? nsm : 1) * (occ > 0 ? occ : 1);
        return (int)(w < kMaxRedBlocks ? w : kMaxRedBlocks);
    }();
    return g;
}

template <typename T>
void launch_precond_out(const Grid& G, const T* C, double dt, int nf, const T* rp, const T* re, const T* ru,
                        const MGLevel& L0, T* z, const ZFinish& Z, cudaStream_t s) {
    CellLaunch cl = cell_launch(G.n);
    const long long nt = (long long)cl.grid.x * cl.grid.y * cl.grid.z;
    const int ntiles = (int)nt;
    int g = G.ndim == 3 ? one_wave<k_precond_out<3, T>>(cl.block.x * cl.block.y)
                        : one_wave<k_precond_out<2, T>>(cl.block.x * cl.block.y);
    if (g > ntiles) g = ntiles;
    ++g_launch_count;
    if (G.ndim == 3)
        launch_k(k_precond_out<3, T>, g, cl.block, 0, s, G, C, dt, 1.0 / dt, nf, rp, re, ru, (const T*)L0.x, z, Z, ntiles);
    else
        launch_k(k_precond_out<2, T>, g, cl.block, 0, s, G, C, dt, 1.0 / dt, nf, rp, re, ru, (const T*)L0.x, z, Z, ntiles);
}
template void launch_precond_out<double>(const Grid&, const double*, double, int, const double*, const double*,
                                        const double*, const MGLevel&, double*, const ZFinish&, cudaStream_t);
template void launch_precond_out<float>(const Grid&, const float*, double, int, const float*, const float*,
                                       const float*, const MGLevel&, float*, const ZFinish&, cudaStream_t);

}  // namespace jfnk
