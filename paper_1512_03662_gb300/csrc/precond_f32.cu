// The FP32 preconditioner's transforms for the internal energy form, with L and
// R of the same state as the semi-implicit coefficients (precond.cu holds the
// general ones: double, total energy, frozen coefficients).
//
// Everything that is a product of coefficients is formed once per
// linearisation in double and rounded once, so an apply reads 13 values per cell
// and writes 8 on the way in, and 14 and 5 on the way out (22 and 5, 20 and 5 in
// the general form).  With the ideal gas' closed forms (k_pc_setup) and L_rho =
// rho, L_E = rho e, R_rho = rho, R_e = e:
//   r_rho = rho v_rho
//   rhs   = ( v_rho / c1,  (rho e / theta) (v_e - gamma v_rho) )           two fields
//         = v_e / (c1 gamma)                                              one field
//   z_u'  = dt (al v_u - be (r_rho + r_rho of the lower cell))  = dt R_u^-1 r_u
//   z_rho = (dp - (gamma-1) rho de) / (rho T),   z_e = de / e
//   de    = dt e (v_e / gamma - v_rho) + dp / (gamma rho)                 one field
// (T + e = gamma e).  The differences of v_e and v_rho vanish for isentropic
// perturbations, so their factor is taken as the sum of two floats.
//   z_u   = z_u' - g (dp - dp of the lower cell)
// with al = R_u^-1 L_u / rho_f, be = R_u^-1 u / (2 rho_f) and
// g = dt theta R_u^-1 / (dx rho_f), zero on wall faces.  (dt stays outside al and
// be: dt / rho alone may leave the range of a float.)  z_u' is kept in the
// output vector itself.  Four cells along x per thread, 16-byte accesses.
#include "common.cuh"
#include "kernels.h"

namespace jfnk {

// Fields of C.  CfE: rho e / theta with two fields, e with one; CfA: 1 / (rho T);
// CfB: (gamma-1) rho; CfIE: 1 / e; CfCde: 1 / (gamma rho), one field only
enum { CfRho = 0, CfE, CfA, CfB, CfIE, CfCde, CfAl, CfBe = CfAl + 3, CfG = CfBe + 3 };

// Coefficients of one cell; products and reciprocals on the integer pipes with
// checked Ops (false, nothing written, where one was out of range)
template <int ND, int NF, class O>
__device__ __forceinline__ bool pcf_setup_cell(O ops, const Grid& G, const double* __restrict__ X,
                                               const double* __restrict__ Tg, const double* __restrict__ chi,
                                               const double* __restrict__ L, const double* __restrict__ Rinv,
                                               double dt, double ic1, double ith, double idt, float* __restrict__ C,
                                               float* __restrict__ M, float* __restrict__ K, const Idx3& P,
                                               long long cc) {
    const long long nc = G.ncell;
    const double rho = X[cc], Tc = Tg[cc], irho = Rinv[cc];
    const double iT = ops.recip(Tc);
    const double A = ops.mul(irho, iT);
    float m[4], cf[4], k[2 * ND], al[ND], be[ND], g[ND];
    if (NF == 2) {
        m[0] = d2f_rn(ops.mul(ic1 * idt, A));
        m[1] = d2f_rn(ops.mul(-G.gm1 * ic1 * idt, iT));
        m[2] = d2f_rn(-ith * idt);
        m[3] = d2f_rn(ops.mul(G.gamma * ith * idt, rho));
    } else {
        m[0] = d2f_rn(ops.mul(ic1 * G.igamma * idt, A));
    }
    cf[0] = d2f_rn(A);
    cf[1] = d2f_rn(ops.mul(G.gm1, rho));
    cf[2] = NF == 1 ? d2f_rn(ops.mul(G.igamma, irho)) : 0.f;
    cf[3] = NF == 2 ? d2f_rn(ops.mul(ith, L[nc + cc])) : d2f_rn(X[nc + cc]);
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        const bool wall = is_wall_slot(G, c, P);
        const int o = cell_off(G, P, c, -1);
        const double irs = ops.recip(X[cc + o] + rho);                    // 1 / (2 rho_f)
        k[c] = wall ? 0.f : d2f_rn(ops.mul(2.0 * G.idx2[c], irs));
        if (NF == 2) {
            const double chis = G.has_cond ? chi[cc + o] + chi[cc] : 0.0;
            k[ND + c] = wall ? 0.f : d2f_rn(ops.mul(chis, 0.5 * G.gm1 * G.idx2[c]));
        }
        const double q = ops.mul(ops.mul(Rinv[(2 + c) * nc + cc], irs), 2.0);           // R_u^-1 / rho_f
        al[c] = wall ? 0.f : d2f_rn(ops.mul(q, L[(2 + c) * nc + cc]));
        be[c] = wall ? 0.f : 0.5f * d2f_rn(ops.mul(q, X[(2 + c) * nc + cc]));
        g[c] = wall ? 0.f : d2f_rn(ops.mul(q, dt * G.theta * G.idx[c]));
    }
    if (!ops.valid()) return false;
    const long long mi = rb_index(G.n[0], G.n[1], nc, P.i[0], P.i[1], P.i[2]);
#pragma unroll
    for (int q = 0; q < NF * NF; ++q) M[q * nc + mi] = m[q];
#pragma unroll
    for (int q = 0; q < NF * ND; ++q) K[q * nc + mi] = k[q];
    C[CfRho * nc + cc] = d2f_rn(rho);
    C[CfE * nc + cc] = cf[3];
    C[CfA * nc + cc] = cf[0];
    C[CfB * nc + cc] = cf[1];
    C[CfIE * nc + cc] = d2f_rn(Rinv[nc + cc]);
    if (NF == 1) C[CfCde * nc + cc] = cf[2];
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        C[(CfAl + c) * nc + cc] = al[c];
        C[(CfBe + c) * nc + cc] = be[c];
        C[(CfG + c) * nc + cc] = g[c];
    }
    return true;
}

// plain operators for the redo; recip is a division
struct PcfFp : FpOps {
    __device__ __forceinline__ double recip(double d) { return 1.0 / d; }
};

template <int ND, int NF>
__device__ __noinline__ void pcf_setup_cell_fp64(const Grid G, const double* __restrict__ X,
                                                 const double* __restrict__ Tg, const double* __restrict__ chi,
                                                 const double* __restrict__ L, const double* __restrict__ Rinv,
                                                 double dt, double ic1, double ith, double idt, float* __restrict__ C,
                                                 float* __restrict__ M, float* __restrict__ K, const Idx3 P,
                                                 long long cc) {
    pcf_setup_cell<ND, NF>(PcfFp(), G, X, Tg, chi, L, Rinv, dt, ic1, ith, idt, C, M, K, P, cc);
}

// Bound by the ALU pipe (70 % busy): 197 us at 128^3 with at least 12 blocks of 128
// threads per SM (40 registers), 8 % more with 8; 1.50 ms at 256^3, where the general
// setup with its products, conductivities and determinant on the FP64 pipe took
// 3.59 ms.
template <int ND, int NF>
__global__ void __launch_bounds__(128, 12) k_pcf_setup(Grid G, const double* X,
                                                      const double* Tg, const double* chi,
                                                      const double* L, const double* Rinv,
                                                      double dt, double ic1, double ith, double idt,
                                                      float* C, float* M,
                                                      float* K) {
    pdl_wait();
    Idx3 P;
    long long cc;
    if (!cell_pos(G.n, P, cc)) return;
    if (!pcf_setup_cell<ND, NF>(IntOps(), G, X, Tg, chi, L, Rinv, dt, ic1, ith, idt, C, M, K, P, cc))
        pcf_setup_cell_fp64<ND, NF>(G, X, Tg, chi, L, Rinv, dt, ic1, ith, idt, C, M, K, P, cc);
}

// dispatch over the dimension and the field count
#define PCF_LAUNCH(KERNEL, GRID, BLOCK, ...)                                                  \
    do {                                                                                      \
        ++g_launch_count;                                                                     \
        if (nf == 1 && G.ndim == 3) launch_k(KERNEL<3, 1>, GRID, BLOCK, 0, s, __VA_ARGS__);         \
        else if (nf == 1) launch_k(KERNEL<2, 1>, GRID, BLOCK, 0, s, __VA_ARGS__);                   \
        else if (G.ndim == 3) launch_k(KERNEL<3, 2>, GRID, BLOCK, 0, s, __VA_ARGS__);               \
        else launch_k(KERNEL<2, 2>, GRID, BLOCK, 0, s, __VA_ARGS__);                                \
    } while (0)

void launch_pcf_setup(const Grid& G, const double* X, const double* Tg, const double* chi, const double* L,
                      const double* Rinv, double dt, int nf, float* C, MGLevel& L0, cudaStream_t s) {
    const CellLaunch cl = cell_launch(G.n);
    PCF_LAUNCH(k_pcf_setup, cl.grid, cl.block, G, X, Tg, chi, L, Rinv, dt, 1.0 / (G.theta * G.theta * dt),
               1.0 / G.theta, 1.0 / dt, C, (float*)L0.M, (float*)L0.K);
}

struct F4 {
    float v[4];
};
__device__ __forceinline__ F4 ld4(const float* p) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    return F4{{q.x, q.y, q.z, q.w}};
}
__device__ __forceinline__ void st4(float* p, const F4& a) {
    *reinterpret_cast<float4*>(p) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
}

// Cells a .. a+3 of row (b,c): flat index i (a multiple of 4), and in the
// colour-split multigrid arrays the even and odd cells as pairs at je and jo
struct Quad {
    int a, b, c;
    long long i, je, jo;
    __device__ __forceinline__ bool set(const Grid& G, int t, int bb, int cz) {
        a = 4 * t;
        b = bb;
        c = cz;
        if (a >= G.n[0] || b >= G.n[1]) return false;
        i = ((long long)c * G.n[1] + b) * G.n[0] + a;
        set_pairs(G, i, (b + c) & 1, je, jo);
        return true;
    }
    __device__ __forceinline__ static void set_pairs(const Grid& G, long long i, int odd, long long& je,
                                                     long long& jo) {
        const long long half = G.ncell >> 1;
        je = (odd ? half : 0) + (i >> 1);
        jo = (odd ? 0 : half) + (i >> 1);
    }
    // flat index of the quad's row one cell lower along d = 1, 2 (mirrored onto
    // itself at a wall), and the row's parity
    __device__ __forceinline__ long long lower(const Grid& G, int d, int& odd) const {
        const int k = d == 1 ? b : c, m = cell_map(k - 1, G.n[d], G.bc[d]);
        odd = (b + c + m - k) & 1;
        return i + (long long)(m - k) * (d == 1 ? G.n[0] : (long long)G.n[0] * G.n[1]);
    }
};
__device__ __forceinline__ F4 ld_pairs(const float* x, long long je, long long jo) {
    const float2 e = *reinterpret_cast<const float2*>(x + je), o = *reinterpret_cast<const float2*>(x + jo);
    return F4{{e.x, o.x, e.y, o.y}};
}
__device__ __forceinline__ void st_pairs(float* x, long long je, long long jo, const F4& a) {
    *reinterpret_cast<float2*>(x + je) = make_float2(a.v[0], a.v[2]);
    *reinterpret_cast<float2*>(x + jo) = make_float2(a.v[1], a.v[3]);
}

// 197 us at 256^3 with two fields, 71 B per cell at 6.0 TB/s; the general transform
// (one cell per thread, 120 B) takes 448 us.
template <int ND, int NF>
__global__ void __launch_bounds__(128) k_pcf_in(Grid G, const float* C, const float* v,
                                                const double* vscale, int vslot, float ic1, float gh, float gl,
                                                float dt, float* z, float* q, float* rhs, float* x0, const float* D,
                                                int nu1) {
    pdl_wait();
    Quad Q;
    if (!Q.set(G, blockIdx.x * blockDim.x + threadIdx.x, blockIdx.y * blockDim.y + threadIdx.y, blockIdx.z)) return;
    const long long nc = G.ncell, i = Q.i;
    const float s = vslot >= 0 ? (float)vscale[vslot] : 1.f;
    const F4 rho = ld4(C + CfRho * nc + i), E = ld4(C + CfE * nc + i);
    F4 vr = ld4(v + i), ve = ld4(v + nc + i), w, b0, b1;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        vr.v[k] = s * vr.v[k];
        ve.v[k] = s * ve.v[k];
        w.v[k] = rho.v[k] * vr.v[k];                                      // r_rho
    }
    // velocity rows
    const long long il = i + (cell_map(Q.a - 1, G.n[0], G.bc[0]) - Q.a);
    const float wl0 = C[CfRho * nc + il] * (s * v[il]);
#pragma unroll
    for (int c = 0; c < ND; ++c) {
        F4 wl;
        if (c == 0) {
            wl = F4{{wl0, w.v[0], w.v[1], w.v[2]}};
        } else {
            int odd;
            const long long j = Q.lower(G, c, odd);
            const F4 rl = ld4(C + CfRho * nc + j), vl = ld4(v + j);
#pragma unroll
            for (int k = 0; k < 4; ++k) wl.v[k] = rl.v[k] * (s * vl.v[k]);
        }
        const F4 vu = ld4(v + (2 + c) * nc + i), al = ld4(C + (CfAl + c) * nc + i), be = ld4(C + (CfBe + c) * nc + i);
        F4 o;
#pragma unroll
        for (int k = 0; k < 4; ++k) o.v[k] = dt * (al.v[k] * (s * vu.v[k]) - be.v[k] * (wl.v[k] + w.v[k]));
        st4(z + (2 + c) * nc + i, o);
    }
    // right-hand side
    if (NF == 2) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            b0.v[k] = ic1 * vr.v[k];
            b1.v[k] = E.v[k] * fmaf(-gl, vr.v[k], fmaf(-gh, vr.v[k], ve.v[k]));
        }
        st_pairs(rhs, Q.je, Q.jo, b0);
        st_pairs(rhs + nc, Q.je, Q.jo, b1);
    } else {
        // the part of de without dp is kept in q
        F4 qo;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            b0.v[k] = ic1 * ve.v[k];
            qo.v[k] = dt * (E.v[k] * fmaf(gl, ve.v[k], fmaf(gh, ve.v[k], -vr.v[k])));
        }
        st_pairs(rhs, Q.je, Q.jo, b0);
        st4(q + i, qo);
    }
    // multigrid start: the zero start's first half sweep on the red cells, one
    // of the quad's two pairs
    if (nu1 == 0) {
        const F4 zero = {{0.f, 0.f, 0.f, 0.f}};
        st_pairs(x0, Q.je, Q.jo, zero);
        if (NF == 2) st_pairs(x0 + nc, Q.je, Q.jo, zero);
        return;
    }
    const bool even = Q.je < Q.jo;                                        // the even cells are red
    const long long j = even ? Q.je : Q.jo;
    const float g0x = even ? b0.v[0] : b0.v[1], g0y = even ? b0.v[2] : b0.v[3];
    auto ld2 = [&](int f) { return *reinterpret_cast<const float2*>(D + f * nc + j); };
    if (NF == 1) {
        const float2 d = ld2(0);
        *reinterpret_cast<float2*>(x0 + j) = make_float2(d.x * g0x, d.y * g0y);
    } else {
        const float g1x = even ? b1.v[0] : b1.v[1], g1y = even ? b1.v[2] : b1.v[3];
        const float2 d0 = ld2(0), d1 = ld2(1), d2 = ld2(2), d3 = ld2(3);
        *reinterpret_cast<float2*>(x0 + j) = make_float2(d0.x * g0x + d1.x * g1x, d0.y * g0y + d1.y * g1y);
        *reinterpret_cast<float2*>(x0 + nc + j) = make_float2(d2.x * g0x + d3.x * g1x, d2.y * g0y + d3.y * g1y);
    }
}

// blocks of 128 threads, four cells along x each
static CellLaunch quad_launch(const Grid& G) {
    const int nt = G.n[0] / 4;
    int bx = 1;
    while (bx < nt && bx < 32) bx *= 2;
    const int by = 128 / bx;
    CellLaunch L;
    L.block = dim3(bx, by, 1);
    L.grid = dim3((nt + bx - 1) / bx, (G.n[1] + by - 1) / by, G.n[2]);
    return L;
}

void launch_pcf_in(const Grid& G, const float* C, const float* v, const double* vscale, int vslot, double dt, int nf,
                   float* z, float* q, MGLevel& L0, cudaStream_t s, int nu1) {
    const CellLaunch cl = quad_launch(G);
    const double c1 = G.theta * G.theta * dt;
    const double g = nf == 2 ? G.gamma : G.igamma;                        // as the sum of two floats
    const float gh = (float)g, gl = (float)(g - (double)gh);
    PCF_LAUNCH(k_pcf_in, cl.grid, cl.block, G, C, v, vscale, vslot, (float)(nf == 2 ? 1.0 / c1 : G.igamma / c1), gh,
               gl, (float)dt, z, q, (float*)L0.rhs, (float*)L0.x, (const float*)L0.D, nu1);
}

// Back substitution, in place on the velocity rows of z, and partial sums of
// |z|^2: compensated float pairs, converted once per thread, or redone in
// double from the stored z by a thread whose values are too large or too small
// for float squares (sq_range_unsafe).  One wave of blocks visits the tiles of
// a quad_launch grid, so each block reduces its partial sum once.
// 160 us at 256^3 with two fields, against 345 us for the general transform.
template <int ND, int NF>
__global__ void __launch_bounds__(128) k_pcf_out(Grid G, const float* C, const float* q,
                                                 const float* x, float* z,
                                                 ZFinish Z, int gx, int gy, int ntiles) {
    pdl_wait();
    __shared__ double sh[32];
    CompF acc = {0.f, 0.f};
    float mx = 0.f;
    const long long nc = G.ncell;
    auto tile_quad = [&](int tile, Quad& Q) {
        const int r = tile / gx;
        return Q.set(G, (tile - r * gx) * blockDim.x + threadIdx.x, (r % gy) * blockDim.y + threadIdx.y, r / gy);
    };
    auto count = [&](const F4& o) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            comp_fma(acc, o.v[k], o.v[k]);
            mx = fmaxf(mx, fabsf(o.v[k]));
        }
    };
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        Quad Q;
        if (!tile_quad(tile, Q)) continue;
        const long long i = Q.i;
        const F4 dp = ld_pairs(x, Q.je, Q.jo);
        F4 de;
        if (NF == 2) {
            de = ld_pairs(x + nc, Q.je, Q.jo);
        } else {
            const F4 qi = ld4(q + i), cde = ld4(C + CfCde * nc + i);
#pragma unroll
            for (int k = 0; k < 4; ++k) de.v[k] = qi.v[k] + dp.v[k] * cde.v[k];
        }
        const F4 A = ld4(C + CfA * nc + i), B = ld4(C + CfB * nc + i), IE = ld4(C + CfIE * nc + i);
        F4 o0, o1;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            o0.v[k] = A.v[k] * (dp.v[k] - B.v[k] * de.v[k]);
            o1.v[k] = IE.v[k] * de.v[k];
        }
        st4(z + i, o0);
        st4(z + nc + i, o1);
        count(o0);
        count(o1);
        // dp of the cell below the quad along x: an odd cell of this row (or,
        // at a wall, the quad's own first cell, whose g is zero)
        const int al = cell_map(Q.a - 1, G.n[0], G.bc[0]);
        const float dl0 = x[rb_index(G.n[0], G.n[1], nc, al, Q.b, Q.c)];
#pragma unroll
        for (int c = 0; c < ND; ++c) {
            F4 dl;
            if (c == 0) {
                dl = F4{{dl0, dp.v[0], dp.v[1], dp.v[2]}};
            } else {
                int odd;
                long long je, jo;
                const long long j = Q.lower(G, c, odd);
                Quad::set_pairs(G, j, odd, je, jo);
                dl = ld_pairs(x, je, jo);
            }
            const F4 g = ld4(C + (CfG + c) * nc + i);
            F4 o = ld4(z + (2 + c) * nc + i);
#pragma unroll
            for (int k = 0; k < 4; ++k) o.v[k] = o.v[k] - g.v[k] * (dp.v[k] - dl.v[k]);
            st4(z + (2 + c) * nc + i, o);
            count(o);
        }
    }
    double sum = (double)acc.s + (double)acc.e;
    if (sq_range_unsafe(mx)) {
        sum = 0.0;
        for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
            Quad Q;
            if (!tile_quad(tile, Q)) continue;
            for (int f = 0; f < 2 + ND; ++f)
                for (int k = 0; k < 4; ++k) {
                    const double zd = (double)z[f * nc + Q.i + k];
                    sum += zd * zd;
                }
        }
    }
    finish_znorm(sum, sh, Z);
}

// blocks of one wave (occupancy query, once per kernel)
template <int ND, int NF>
static int out_wave() {
    static const int g = [] {
        int dev = 0, nsm = 0, occ = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_pcf_out<ND, NF>, 128, 0);
        const long long w = (long long)(nsm > 0 ? nsm : 1) * (occ > 0 ? occ : 1);
        return (int)(w < kMaxRedBlocks ? w : kMaxRedBlocks);
    }();
    return g;
}

void launch_pcf_out(const Grid& G, const float* C, int nf, const float* q, const MGLevel& L0, float* z,
                    const ZFinish& Z, cudaStream_t s) {
    const CellLaunch cl = quad_launch(G);
    const int ntiles = (int)(cl.grid.x * cl.grid.y * cl.grid.z);
    int g = nf == 1 ? (G.ndim == 3 ? out_wave<3, 1>() : out_wave<2, 1>())
                    : (G.ndim == 3 ? out_wave<3, 2>() : out_wave<2, 2>());
    if (g > ntiles) g = ntiles;
    PCF_LAUNCH(k_pcf_out, g, cl.block, G, C, q, (const float*)L0.x, z, Z, (int)cl.grid.x, (int)cl.grid.y, ntiles);
}

}  // namespace jfnk
