// Multigrid of the preconditioner's semi-implicit system
//     M x - [div(K_p grad dp); div(K_e grad de)] = rhs
// (paper Sects. 3.3-3.4; geometric multigrid in place of the paper's AMG):
// fixed V-cycles of red-black (point-block) Gauss-Seidel, mean restriction,
// cell-centred linear prolongation, an exact one-cell coarsest level and
// coarse coefficients by averaging.  It runs in the basis precision T.
//
// What the coefficients hold.  K is stored over the squared cell width of its
// level, and D is the inverse of the diagonal block (M plus the face
// coefficients around the cell), formed once per linearisation, so a half
// sweep is x = D (rhs + sum K x_neighbour): two multiply-adds per direction
// and field and one small matrix product.  Forming the diagonal block and
// dividing in every sweep took about 65 FP64 instructions per cell of the
// 2D two-field system instead of 12, and on one SM's two FP64 lanes that was
// the time of the coarse levels; D replaces M in the sweep, so the bytes are
// the same.
#include "common.cuh"
#include "kernels.h"

namespace jfnk {

// Cells of the smallest FP32 level whose row kernels move 16 bytes per access.
// V(2,2) cycles (with all coarser levels, one / two fields): 44.1 / 56.6 us with
// vectors and 45.2 / 56.8 without at 64 x 32 x 32 = 65,536 cells, 59.4 / 81.3 and
// 63.9 / 84.6 at 64^3; 2D V(3,3) cycles 62.2 / 81.2 and 62.5 / 82.8 at 256^2, 88.8 /
// 114.3 and 94.1 / 122.1 at 512^2; below that size the two are alike.  FP64 rows
// take one cell per thread: two per thread leave the FP64 lanes fewer warps (64^3
// 107 / 176 us against 104 / 168, 128 x 128 x 64 228 / 429 against 226 / 419).
constexpr long long kRowVCells = 1 << 16;

struct LvlDev {
    int n[3];
    long long nc;
};

static inline LvlDev lvl(const MGLevel& L) {
    LvlDev d;
    for (int i = 0; i < 3; ++i) d.n[i] = L.n[i];
    d.nc = L.ncell;
    return d;
}

__device__ __forceinline__ long long lflat(const LvlDev& L, int a, int b, int c) {
    return rb_index(L.n[0], L.n[1], L.nc, a, b, c);
}

__device__ __forceinline__ int wrapi(int k, int n) { return k < 0 ? k + n : (k >= n ? k - n : k); }
__device__ __forceinline__ int wrap_up(int i, int n) { return i + 1 == n ? 0 : i + 1; }
__device__ __forceinline__ int wrap_dn(int i, int n) { return i == 0 ? n - 1 : i - 1; }

// Storage indices of the upper and lower neighbours of (a,b,c) along d
// (periodic wrap; wall neighbours carry zero face coefficients).
__device__ __forceinline__ void nb_index(const LvlDev& L, int d, int a, int b, int c, long long& ju, long long& jd) {
    if (d == 0) {
        ju = lflat(L, wrap_up(a, L.n[0]), b, c);
        jd = lflat(L, wrap_dn(a, L.n[0]), b, c);
    } else if (d == 1) {
        ju = lflat(L, a, wrap_up(b, L.n[1]), c);
        jd = lflat(L, a, wrap_dn(b, L.n[1]), c);
    } else {
        ju = lflat(L, a, b, wrap_up(c, L.n[2]));
        jd = lflat(L, a, b, wrap_dn(c, L.n[2]));
    }
}

__device__ __forceinline__ bool lvl_pos(const LvlDev& L, int i[3], long long& c) {
    i[0] = blockIdx.x * blockDim.x + threadIdx.x;
    i[1] = blockIdx.y * blockDim.y + threadIdx.y;
    i[2] = blockIdx.z;
    if (i[0] >= L.n[0] || i[1] >= L.n[1]) return false;
    c = lflat(L, i[0], i[1], i[2]);
    return true;
}

// launch over the dimension and the field count (nf = 1 or 2) as template arguments
#define MG_DISPATCH(KERNEL, GRID, BLOCK, ...)                                                 \
    do {                                                                                      \
        ++g_launch_count;                                                                     \
        if (nf == 1 && G.ndim == 3) launch_k(KERNEL<T, 1, 3>, GRID, BLOCK, 0, s, __VA_ARGS__);      \
        else if (nf == 1) launch_k(KERNEL<T, 1, 2>, GRID, BLOCK, 0, s, __VA_ARGS__);                \
        else if (G.ndim == 3) launch_k(KERNEL<T, 2, 3>, GRID, BLOCK, 0, s, __VA_ARGS__);            \
        else launch_k(KERNEL<T, 2, 2>, GRID, BLOCK, 0, s, __VA_ARGS__);                             \
    } while (0)

// the same with a vector width
#define MG_DISPATCH_V(KERNEL, V, GRID, BLOCK, ...)                                            \
    do {                                                                                      \
        ++g_launch_count;                                                                     \
        if (nf == 1 && G.ndim == 3) launch_k(KERNEL<T, 1, 3, V>, GRID, BLOCK, 0, s, __VA_ARGS__);   \
        else if (nf == 1) launch_k(KERNEL<T, 1, 2, V>, GRID, BLOCK, 0, s, __VA_ARGS__);             \
        else if (G.ndim == 3) launch_k(KERNEL<T, 2, 3, V>, GRID, BLOCK, 0, s, __VA_ARGS__);         \
        else launch_k(KERNEL<T, 2, 2, V>, GRID, BLOCK, 0, s, __VA_ARGS__);                          \
    } while (0)

// out = D v, D^T v with tr
template <typename T, int NF>
__device__ __forceinline__ void block_times(const T* D, long long nc, long long i, const T (&v)[NF], T (&out)[NF],
                                            int tr) {
    if constexpr (NF == 1) {
        out[0] = D[i] * v[0];
    } else {
        const T d01 = D[nc + i], d10 = D[2 * nc + i];
        out[0] = D[i] * v[0] + (tr ? d10 : d01) * v[1];
        out[1] = (tr ? d01 : d10) * v[0] + D[3 * nc + i] * v[1];
    }
}

// Sum of the face coefficients around a cell, two at a time: in the basis
// precision of a double basis, as an unevaluated pair of a float one.
template <typename T> struct FaceSum;
template <> struct FaceSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double a, double b) { s = s + (a + b); }
};
template <> struct FaceSum<float> {
    CompF s = {0.f, 0.f};
    __device__ __forceinline__ void add(float a, float b) {
        comp_add(s, a);
        comp_add(s, b);
    }
};

// Unevaluated pairs s + e of floats (Dekker, Numer. Math. 18 (1971) 224-242)
__device__ __forceinline__ CompF pair_norm(CompF a) {
    const float s = __fadd_rn(a.s, a.e);
    return CompF{s, __fsub_rn(a.e, __fsub_rn(s, a.s))};
}
__device__ __forceinline__ CompF pair_add(CompF a, float b) {
    comp_add(a, b);
    return pair_norm(a);
}
// x y + more, the product formed exactly
__device__ __forceinline__ CompF pair_mul(float x, float y, float more) {
    const float p = __fmul_rn(x, y);
    return CompF{p, __fadd_rn(fmaf(x, y, -p), more)};
}
// a / d rounded once, up to some 2^-40, with rc = 1 / d.s: a quotient from the
// reciprocal and one correction, or, where the reciprocal is near the ends of the
// range, from divisions (a quotient that overflows stays as it is)
__device__ __forceinline__ float pair_quot(CompF a, CompF d, float rc) {
    if (fabsf(rc) > 0x1p-120f && fabsf(rc) < 0x1p120f) {
        const float q = __fmul_rn(a.s, rc);
        return fmaf(__fadd_rn(fmaf(-q, d.s, a.s), fmaf(-q, d.e, a.e)), rc, q);
    }
    const float q = __fdiv_rn(a.s, d.s);
    const float r = __fadd_rn(fmaf(-q, d.s, a.s), fmaf(-q, d.e, a.e));
    const float c = __fadd_rn(q, __fdiv_rn(r, d.s));
    return c == c ? c : q;
}

// Inverse of the diagonal block m + diag(dg).  A relative error of the inverse
// acts in every sweep like one of the diagonal, which is large against M: on
// smooth fields it is amplified by the ratio of the two.  So the float inverse
// is formed from pairs and rounded once per entry; rounding its sums,
// determinant and products one by one raised the error of an FP32 apply by a
// tenth to a fifth over dividing in each sweep.
template <int NF>
__device__ __forceinline__ void write_block_inverse(const double* m, const FaceSum<double> (&dg)[NF], double* D,
                                                    long long nc, long long i) {
    if constexpr (NF == 1) {
        D[i] = 1.0 / (m[0] + dg[0].s);
    } else {
        const double a11 = m[0] + dg[0].s, a12 = m[1], a21 = m[2], a22 = m[3] + dg[1].s;
        const double id = 1.0 / (a11 * a22 - a12 * a21);
        D[i] = a22 * id;
        D[nc + i] = -a12 * id;
        D[2 * nc + i] = -a21 * id;
        D[3 * nc + i] = a11 * id;
    }
}
template <int NF>
__device__ __forceinline__ void write_block_inverse(const float* m, const FaceSum<float> (&dg)[NF], float* D,
                                                    long long nc, long long i) {
    const CompF a11 = pair_add(dg[0].s, m[0]);
    if constexpr (NF == 1) {
        D[i] = pair_quot(CompF{1.f, 0.f}, a11, __frcp_rn(a11.s));
    } else {
        const CompF a22 = pair_add(dg[1].s, m[3]);
        CompF det = pair_mul(a11.s, a22.s, fmaf(a11.s, a22.e, __fmul_rn(a11.e, a22.s)));
        const CompF off = pair_mul(m[1], m[2], 0.f);
        comp_add(det, -off.s);
        det.e = __fsub_rn(det.e, off.e);
        det = pair_norm(det);
        const float rc = __frcp_rn(det.s);
        D[i] = pair_quot(a22, det, rc);
        D[nc + i] = pair_quot(CompF{-m[1], 0.f}, det, rc);
        D[2 * nc + i] = pair_quot(CompF{-m[2], 0.f}, det, rc);
        D[3 * nc + i] = pair_quot(a11, det, rc);
    }
}

template <typename T, int NF, int ND>
__global__ void k_block_inverse(LvlDev L, const T* M, const T* K, T* D) {
    pdl_wait();
    int i[3];
    long long cc;
    if (!lvl_pos(L, i, cc)) return;
    T m[NF * NF];
    FaceSum<T> dg[NF];
#pragma unroll
    for (int q = 0; q < NF * NF; ++q) m[q] = M[q * L.nc + cc];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        if (L.n[d] == 1) continue;
        long long ju, jd;
        nb_index(L, d, i[0], i[1], i[2], ju, jd);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const T* Kd = K + (long long)(f * ND + d) * L.nc;
            dg[f].add(Kd[cc], Kd[ju]);
        }
    }
    write_block_inverse<NF>(m, dg, D, L.nc, cc);
}

template <typename T>
void launch_block_inverse(const Grid& G, int nf, MGLevel& L, cudaStream_t s) {
    const CellLaunch cl = cell_launch(L.n);
    MG_DISPATCH(k_block_inverse, cl.grid, cl.block, lvl(L), (const T*)L.M, (const T*)L.K, (T*)L.D);
}
template void launch_block_inverse<double>(const Grid&, int, MGLevel&, cudaStream_t);
template void launch_block_inverse<float>(const Grid&, int, MGLevel&, cudaStream_t);

// ---------------------------------------------------------------------------
// coarse coefficients
// ---------------------------------------------------------------------------

// Sum of values in the basis precision: in double for a double basis; for a
// float one as a compensated float pair, rounded once, which gives the digits
// of a double sum without the FP64 pipe (the conversions and sums of the
// two-field coarse coefficients took 0.75 ms at 256^3 on it).
template <typename T> struct MeanSum;
template <> struct MeanSum<double> {
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s = s + v; }
    __device__ __forceinline__ double get() const { return s; }
};
template <> struct MeanSum<float> {
    CompF a = {0.f, 0.f};
    __device__ __forceinline__ void add(float v) { comp_add(a, v); }
    __device__ __forceinline__ float get() const { return a.s + a.e; }
};

// sum of f over the 2^k fine cells from (x0,y0,z0) on (mx, my, mz: two cells
// along that direction)
template <typename T>
__device__ __forceinline__ T child_sum(const T* f, const LvlDev& F, bool mx, bool my, bool mz, int x0, int y0,
                                       int z0) {
    MeanSum<T> m;
#pragma unroll
    for (int kz = 0; kz < 2; ++kz) {
        if (kz && !mz) break;
#pragma unroll
        for (int ky = 0; ky < 2; ++ky) {
            if (ky && !my) break;
            m.add(f[lflat(F, x0, y0 + ky, z0 + kz)]);
            if (mx) m.add(f[lflat(F, x0 + 1, y0 + ky, z0 + kz)]);
        }
    }
    return m.get();
}

// One thread per coarse cell: M the mean of the children, K_d the mean of the
// fine faces that form the coarse face (those of the even children along d)
// over four, the cell width of a coarsened direction having doubled; a
// direction left with a single cell carries no flux.  D needs the face
// coefficients above the cell too, which the thread averages for itself.
template <typename T, int NF, int ND>
__global__ void k_coarsen(LvlDev F, LvlDev C, const T* Mf, const T* Kf, T* Mc,
                          T* Kc, T* Dc) {
    pdl_wait();
    int ic[3];
    long long cc;
    if (!lvl_pos(C, ic, cc)) return;
    const bool cd[3] = {F.n[0] != C.n[0], F.n[1] != C.n[1], F.n[2] != C.n[2]};
    int o[3];
    T w[3], wm = (T)1;      // weights of a sum over a coarsened direction
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        o[d] = cd[d] ? 2 * ic[d] : ic[d];
        w[d] = cd[d] ? (T)0.5 : (T)1;
        wm = wm * w[d];
    }
    T m[NF * NF];
    FaceSum<T> dg[NF];
#pragma unroll
    for (int q = 0; q < NF * NF; ++q) {
        m[q] = wm * child_sum<T>(Mf + q * F.nc, F, cd[0], cd[1], cd[2], o[0], o[1], o[2]);
        Mc[q * C.nc + cc] = m[q];
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) {
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const T* k = Kf + (long long)(f * ND + d) * F.nc;
            T v = (T)0;
            if (C.n[d] > 1) {
                // the mean over the other directions, and a quarter where the cell width along d doubled
                const T wk = wm * w[d];
                auto face = [&](const int (&p)[3]) -> T {
                    return wk * child_sum<T>(k, F, cd[0] && d != 0, cd[1] && d != 1, cd[2] && d != 2, p[0], p[1], p[2]);
                };
                v = face(o);
                int up[3] = {o[0], o[1], o[2]};
                up[d] = wrapi(o[d] + (cd[d] ? 2 : 1), F.n[d]);
                dg[f].add(v, face(up));
            }
            Kc[(long long)(f * ND + d) * C.nc + cc] = v;
        }
    }
    write_block_inverse<NF>(m, dg, Dc, C.nc, cc);
}

template <typename T>
void launch_coarsen(const Grid& G, int nf, const MGLevel& F, MGLevel& C, cudaStream_t s) {
    const CellLaunch cl = cell_launch(C.n);
    MG_DISPATCH(k_coarsen, cl.grid, cl.block, lvl(F), lvl(C), (const T*)F.M, (const T*)F.K, (T*)C.M, (T*)C.K,
                (T*)C.D);
}
template void launch_coarsen<double>(const Grid&, int, const MGLevel&, MGLevel&, cudaStream_t);
template void launch_coarsen<float>(const Grid&, int, const MGLevel&, MGLevel&, cudaStream_t);

// ---------------------------------------------------------------------------
// rows of one colour
// ---------------------------------------------------------------------------

// V consecutive elements, moved as one 8- or 16-byte access where V > 1
template <typename T, int V>
struct alignas(sizeof(T) * V) Pack {
    T v[V];
};
template <typename T, int V>
__device__ __forceinline__ Pack<T, V> load_pack(const T* p) {
    return *reinterpret_cast<const Pack<T, V>*>(p);
}
template <typename T, int V>
__device__ __forceinline__ void store_pack(T* p, const Pack<T, V>& a) {
    *reinterpret_cast<Pack<T, V>*>(p) = a;
}

// The cells t .. t+V-1 of one colour in row (b,c) of a colour-split level and
// their neighbours, which all have the other colour: across y and z they
// stand at the same t of the neighbouring rows; along x one of the two
// neighbours of cell t stands at t of the own row and the other at t+1 (odd
// first cell) or t-1 (even first cell), so a vector of them is the aligned
// vector shifted by one element from `edge`.
template <int ND>
struct Row {
    long long own, opp, edge;     // own cells; same t in the other colour; the element that completes the shifted vector
    long long yu, yd, zu, zd;
    bool odd;                     // the cells of the colour sit at odd x

    template <int V>
    __device__ __forceinline__ void set(const LvlDev& L, int colour, int t, int b, int c, std::integral_constant<int, V>) {
        const int nt = L.n[0] >> 1;
        const long long half = L.nc >> 1;
        const long long ob = colour ? 0 : half;
        const long long row = ((long long)c * L.n[1] + b) * nt;
        odd = (b + c + colour) & 1;
        own = (colour ? half : 0) + row + t;
        opp = ob + row + t;
        edge = ob + row + (odd ? (t + V == nt ? 0 : t + V) : (t == 0 ? nt - 1 : t - 1));
        yu = ob + ((long long)c * L.n[1] + wrap_up(b, L.n[1])) * nt + t;
        yd = ob + ((long long)c * L.n[1] + wrap_dn(b, L.n[1])) * nt + t;
        if (ND == 3) {
            zu = ob + ((long long)wrap_up(c, L.n[2]) * L.n[1] + b) * nt + t;
            zd = ob + ((long long)wrap_dn(c, L.n[2]) * L.n[1] + b) * nt + t;
        }
    }
};

// values of f at the upper and lower x neighbours
template <typename T, int V>
__device__ __forceinline__ void x_neighbours(const Pack<T, V>& a, T e, bool odd, Pack<T, V>& up, Pack<T, V>& dn) {
#pragma unroll
    for (int q = 0; q < V; ++q) {
        up.v[q] = odd ? (q + 1 < V ? a.v[q + 1 < V ? q + 1 : 0] : e) : a.v[q];
        dn.v[q] = odd ? a.v[q] : (q > 0 ? a.v[q > 0 ? q - 1 : 0] : e);
    }
}

// sum over the faces of K x_neighbour (FULL: of K (x_neighbour - x_own), xo
// the own values) for field f of the cells of a row
template <typename T, int ND, int V, bool FULL>
__device__ __forceinline__ Pack<T, V> face_sum(const LvlDev& L, const Row<ND>& r, const T* K, const T* x, int f,
                                               const Pack<T, V>& xo) {
    Pack<T, V> s;
#pragma unroll
    for (int q = 0; q < V; ++q) s.v[q] = (T)0;
    const T* xf = x + (long long)f * L.nc;
    auto add = [&](const Pack<T, V>& Ku, const Pack<T, V>& Kl, const Pack<T, V>& xu, const Pack<T, V>& xd) {
#pragma unroll
        for (int q = 0; q < V; ++q) {
            if (FULL) s.v[q] = s.v[q] + (Ku.v[q] * (xu.v[q] - xo.v[q]) - Kl.v[q] * (xo.v[q] - xd.v[q]));
            else s.v[q] = s.v[q] + (Ku.v[q] * xu.v[q] + Kl.v[q] * xd.v[q]);
        }
    };
    {
        const T* Kd = K + (long long)(f * ND) * L.nc;
        const Pack<T, V> ka = load_pack<T, V>(Kd + r.opp), xa = load_pack<T, V>(xf + r.opp);
        const T ke = Kd[r.edge], xe = xf[r.edge];
        Pack<T, V> Ku, Kx, xu, xd;
        x_neighbours<T, V>(ka, ke, r.odd, Ku, Kx);
        x_neighbours<T, V>(xa, xe, r.odd, xu, xd);
        add(Ku, load_pack<T, V>(Kd + r.own), xu, xd);
    }
    if (L.n[1] > 1) {
        const T* Kd = K + (long long)(f * ND + 1) * L.nc;
        add(load_pack<T, V>(Kd + r.yu), load_pack<T, V>(Kd + r.own), load_pack<T, V>(xf + r.yu),
            load_pack<T, V>(xf + r.yd));
    }
    if (ND == 3 && L.n[2] > 1) {
        const T* Kd = K + (long long)(f * ND + 2) * L.nc;
        add(load_pack<T, V>(Kd + r.zu), load_pack<T, V>(Kd + r.own), load_pack<T, V>(xf + r.zu),
            load_pack<T, V>(xf + r.zd));
    }
    return s;
}

// widest vector of the row kernels: 16 bytes per access in FP32, single FP64 cells
template <typename T> constexpr int kRowV = sizeof(T) == 4 ? 4 : 1;

// Vectors where the rows divide into them and the level is large enough that
// the wider loads matter (a smaller one lasts as long as one thread's loads,
// and single cells spread it over more threads).
template <typename T>
static bool row_vector(const MGLevel& L) {
    return kRowV<T> > 1 && (L.n[0] >> 1) % kRowV<T> == 0 && L.ncell >= kRowVCells;
}

// launch over the cells of one colour (or the coarse cells below them), nt
// threads along x
static inline CellLaunch row_launch(int nt, int ny, int nz) {
    int bx = 1;
    while (bx < nt && bx < 32) bx *= 2;
    const int by = 128 / bx;
    CellLaunch L;
    L.block = dim3(bx, by, 1);
    L.grid = dim3((nt + bx - 1) / bx, (ny + by - 1) / by, nz);
    return L;
}

// ---------------------------------------------------------------------------
// smoother
// ---------------------------------------------------------------------------

// Red-black Gauss-Seidel half sweep over the cells of one colour (parity of
// i+j+k), V cells along x per thread.  Bound by memory: per cell of the colour
// it reads rhs, D, K on both sides and the neighbours' x and writes x.  Two
// FP32 fields at 256^3: 105 us a half sweep, 44 algorithmic bytes per cell at 7.0
// TB/s (part of the neighbours' values comes from the L2), where
// single cells per thread (one 4-byte load per value) took 137 us.
template <typename T, int NF, int ND, int V>
__global__ void __launch_bounds__(128) k_smooth(LvlDev L, const T* K, const T* D, T* x,
                                                const T* rhs, int colour, int tr) {
    pdl_wait();
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    const int b = blockIdx.y * blockDim.y + threadIdx.y;
    const int c = blockIdx.z;
    if (t >= (L.n[0] >> 1) || b >= L.n[1]) return;
    Row<ND> r;
    r.set(L, colour, t, b, c, std::integral_constant<int, V>());
    Pack<T, V> w[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const Pack<T, V> g = load_pack<T, V>(rhs + (long long)f * L.nc + r.own);
        w[f] = face_sum<T, ND, V, false>(L, r, K, x, f, g);
#pragma unroll
        for (int q = 0; q < V; ++q) w[f].v[q] = g.v[q] + w[f].v[q];
    }
    if constexpr (NF == 1) {
        const Pack<T, V> d = load_pack<T, V>(D + r.own);
#pragma unroll
        for (int q = 0; q < V; ++q) w[0].v[q] = d.v[q] * w[0].v[q];
        store_pack<T, V>(x + r.own, w[0]);
    } else {
        const Pack<T, V> d0 = load_pack<T, V>(D + r.own), d1 = load_pack<T, V>(D + (tr ? 2 : 1) * L.nc + r.own);
        const Pack<T, V> d2 = load_pack<T, V>(D + (tr ? 1 : 2) * L.nc + r.own), d3 = load_pack<T, V>(D + 3 * L.nc + r.own);
        Pack<T, V> o0, o1;
#pragma unroll
        for (int q = 0; q < V; ++q) {
            o0.v[q] = d0.v[q] * w[0].v[q] + d1.v[q] * w[1].v[q];
            o1.v[q] = d2.v[q] * w[0].v[q] + d3.v[q] * w[1].v[q];
        }
        store_pack<T, V>(x + r.own, o0);
        store_pack<T, V>(x + L.nc + r.own, o1);
    }
}

// half sweep at one cell, for levels in natural order (a single cell along x)
template <typename T, int NF, int ND>
__device__ __forceinline__ void smooth_cell(const LvlDev& Lv, const T* K, const T* D, T* x, const T* rhs, int a, int b,
                                            int c, int tr) {
    const long long cc = lflat(Lv, a, b, c);
    T w[NF], o[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) w[f] = (T)0;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        if (Lv.n[d] == 1) continue;
        long long ju, jd;
        nb_index(Lv, d, a, b, c, ju, jd);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const T* Kd = K + (long long)(f * ND + d) * Lv.nc;
            const T* xf = x + (long long)f * Lv.nc;
            w[f] = w[f] + (Kd[ju] * xf[ju] + Kd[cc] * xf[jd]);
        }
    }
#pragma unroll
    for (int f = 0; f < NF; ++f) w[f] = rhs[(long long)f * Lv.nc + cc] + w[f];
    block_times<T, NF>(D, Lv.nc, cc, w, o, tr);
#pragma unroll
    for (int f = 0; f < NF; ++f) x[(long long)f * Lv.nc + cc] = o[f];
}

template <typename T, int NF, int ND>
__global__ void k_smooth_nat(LvlDev L, const T* K, const T* D, T* x,
                             const T* rhs, int colour, int tr) {
    pdl_wait();
    int i[3];
    long long cc;
    if (!lvl_pos(L, i, cc)) return;
    if (((i[0] + i[1] + i[2]) & 1) != colour) return;
    smooth_cell<T, NF, ND>(L, K, D, x, rhs, i[0], i[1], i[2], tr);
}

template <typename T>
void launch_smooth(const Grid& G, int nf, MGLevel& Lv, int colour, cudaStream_t s, int tr) {
    const LvlDev L = lvl(Lv);
    const T *K = (const T*)Lv.K, *D = (const T*)Lv.D, *rhs = (const T*)Lv.rhs;
    T* x = (T*)Lv.x;
    const int nt = Lv.n[0] >> 1;
    if (Lv.n[0] & 1) {
        const CellLaunch cl = cell_launch(Lv.n);
        MG_DISPATCH(k_smooth_nat, cl.grid, cl.block, L, K, D, x, rhs, colour, tr);
    } else if (row_vector<T>(Lv)) {
        const CellLaunch cl = row_launch(nt / kRowV<T>, Lv.n[1], Lv.n[2]);
        MG_DISPATCH_V(k_smooth, kRowV<T>, cl.grid, cl.block, L, K, D, x, rhs, colour, tr);
    } else {
        const CellLaunch cl = row_launch(nt, Lv.n[1], Lv.n[2]);
        MG_DISPATCH_V(k_smooth, 1, cl.grid, cl.block, L, K, D, x, rhs, colour, tr);
    }
}
template void launch_smooth<double>(const Grid&, int, MGLevel&, int, cudaStream_t, int);
template void launch_smooth<float>(const Grid&, int, MGLevel&, int, cudaStream_t, int);

// ---------------------------------------------------------------------------
// residual and restriction
// ---------------------------------------------------------------------------

// residual rhs - A x at fine cell (a,b,c), field f
template <typename T, int NF, int ND>
__device__ __forceinline__ T fine_residual(const LvlDev& F, const T* M, const T* K, const T* x, const T* rhs, int f,
                                           int a, int b, int c, int tr) {
    const long long cc = lflat(F, a, b, c);
    T out;
    if (NF == 1) out = M[cc] * x[cc];
    else if (!tr) out = M[(f * 2 + 0) * F.nc + cc] * x[cc] + M[(f * 2 + 1) * F.nc + cc] * x[F.nc + cc];
    else out = M[(0 * 2 + f) * F.nc + cc] * x[cc] + M[(1 * 2 + f) * F.nc + cc] * x[F.nc + cc];
    const T* xf = x + (long long)f * F.nc;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        if (F.n[d] == 1) continue;
        long long ju, jd;
        nb_index(F, d, a, b, c, ju, jd);
        const T* Kd = K + (long long)(f * ND + d) * F.nc;
        T Kl = Kd[cc], Ku = Kd[ju];
        out = out - (Ku * (xf[ju] - xf[cc]) - Kl * (xf[cc] - xf[jd]));
    }
    return rhs[(long long)f * F.nc + cc] - out;
}

// fine residual r = rhs - A x, one thread per fine cell
template <typename T, int NF, int ND>
__global__ void k_residual_mg(LvlDev F, const T* M, const T* K, const T* x,
                             const T* rhs, T* r, int tr) {
    pdl_wait();
    int i[3];
    long long cc;
    if (!lvl_pos(F, i, cc)) return;
#pragma unroll
    for (int f = 0; f < NF; ++f)
        r[(long long)f * F.nc + cc] = fine_residual<T, NF, ND>(F, M, K, x, rhs, f, i[0], i[1], i[2], tr);
}

// mean of value(x,y,z) over the children of coarse cell ic (pairs along x,
// then y, then z; with red_only the black children, whose residual is zero,
// are not evaluated)
template <typename T, class Fn>
__device__ __forceinline__ T children_mean(const LvlDev& F, const LvlDev& C, const int ic[3], bool red_only, Fn value) {
    const bool cx = F.n[0] != C.n[0], cy = F.n[1] != C.n[1], cz = F.n[2] != C.n[2];
    const int x0 = cx ? 2 * ic[0] : ic[0], y0 = cy ? 2 * ic[1] : ic[1], z0 = cz ? 2 * ic[2] : ic[2];
    auto child = [&](int xx, int yy, int zz) -> T {
        return (red_only && ((xx + yy + zz) & 1)) ? (T)0 : value(xx, yy, zz);
    };
    auto xm = [&](int yy, int zz) -> T {
        T a = child(x0, yy, zz);
        return cx ? (a + child(x0 + 1, yy, zz)) / (T)2 : a;
    };
    auto ym = [&](int zz) -> T {
        T a = xm(y0, zz);
        return cy ? (a + xm(y0 + 1, zz)) / (T)2 : a;
    };
    T a = ym(z0);
    return cz ? (a + ym(z0 + 1)) / (T)2 : a;
}

// coarse right-hand side from the stored fine residual; the coarse correction
// starts from zero (no pre-smoothing: every child counts)
template <typename T, int NF, int ND>
__global__ void k_restrict(LvlDev F, LvlDev C, const T* r, T* rhsc, T* xc) {
    pdl_wait();
    int ic[3];
    long long cc;
    if (!lvl_pos(C, ic, cc)) return;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const T* q = r + (long long)f * F.nc;
        rhsc[(long long)f * C.nc + cc] =
            children_mean<T>(F, C, ic, false, [&](int a, int b, int c) { return q[lflat(F, a, b, c)]; });
        xc[(long long)f * C.nc + cc] = (T)0;
    }
}

// writes the coarse right-hand side g at cell cc and, on a red cell, the red
// half sweep of the coarse level's zero start
template <typename T, int NF>
__device__ __forceinline__ void write_coarse(const LvlDev& C, const T* Dc, T* rhsc, T* xc, const T (&g)[NF],
                                             long long cc, bool red, int tr) {
#pragma unroll
    for (int f = 0; f < NF; ++f) rhsc[(long long)f * C.nc + cc] = g[f];
    if (red) {
        T o[NF];
        block_times<T, NF>(Dc, C.nc, cc, g, o, tr);
#pragma unroll
        for (int f = 0; f < NF; ++f) xc[(long long)f * C.nc + cc] = o[f];
    }
}

// Residual and restriction in one pass after a black half sweep (the black
// residual is zero), for levels in natural order
template <typename T, int NF, int ND>
__global__ void k_residual_restrict_nat(LvlDev F, LvlDev C, const T* M, const T* K,
                                        const T* x, const T* rhs, const T* Dc,
                                        T* rhsc, T* xc, int tr) {
    pdl_wait();
    int ic[3];
    long long cc;
    if (!lvl_pos(C, ic, cc)) return;
    T g[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f)
        g[f] = children_mean<T>(F, C, ic, true, [&](int a, int b, int c) {
            return fine_residual<T, NF, ND>(F, M, K, x, rhs, f, a, b, c, tr);
        });
    write_coarse<T, NF>(C, Dc, rhsc, xc, g, cc, ((ic[0] + ic[1] + ic[2]) & 1) == 0, tr);
}

// The same for colour-split levels.  The red children of coarse cell (a,b,c)
// stand at t = a of the fine rows (2b+dy, 2c+dz): each thread takes V cells of
// one of these rows, with the loads of the smoother, and the rows are added
// through shared memory: 118 us at 256^3 with two FP32 fields, 6.4 TB/s.  (All
// four rows in one thread needed 92 registers and took 194 us.)  The coarse
// level's first half sweep costs no launch of its own.
template <typename T, int NF, int ND, int V>
__global__ void __launch_bounds__(128) k_residual_restrict(LvlDev F, LvlDev C, const T* M,
                                                           const T* K, const T* x,
                                                           const T* rhs, const T* Dc,
                                                           T* rhsc, T* xc, int tr) {
    pdl_wait();
    constexpr int NR = ND == 3 ? 4 : 2;                 // fine rows of a coarse row
    __shared__ __align__(16) T sh[NF][128 * V];         // written as packs of up to 16 bytes
    const int row = threadIdx.y % NR, lb = threadIdx.y / NR;
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) * V;
    const int b = blockIdx.y * (blockDim.y / NR) + lb;
    const int c = blockIdx.z;
    const int ny = F.n[1] != C.n[1] ? 2 : 1, nz = F.n[2] != C.n[2] ? 2 : 1;
    const int dy = row & 1, dz = row >> 1;
    const bool in = t < (F.n[0] >> 1) && b < C.n[1];
    Pack<T, V> g[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f)
#pragma unroll
        for (int q = 0; q < V; ++q) g[f].v[q] = (T)0;
    if (in && dy < ny && dz < nz) {
        Row<ND> r;
        r.set(F, 0, t, ny * b + dy, nz * c + dz, std::integral_constant<int, V>());
        Pack<T, V> xo[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) xo[f] = load_pack<T, V>(x + (long long)f * F.nc + r.own);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            Pack<T, V> mx;
            const Pack<T, V> m0 = load_pack<T, V>(M + (NF == 1 ? 0 : (tr ? f : 2 * f)) * F.nc + r.own);
#pragma unroll
            for (int q = 0; q < V; ++q) mx.v[q] = m0.v[q] * xo[0].v[q];
            if constexpr (NF == 2) {
                const Pack<T, V> m1 = load_pack<T, V>(M + (tr ? 2 + f : 2 * f + 1) * F.nc + r.own);
#pragma unroll
                for (int q = 0; q < V; ++q) mx.v[q] = mx.v[q] + m1.v[q] * xo[1].v[q];
            }
            const Pack<T, V> fs = face_sum<T, ND, V, true>(F, r, K, x, f, xo[f]);
            const Pack<T, V> rh = load_pack<T, V>(rhs + (long long)f * F.nc + r.own);
#pragma unroll
            for (int q = 0; q < V; ++q) g[f].v[q] = rh.v[q] - (mx.v[q] - fs.v[q]);
        }
    }
    const int bx = blockDim.x, i0 = threadIdx.y * bx + threadIdx.x;
#pragma unroll
    for (int f = 0; f < NF; ++f) store_pack<T, V>(&sh[f][i0 * V], g[f]);
    __syncthreads();
    // The block's coarse cells, one per thread and step.  Pairs along x, then
    // y, then z, the black children counting as zero: the halvings are exact,
    // so the sum of the red residuals is scaled once.
    const T scale = (T)1 / (T)(2 * ny * nz);
    const int w = bx * V, total = w * (blockDim.y / NR);
    for (int i = i0; i < total; i += bx * blockDim.y) {
        const int l = i / w, k = i - l * w;
        const int a = blockIdx.x * w + k, bb = blockIdx.y * (blockDim.y / NR) + l;
        if (a >= (F.n[0] >> 1) || bb >= C.n[1]) continue;
        T gq[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const T* p = &sh[f][l * NR * w + k];
            T v = p[0] + p[w];
            if (NR == 4) v = v + (p[2 * w] + p[3 * w]);
            gq[f] = scale * v;
        }
        write_coarse<T, NF>(C, Dc, rhsc, xc, gq, lflat(C, a, bb, c), ((a + bb + c) & 1) == 0, tr);
    }
}

template <typename T>
void launch_restrict(const Grid& G, int nf, MGLevel& F, MGLevel& C, cudaStream_t s, int tr, int pre_smoothed) {
    const CellLaunch cl = cell_launch(C.n);
    const T *M = (const T*)F.M, *K = (const T*)F.K, *x = (const T*)F.x, *rhs = (const T*)F.rhs, *Dc = (const T*)C.D;
    if (!pre_smoothed) {
        const CellLaunch fl = cell_launch(F.n);
        MG_DISPATCH(k_residual_mg, fl.grid, fl.block, lvl(F), M, K, x, rhs, (T*)F.r, tr);
        MG_DISPATCH(k_restrict, cl.grid, cl.block, lvl(F), lvl(C), (const T*)F.r, (T*)C.rhs, (T*)C.x);
        return;
    }
    const int nt = F.n[0] >> 1, rows = G.ndim == 3 ? 4 : 2;
    // blocks of 128 threads: V cells each of the fine rows of a few coarse rows
    auto shape = [&](int v) {
        int bx = 1;
        while (bx < nt / v && bx < 32) bx *= 2;
        const int lb = 128 / (bx * rows);
        CellLaunch r;
        r.block = dim3(bx, rows * lb, 1);
        r.grid = dim3((nt / v + bx - 1) / bx, (C.n[1] + lb - 1) / lb, C.n[2]);
        return r;
    };
    if (F.n[0] & 1) {
        MG_DISPATCH(k_residual_restrict_nat, cl.grid, cl.block, lvl(F), lvl(C), M, K, x, rhs, Dc, (T*)C.rhs, (T*)C.x,
                    tr);
    } else if (row_vector<T>(F)) {
        const CellLaunch rl = shape(kRowV<T>);
        MG_DISPATCH_V(k_residual_restrict, kRowV<T>, rl.grid, rl.block, lvl(F), lvl(C), M, K, x, rhs, Dc, (T*)C.rhs,
                      (T*)C.x, tr);
    } else {
        const CellLaunch rl = shape(1);
        MG_DISPATCH_V(k_residual_restrict, 1, rl.grid, rl.block, lvl(F), lvl(C), M, K, x, rhs, Dc, (T*)C.rhs,
                      (T*)C.x, tr);
    }
}
template void launch_restrict<double>(const Grid&, int, MGLevel&, MGLevel&, cudaStream_t, int, int);
template void launch_restrict<float>(const Grid&, int, MGLevel&, MGLevel&, cudaStream_t, int, int);

// r = rhs - A x on every cell of level F (the inner-solve residual that the
// preconditioner's accuracy monitor and its tolerance-driven cycling read)
template <typename T>
void launch_mg_residual(const Grid& G, int nf, MGLevel& F, cudaStream_t s) {
    const CellLaunch fl = cell_launch(F.n);
    MG_DISPATCH(k_residual_mg, fl.grid, fl.block, lvl(F), (const T*)F.M, (const T*)F.K, (const T*)F.x,
                (const T*)F.rhs, (T*)F.r, 0);
}
template void launch_mg_residual<double>(const Grid&, int, MGLevel&, cudaStream_t);
template void launch_mg_residual<float>(const Grid&, int, MGLevel&, cudaStream_t);

// ---------------------------------------------------------------------------
// prolongation
// ---------------------------------------------------------------------------

// Cell-centred linear prolongation x_f += P x_c for one coarse cell: load
// the coarse neighbourhood once (3 values along each coarsened direction)
// and update the cell's 2^k children (red_only: the red ones).  A child at
// offset delta along a coarsened direction interpolates 3/4 of its parent and
// 1/4 of the parent's neighbour on its side (periodic wrap; at a wall the
// parent itself), along x, then y, then z.
template <typename T, int NF, int ND>
__device__ __forceinline__ void prolong_cell(int bc0, int bc1, int bc2, const LvlDev& F, const LvlDev& C,
                                             const T* xc, T* xf, const int ic[3], int red_only) {
    const bool cd[3] = {F.n[0] != C.n[0], F.n[1] != C.n[1], F.n[2] != C.n[2]};
    const int bc[3] = {bc0, bc1, bc2};
    // coarse indices at offsets -1, 0, +1 along each direction
    int nb[3][3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int i = ic[d], n = C.n[d];
        nb[d][1] = i;
        if (!cd[d]) {
            nb[d][0] = nb[d][2] = i;
        } else if (bc[d] == 0) {
            nb[d][0] = wrapi(i - 1, n);
            nb[d][2] = wrapi(i + 1, n);
        } else {
            nb[d][0] = i - 1 < 0 ? i : i - 1;
            nb[d][2] = i + 1 >= n ? i : i + 1;
        }
    }
    const T w0 = (T)0.75, w1 = (T)0.25;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        const T* q = xc + (long long)f * C.nc;
        T* out = xf + (long long)f * F.nc;
        T v[3][3][3];       // v[z][y][x], offsets -1..+1 (only 0 along a direction not coarsened)
#pragma unroll
        for (int kz = 0; kz < 3; ++kz)
#pragma unroll
            for (int ky = 0; ky < 3; ++ky)
#pragma unroll
                for (int kx = 0; kx < 3; ++kx)
                    v[kz][ky][kx] = q[lflat(C, nb[0][kx], nb[1][ky], nb[2][kz])];
#pragma unroll
        for (int dz = 0; dz < 2; ++dz) {
            if (dz && !cd[2]) continue;
#pragma unroll
            for (int dy = 0; dy < 2; ++dy) {
                if (dy && !cd[1]) continue;
#pragma unroll
                for (int dx = 0; dx < 2; ++dx) {
                    if (dx && !cd[0]) continue;
                    const int fx = cd[0] ? 2 * ic[0] + dx : ic[0];
                    const int fy = cd[1] ? 2 * ic[1] + dy : ic[1];
                    const int fz = cd[2] ? 2 * ic[2] + dz : ic[2];
                    if (red_only && ((fx + fy + fz) & 1)) continue;
                    // the other parent lies at offset -1 for child 0 and +1 for child 1
                    auto along_x = [&](int yy, int zz) -> T {
                        const T a = v[zz][yy][1], o = dx ? v[zz][yy][2] : v[zz][yy][0];
                        return cd[0] ? w0 * a + w1 * o : a;
                    };
                    auto along_y = [&](int zz) -> T {
                        const T a = along_x(1, zz), o = dy ? along_x(2, zz) : along_x(0, zz);
                        return cd[1] ? w0 * a + w1 * o : a;
                    };
                    const T a = along_y(1), o = dz ? along_y(2) : along_y(0);
                    const T val = cd[2] ? w0 * a + w1 * o : a;
                    const long long j = lflat(F, fx, fy, fz);
                    out[j] = out[j] + val;
                }
            }
        }
    }
}

// one thread per coarse cell and field (blockIdx.z runs over field, then
// coarse z): one field's 27 coarse values live at a time, which halves the
// registers of the two-field case (128 -> 64) and doubles its occupancy
template <typename T, int ND>
__global__ void k_prolong(int bc0, int bc1, int bc2, LvlDev F, LvlDev C, const T* xc,
                          T* xf, int red_only) {
    pdl_wait();
    const int f = blockIdx.z / C.n[2];
    int ic[3];
    ic[0] = blockIdx.x * blockDim.x + threadIdx.x;
    ic[1] = blockIdx.y * blockDim.y + threadIdx.y;
    ic[2] = blockIdx.z - f * C.n[2];
    if (ic[0] >= C.n[0] || ic[1] >= C.n[1]) return;
    prolong_cell<T, 1, ND>(bc0, bc1, bc2, F, C, xc + (long long)f * C.nc, xf + (long long)f * F.nc, ic, red_only);
}

template <typename T>
void launch_prolong(const Grid& G, int nf, MGLevel& F, MGLevel& C, cudaStream_t s, int red_only) {
    CellLaunch cl = cell_launch(C.n);
    cl.grid.z = (unsigned)(C.n[2] * nf);
    ++g_launch_count;
    if (G.ndim == 3)
        launch_k(k_prolong<T, 3>, cl.grid, cl.block, 0, s, G.bc[0], G.bc[1], G.bc[2], lvl(F), lvl(C), (const T*)C.x,
                 (T*)F.x, red_only);
    else
        launch_k(k_prolong<T, 2>, cl.grid, cl.block, 0, s, G.bc[0], G.bc[1], G.bc[2], lvl(F), lvl(C), (const T*)C.x,
                 (T*)F.x, red_only);
}
template void launch_prolong<double>(const Grid&, int, MGLevel&, MGLevel&, cudaStream_t, int);
template void launch_prolong<float>(const Grid&, int, MGLevel&, MGLevel&, cudaStream_t, int);

// ---------------------------------------------------------------------------
// both sides of a 2D level in one launch each
// ---------------------------------------------------------------------------

// On a 2D level of some ten thousand cells a half sweep lasts little longer than
// its launch, and a V(2,2) cycle has nine of them.  Here a block takes a tile of
// kTileX x kTileY cells and a halo into shared memory and runs all half sweeps of
// its side of the cycle there, each on a region one cell smaller than the one
// before, so the tile itself needs nothing from other blocks: pre-smoothing with
// the residual and restriction, and prolongation with post-smoothing.  A 32 x 16
// tile with a halo of four works on 1.9 times its cells, and reads the
// coefficients once instead of in every half sweep.  Blocks read their halo from
// x while others finish, so the first kernel writes to the scratch r and the
// second back to x.  One field in either precision and two in FP32 (tiled_level),
// so the transposed system needs no case of its own: one field's is the same.
constexpr int kTileX = 32, kTileY = 16, kTileThreads = 256, kTileHalo = 5;

template <typename T, int NF>
struct Tile2D {
    const LvlDev& L;
    T* sm;
    int H, PX, PY, N;        // halo, extents with it, cells
    int ox, oy;              // global position of the tile's first cell
    int par;                 // parity of the tile-local origin (halo corner)

    __device__ __forceinline__ Tile2D(const LvlDev& l, T* s, int h) : L(l), sm(s), H(h) {
        PX = kTileX + 2 * H;
        PY = kTileY + 2 * H;
        N = PX * PY;
        ox = blockIdx.x * kTileX;
        oy = blockIdx.y * kTileY;
        par = (ox + oy) & 1;                       // the corner is at (ox - H, oy - H)
    }
    __device__ __forceinline__ T* x(int f) const { return sm + f * N; }
    __device__ __forceinline__ T* b(int f) const { return sm + (NF + f) * N; }
    __device__ __forceinline__ T* K(int q) const { return sm + (2 * NF + q) * N; }          // f * 2 + d
    __device__ __forceinline__ T* D(int q) const { return sm + (4 * NF + q) * N; }
    __device__ __forceinline__ static int fields() { return 4 * NF + NF * NF; }
    // storage index of the cell at tile position (i, j), wrapped
    __device__ __forceinline__ long long at(int i, int j) const {
        const int a = (ox + i - H) & (L.n[0] - 1), c = (oy + j - H) & (L.n[1] - 1);
        return rb_index(L.n[0], L.n[1], L.nc, a, c, 0);
    }
    __device__ __forceinline__ void load(const T* xg, const T* bg, const T* Kg, const T* Dg) const {
        for (int t = threadIdx.x; t < N; t += kTileThreads) {
            const int j = t / PX, i = t - j * PX;
            const long long g = at(i, j);
            T v[4 * NF + NF * NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                v[f] = xg[f * L.nc + g];
                v[NF + f] = bg[f * L.nc + g];
            }
#pragma unroll
            for (int q = 0; q < 2 * NF; ++q) v[2 * NF + q] = Kg[q * L.nc + g];
#pragma unroll
            for (int q = 0; q < NF * NF; ++q) v[4 * NF + q] = Dg[q * L.nc + g];
#pragma unroll
            for (int q = 0; q < 4 * NF + NF * NF; ++q) sm[q * N + t] = v[q];
        }
    }
    // visits the cells of one colour of the tile grown by m cells
    template <class Fn>
    __device__ __forceinline__ void visit(int colour, int m, Fn fn) const {
        const int w = (kTileX + 2 * m) / 2, rows = kTileY + 2 * m, lo = H - m;
        for (int t = threadIdx.x; t < w * rows; t += kTileThreads) {
            const int r = t / w, j = lo + r;
            const int i0 = lo + 2 * (t - r * w);
            fn(i0 + ((i0 + j + par + colour) & 1), j);
        }
    }
    __device__ __forceinline__ void sweep(int colour, int m) const {
        visit(colour, m, [&](int i, int j) {
            const int p = j * PX + i;
            T w[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const T* xf = x(f);
                T s = K(2 * f)[p + 1] * xf[p + 1] + K(2 * f)[p] * xf[p - 1];
                s = s + (K(2 * f + 1)[p + PX] * xf[p + PX] + K(2 * f + 1)[p] * xf[p - PX]);
                w[f] = b(f)[p] + s;
            }
            if constexpr (NF == 1) {
                x(0)[p] = D(0)[p] * w[0];
            } else {
                x(0)[p] = D(0)[p] * w[0] + D(1)[p] * w[1];
                x(1)[p] = D(2)[p] * w[0] + D(3)[p] * w[1];
            }
        });
        __syncthreads();
    }
    __device__ __forceinline__ void store(T* xg) const {
        for (int t = threadIdx.x; t < kTileX * kTileY; t += kTileThreads) {
            const int j = H + t / kTileX, i = H + t % kTileX;
            const long long g = at(i, j);
#pragma unroll
            for (int f = 0; f < NF; ++f) xg[f * L.nc + g] = x(f)[j * PX + i];
        }
    }
};

// half sweeps h0 .. 2 nu1 - 1 (even: red), then the residual of the red cells and
// the restriction as in k_residual_restrict; x_out gets the smoothed tile
template <typename T, int NF>
__global__ void __launch_bounds__(kTileThreads) k_pre2d(LvlDev F, LvlDev C, const T* M, const T* K, const T* D,
                                                        const T* xin, const T* rhs, const T* Dc, T* xout, T* rhsc,
                                                        T* xc, int h0, int nu1) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char raw[];
    const Tile2D<T, NF> t(F, reinterpret_cast<T*>(raw), 2 * nu1 - h0 + 1);
    t.load(xin, rhs, K, D);
    __syncthreads();
    for (int h = h0; h < 2 * nu1; ++h) t.sweep(h & 1, 2 * nu1 - h);
    // one thread per coarse cell: its red children are (2a, 2b) and (2a+1, 2b+1)
    for (int q = threadIdx.x; q < kTileX * kTileY / 4; q += kTileThreads) {
        const int ia = q % (kTileX / 2), ib = q / (kTileX / 2);
        T g[NF];
#pragma unroll
        for (int f = 0; f < NF; ++f) g[f] = (T)0;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int i = t.H + 2 * ia + k, j = t.H + 2 * ib + k, p = j * t.PX + i;
            const long long gi = t.at(i, j);
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const T* xf = t.x(f);
                const T* K0 = t.K(2 * f);
                const T* K1 = t.K(2 * f + 1);
                T s = K0[p + 1] * (xf[p + 1] - xf[p]) - K0[p] * (xf[p] - xf[p - 1]);
                s = s + (K1[p + t.PX] * (xf[p + t.PX] - xf[p]) - K1[p] * (xf[p] - xf[p - t.PX]));
                T mx = M[NF * f * F.nc + gi] * t.x(0)[p];
                if constexpr (NF == 2) mx = mx + M[(2 * f + 1) * F.nc + gi] * t.x(1)[p];
                g[f] = g[f] + (t.b(f)[p] - (mx - s));
            }
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) g[f] = (T)0.25 * g[f];
        const int a = blockIdx.x * (kTileX / 2) + ia, b = blockIdx.y * (kTileY / 2) + ib;
        write_coarse<T, NF>(C, Dc, rhsc, xc, g, lflat(C, a, b, 0), ((a + b) & 1) == 0, 0);
    }
    t.store(xout);
}

// prolongation to the red cells, then 2 nu2 half sweeps, black first
template <typename T, int NF>
__global__ void __launch_bounds__(kTileThreads) k_post2d(int bc0, int bc1, LvlDev F, LvlDev C, const T* K,
                                                         const T* D, const T* xin, const T* rhs, const T* xc, T* xout,
                                                         int nu2) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char raw[];
    const Tile2D<T, NF> t(F, reinterpret_cast<T*>(raw), 2 * nu2);
    t.load(xin, rhs, K, D);
    __syncthreads();
    t.visit(0, t.H, [&](int i, int j) {
        const int a = (t.ox + i - t.H) & (F.n[0] - 1), b = (t.oy + j - t.H) & (F.n[1] - 1);
        const int a0 = a >> 1, b0 = b >> 1;
        auto side = [](int k, int odd, int n, int bc) {
            const int m = k + (odd ? 1 : -1);
            return bc == 0 ? m & (n - 1) : (m < 0 || m >= n ? k : m);
        };
        const int a1 = side(a0, a & 1, C.n[0], bc0), b1 = side(b0, b & 1, C.n[1], bc1);
        const T w0 = (T)0.75, w1 = (T)0.25;
        const long long j00 = lflat(C, a0, b0, 0), j10 = lflat(C, a1, b0, 0), j01 = lflat(C, a0, b1, 0),
                        j11 = lflat(C, a1, b1, 0);
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const T* q = xc + f * C.nc;
            const T y0 = w0 * q[j00] + w1 * q[j10], y1 = w0 * q[j01] + w1 * q[j11];
            T* x = t.x(f) + j * t.PX + i;
            *x = *x + (w0 * y0 + w1 * y1);
        }
    });
    __syncthreads();
    for (int h = 0; h < 2 * nu2; ++h) t.sweep(1 - (h & 1), 2 * nu2 - 1 - h);
    t.store(xout);
}

template <typename T>
static size_t tile_bytes(int nf, int halo) {
    return (size_t)(4 * nf + nf * nf) * (kTileX + 2 * halo) * (kTileY + 2 * halo) * sizeof(T);
}
// the kernels take more shared memory than the default limit, set once per kernel and device
template <auto FN>
static void allow_smem(size_t bytes) {
    static thread_local int done = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (done == dev) return;
    cudaFuncSetAttribute(FN, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    done = dev;
}

// Levels for the two kernels: 2D, coarsened in both directions, whole tiles, one
// or two sweeps on either side, and up to 262,144 FP32 cells or 131,072 FP64 cells
// of one field.  The halo's part of the half sweeps grows with the level and the
// launches that the tiles save do not.  V(1,1) / V(2,2) cycles with tiles
// against separate kernels on the finest level, in us:
//   FP32, one field   512 x 256   35 / 46 and 38 / 53    512^2        41 / 55 and 43 / 60
//         two fields  512^2       57 / 75 and 54 / 77    1024 x 512   79 / 102 and 69 / 92
//   FP64, one field   256^2       49 / 72 and 51 / 77    512 x 256    60 / 89 and 60 / 91
//         two fields  128^2       60 / 90 and 57 / 87    512 x 256   105 / 160 and 96 / 152
template <typename T>
bool tiled_level(const Grid& G, int nf, const MGLevel& F, const MGLevel& C, int nu1, int nu2) {
    const long long most = sizeof(T) == 4 ? 1 << 18 : (nf == 1 ? 1 << 17 : 0);
    return G.ndim == 2 && F.n[0] % kTileX == 0 && F.n[1] % kTileY == 0 && C.n[0] * 2 == F.n[0] &&
           C.n[1] * 2 == F.n[1] && nu1 >= 1 && nu1 <= 2 && nu2 >= 1 && nu2 <= 2 &&
           F.ncell <= most;
}
template bool tiled_level<double>(const Grid&, int, const MGLevel&, const MGLevel&, int, int);
template bool tiled_level<float>(const Grid&, int, const MGLevel&, const MGLevel&, int, int);

template <typename T, int NF>
static void pre2d(const MGLevel& F, MGLevel& C, int nu1, int started, cudaStream_t s) {
    allow_smem<k_pre2d<T, NF>>(tile_bytes<T>(NF, kTileHalo));
    ++g_launch_count;
    launch_k(k_pre2d<T, NF>, dim3(F.n[0] / kTileX, F.n[1] / kTileY), kTileThreads,
             tile_bytes<T>(NF, 2 * nu1 - started + 1), s, lvl(F), lvl(C), (const T*)F.M, (const T*)F.K, (const T*)F.D,
             (const T*)F.x, (const T*)F.rhs, (const T*)C.D, (T*)F.r, (T*)C.rhs, (T*)C.x, started, nu1);
}
template <typename T>
void launch_pre2d(int nf, MGLevel& F, MGLevel& C, int nu1, int started, cudaStream_t s) {
    if (nf == 1) pre2d<T, 1>(F, C, nu1, started, s);
    else if constexpr (sizeof(T) == 4) pre2d<T, 2>(F, C, nu1, started, s);
}
template void launch_pre2d<double>(int, MGLevel&, MGLevel&, int, int, cudaStream_t);
template void launch_pre2d<float>(int, MGLevel&, MGLevel&, int, int, cudaStream_t);

template <typename T, int NF>
static void post2d(const Grid& G, const MGLevel& F, const MGLevel& C, int nu2, cudaStream_t s) {
    allow_smem<k_post2d<T, NF>>(tile_bytes<T>(NF, kTileHalo));
    ++g_launch_count;
    launch_k(k_post2d<T, NF>, dim3(F.n[0] / kTileX, F.n[1] / kTileY), kTileThreads, tile_bytes<T>(NF, 2 * nu2), s,
             G.bc[0], G.bc[1], lvl(F), lvl(C), (const T*)F.K, (const T*)F.D, (const T*)F.r, (const T*)F.rhs,
             (const T*)C.x, (T*)F.x, nu2);
}
template <typename T>
void launch_post2d(const Grid& G, int nf, MGLevel& F, MGLevel& C, int nu2, cudaStream_t s) {
    if (nf == 1) post2d<T, 1>(G, F, C, nu2, s);
    else if constexpr (sizeof(T) == 4) post2d<T, 2>(G, F, C, nu2, s);
}
template void launch_post2d<double>(const Grid&, int, MGLevel&, MGLevel&, int, cudaStream_t);
template void launch_post2d<float>(const Grid&, int, MGLevel&, MGLevel&, int, cudaStream_t);

// ---------------------------------------------------------------------------
// coarsest level
// ---------------------------------------------------------------------------

// the single cell's system: D is the inverse of M there (no faces)
template <typename T, int NF>
__device__ __forceinline__ void coarsest_cell(const T* D, const T* rhs, T* x, int tr) {
    T g[NF], o[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) g[f] = rhs[f];
    block_times<T, NF>(D, 1, 0, g, o, tr);
#pragma unroll
    for (int f = 0; f < NF; ++f) x[f] = o[f];
}

template <typename T>
__global__ void k_coarsest(int nf, const T* D, const T* rhs, T* x, int tr) {
    pdl_wait();
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    if (nf == 1) coarsest_cell<T, 1>(D, rhs, x, tr);
    else coarsest_cell<T, 2>(D, rhs, x, tr);
}

template <typename T>
void launch_coarsest(int nf, MGLevel& C, cudaStream_t s, int tr) {
    ++g_launch_count;
    launch_k(k_coarsest<T>, 1, 32, 0, s, nf, (const T*)C.D, (const T*)C.rhs, (T*)C.x, tr);
}
template void launch_coarsest<double>(int, MGLevel&, cudaStream_t, int);
template void launch_coarsest<float>(int, MGLevel&, cudaStream_t, int);

}  // namespace jfnk
