// Shared device-side definitions of the JFNK library: grid descriptor,
// neighbour indexing with periodic / reflecting-wall ghosts, the van Leer
// slope, and deterministic block reductions.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>
#include <utility>

#include "emu64.cuh"

namespace jfnk {

constexpr int kBlock = 256;          // threads per block of the pointwise kernels
constexpr int kRedBlocks = 1024;     // fixed block count of grid-stride reductions
constexpr int kMaxRedBlocks = 2048;  // cap of the occupancy-sized reduction grids

struct Grid {
    int ndim;
    int n[3];
    long long ncell;
    double dx[3], idx[3], idx2[3], tidx[3];   // tidx = 2 / dx
    double hidx[3];                           // 0.5 / dx
    int bc[3];                       // 0 periodic, 1 wall
    double gamma, gm1;
    double g[3];
    double hg[3];                    // g / 2 (the face density enters as the cell sum)
    double K0, chi_exp;
    int energy_form;                 // 0 internal e, 1 total eps_t
    double theta;
    // integer copies of the tests on the parameters above, so kernels branch
    // on them without FP64 compares: bit d of gmask = (g[d] != 0),
    // has_cond = (K0 != 0), chi3 = (chi_exp == 3)
    int gmask, has_cond, chi3;
    double igm1, igamma;             // 1/(gamma-1) = c_v and 1/gamma, formed on the host
    double ggm1;                     // gamma (gamma-1): c_s^2 = ggm1 e
};

inline void set_grid_flags(Grid& G) {
    G.gmask = 0;
    for (int d = 0; d < 3; ++d)
        if (G.g[d] != 0.0) G.gmask |= 1 << d;
    G.has_cond = G.K0 != 0.0;
    G.chi3 = G.chi_exp == 3.0;
    G.igm1 = 1.0 / G.gm1;
    G.igamma = 1.0 / G.gamma;
    G.ggm1 = G.gamma * G.gm1;
    for (int d = 0; d < 3; ++d) G.hg[d] = 0.5 * G.g[d];
}

// Programmatic dependent launch.  Every kernel of the library starts with
// pdl_wait and is launched by launch_k: its blocks may be placed as soon as the
// blocks of the kernel before it in the stream have exited, and wait there, before
// they touch memory, until that kernel has completed and its writes are visible.
// As each kernel waits first, completion is transitive and the stream's order is
// kept whatever kernel comes before or after; what overlaps is the end of one
// kernel with the launch of the next, some microseconds between kernels that
// last no longer on the small grids.
//
// No kernel lets its dependent in earlier (griddepcontrol.launch_dependents).
// With the trigger at their start, kernels that were queued without a host read
// in between piled up on the SMs, several of them waiting: the blocks of each
// later one went to whichever SMs were left, unevenly, and the residual took 74 us
// instead of 30 at 64 x 512 cells, 140 instead of 60 at 4096 x 4 x 4 (45 and 82
// with ordinary launches of the kernels before them).  With it after the wait:
// 37 and 88 us.  A 256^2 FP64 apply takes 209 us, 253 with the early trigger; the
// adjoint at 128^2 4.03 and 4.47 ms, the 256^2 mixed step 9.1 and 10.6 ms.
//
// The data that a kernel reads may thus be written during its lifetime, up to the
// wait.  Loads through the read-only path (__ldg, and what the compiler may
// make of const __restrict__ kernel parameters) are defined only for data that
// stay as they are for the whole kernel, and no-alias parameters let the
// compiler move their accesses across the wait.  So kernel parameters carry no
// __restrict__ and every load is an ordinary one; functions that run after the
// wait may take __restrict__ parameters, whose promise begins with the call.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
inline void launch_k(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

struct Idx3 { int i[3]; };

// Launch shape of the cell kernels: x along threadIdx.x (coalesced), y and
// z from the grid, so no thread decomposes a flat index by division.
struct CellLaunch {
    dim3 grid, block;
};

inline CellLaunch cell_launch(const int n[3]) {
    int bx = 32;
    while (bx < n[0] && bx < 128) bx *= 2;
    int by = 128 / bx;
    CellLaunch L;
    L.block = dim3(bx, by, 1);
    L.grid = dim3((n[0] + bx - 1) / bx, (n[1] + by - 1) / by, n[2]);
    return L;
}

// Position of this thread in a cell_launch grid; false outside the grid.
__device__ __forceinline__ bool cell_pos(const int n[3], Idx3& P, long long& c) {
    P.i[0] = blockIdx.x * blockDim.x + threadIdx.x;
    P.i[1] = blockIdx.y * blockDim.y + threadIdx.y;
    P.i[2] = blockIdx.z;
    if (P.i[0] >= n[0] || P.i[1] >= n[1]) return false;
    c = ((long long)P.i[2] * n[1] + P.i[1]) * n[0] + P.i[0];
    return true;
}

// Position of this thread in tile `tile` of a cell_launch tiling (tiles in
// x, then y, then z order), for grid-stride kernels that visit several tiles
// per block; false outside the grid.
__device__ __forceinline__ bool cell_pos_tile(const int n[3], int tile, Idx3& P, long long& c) {
    const int gx = (n[0] + (int)blockDim.x - 1) / (int)blockDim.x;
    const int gy = (n[1] + (int)blockDim.y - 1) / (int)blockDim.y;
    const int r = tile / gx;
    P.i[0] = (tile - r * gx) * blockDim.x + threadIdx.x;
    P.i[1] = (r % gy) * blockDim.y + threadIdx.y;
    P.i[2] = r / gy;
    if (P.i[0] >= n[0] || P.i[1] >= n[1]) return false;
    c = ((long long)P.i[2] * n[1] + P.i[1]) * n[0] + P.i[0];
    return true;
}

__device__ __forceinline__ int block_linear() {
    return blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
}

__device__ __forceinline__ int thread_linear() { return threadIdx.x + blockDim.x * threadIdx.y; }

__device__ __forceinline__ Idx3 decompose(const Grid& G, long long c) {
    Idx3 r;
    r.i[0] = (int)(c % G.n[0]);
    long long t = c / G.n[0];
    r.i[1] = (int)(t % G.n[1]);
    r.i[2] = (int)(t / G.n[1]);
    return r;
}

__device__ __forceinline__ long long flat(const Grid& G, int i0, int i1, int i2) {
    return ((long long)i2 * G.n[1] + i1) * G.n[0] + i0;
}

// Storage index of cell (a,b,c) in a multigrid array.  With an even x extent
// the arrays are colour-split: all cells with i+j+k even first, then the odd
// ones, each in x-fastest order (the two cells of an x pair share flat/2), so
// a red-black half sweep reads and writes contiguous memory.  Levels with an
// odd x extent (a single cell along x) keep the natural order.
__device__ __forceinline__ long long rb_index(int n0, int n1, long long nc, int a, int b, int c) {
    long long f = ((long long)c * n1 + b) * n0 + a;
    if (n0 & 1) return f;
    return (long long)((a + b + c) & 1) * (nc >> 1) + (f >> 1);
}

// Cell-quantity index of position k along a direction of size n: periodic
// wrap, or mirror about the wall faces (k -> -k-1, k -> 2n-1-k).  Stencil
// offsets never exceed the grid size (n >= 4, |offset| <= 3), so one
// conditional wrap replaces an integer modulo.
__device__ __forceinline__ int cell_map(int k, int n, int bc) {
    if (bc == 0) return k < 0 ? k + n : (k >= n ? k - n : k);
    if (k < 0) return -k - 1;
    if (k >= n) return 2 * n - 1 - k;
    return k;
}

// Load of a cell quantity at (pos + off) with ghost mapping in every direction.
__device__ __forceinline__ double load_cell(const Grid& G, const double* __restrict__ f, const Idx3& p,
                                            int o0, int o1, int o2) {
    int a = cell_map(p.i[0] + o0, G.n[0], G.bc[0]);
    int b = cell_map(p.i[1] + o1, G.n[1], G.bc[1]);
    int c = cell_map(p.i[2] + o2, G.n[2], G.bc[2]);
    return f[flat(G, a, b, c)];
}

// Load of the velocity normal to the faces of direction `c` at slot
// (pos + off): odd mirror about the wall faces, zero on both wall faces;
// cell mapping in the other directions.
__device__ __forceinline__ double load_normal(const Grid& G, const double* __restrict__ u, int c, const Idx3& p,
                                              int o0, int o1, int o2) {
    int k[3] = {p.i[0] + o0, p.i[1] + o1, p.i[2] + o2};
    long long flip = 0;                 // sign-bit mask of the odd mirror
    for (int d = 0; d < 3; ++d) {
        if (d == c && G.bc[d] == 1) {
            int n = G.n[d];
            int kk = k[d];
            if (kk == 0 || kk == n) return 0.0;
            if (kk < 0) { kk = -kk; flip = (long long)0x8000000000000000ULL; }
            else if (kk > n) { kk = 2 * n - kk; flip = (long long)0x8000000000000000ULL; }
            k[d] = kk;
        } else {
            k[d] = cell_map(k[d], G.n[d], G.bc[d]);
        }
    }
    double v = u[flat(G, k[0], k[1], k[2])];
    // sign flip on the sign bit (integer pipe) instead of an FP64 multiply
    return __longlong_as_double(__double_as_longlong(v) ^ flip);
}

// ---------------------------------------------------------------------------
// Branch-free neighbour addressing of the residual kernels.  Offsets are flat
// offsets relative to the thread's own cell (pointers given at that cell):
// k * stride inside the grid; the periodic wrap or the wall mirror changes
// them only where P + k e_d leaves the grid.  The boundary type is a kernel
// parameter (uniform across the warp) and the position tests are selects,
// so no thread-dependent branch splits a warp.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int grid_stride(const Grid& G, int d) {
    return d == 0 ? 1 : (d == 1 ? G.n[0] : G.n[0] * G.n[1]);
}

// offset of the cell quantity at P + k e_d, 1 <= |k| <= 3 (k = 0: 0)
__device__ __forceinline__ int cell_off(const Grid& G, const Idx3& P, int d, int k) {
    const int i = P.i[d], n = G.n[d];
    int m = k;
    if (k < 0) {
        // i + k < 0: periodic i + k + n, wall mirror -(i + k) - 1
        const int w = G.bc[d] == 0 ? k + n : -2 * i - k - 1;
        m = i + k < 0 ? w : k;
    } else if (k > 0) {
        // i + k >= n: periodic i + k - n, wall mirror 2n - 1 - (i + k)
        const int w = G.bc[d] == 0 ? k - n : 2 * n - 1 - 2 * i - k;
        m = i + k >= n ? w : k;
    }
    return m * grid_stride(G, d);
}

// velocity normal to direction c at face slot P + k e_c (uc at the thread's
// own slot): with walls the odd mirror (sign flip on the integer pipe) and
// zero on both wall faces; periodic faces wrap like cells
__device__ __forceinline__ double normal_along(const Grid& G, const double* __restrict__ uc, const Idx3& P, int c,
                                               int k) {
    if (G.bc[c] == 0) return uc[cell_off(G, P, c, k)];
    const int i = P.i[c], n = G.n[c], kk = i + k;
    int m = k;
    bool flip = false, zero = false;
    if (k <= 0) zero = kk == 0;
    if (k >= 0) zero = zero | (kk == n);
    if (k < 0) {
        flip = kk < 0;
        m = flip ? -2 * i - k : k;                  // slot -kk
    } else if (k > 0) {
        flip = kk > n;
        m = flip ? 2 * n - 2 * i - k : k;           // slot 2n - kk
    }
    const double v = uc[(zero ? 0 : m) * grid_stride(G, c)];   // the own slot where the value is zero
    const long long f = flip ? (long long)0x8000000000000000ULL : 0ll;
    return zero ? 0.0 : __longlong_as_double(__double_as_longlong(v) ^ f);
}

// velocity normal to direction c at slot P + k e_d, d != c (tangential
// offsets map like cells); zero when the thread's own slot is a wall face
// of c
__device__ __forceinline__ double normal_across(const Grid& G, const double* __restrict__ uc, const Idx3& P, int c,
                                                int d, int k) {
    const bool wall = (G.bc[c] == 1) & (P.i[c] == 0);
    const double v = uc[cell_off(G, P, d, k)];
    return wall ? 0.0 : v;
}

// face quantity of direction d at the upper face of the cell (slot P + e_d):
// zero at an upper wall
__device__ __forceinline__ double face_up_at(const Grid& G, const double* __restrict__ f, const Idx3& P, int d) {
    const bool top = (G.bc[d] == 1) & (P.i[d] + 1 == G.n[d]);
    const double v = f[top ? 0 : cell_off(G, P, d, 1)];
    return top ? 0.0 : v;
}

// True when slot p is the wall face of direction c.
__device__ __forceinline__ bool is_wall_slot(const Grid& G, int c, const Idx3& p) {
    return G.bc[c] == 1 && p.i[c] == 0;
}

// The two ways in which the residual kernels read their neighbours.  NbGen
// takes any position.  NbIn takes threads whose y and z positions are at least
// two cells from the ends, on grids that are periodic in x: every offset is a
// multiple of a stride or one of four wrapped x offsets, and no wall is near.
// Wrap and mirror selects were more than half of the flux kernels'
// instructions; a block has one row (or a few), so the choice is made per
// block (inner_block) and nearly every block of a large grid takes NbIn.
struct NbGen {
    const Grid& G;
    const Idx3& P;
    __device__ __forceinline__ NbGen(const Grid& g, const Idx3& p) : G(g), P(p) {}
    __device__ __forceinline__ int off(int d, int k) const { return cell_off(G, P, d, k); }
    __device__ __forceinline__ double along(const double* __restrict__ uc, int c, int k) const {
        return normal_along(G, uc, P, c, k);
    }
    __device__ __forceinline__ double across(const double* __restrict__ uc, int c, int d, int k) const {
        return normal_across(G, uc, P, c, d, k);
    }
    __device__ __forceinline__ double up(const double* __restrict__ f, int d) const { return face_up_at(G, f, P, d); }
    __device__ __forceinline__ bool wall(int c) const { return is_wall_slot(G, c, P); }
    // the slot that along / across read: offset, odd mirror, and false for a wall
    // face (a constant zero)
    __device__ __forceinline__ bool slot_along(int c, int k, int& o, bool& flip) const {
        flip = false;
        o = cell_off(G, P, c, k);
        if (G.bc[c] == 0) return true;
        const int i = P.i[c], n = G.n[c], kk = i + k;
        flip = kk < 0 || kk > n;
        const int m = kk < 0 ? -2 * i - k : (kk > n ? 2 * n - 2 * i - k : k);
        const bool zero = kk == 0 || kk == n;
        o = (zero ? 0 : m) * grid_stride(G, c);
        return !zero;
    }
    __device__ __forceinline__ bool slot_across(int c, int d, int k, int& o, bool& flip) const {
        flip = false;
        o = cell_off(G, P, d, k);
        return !is_wall_slot(G, c, P);
    }
    __device__ __forceinline__ bool has_low(int d) const { return !is_wall_slot(G, d, P); }
    // whether the face above the cell along d exists (upper walls have no slot)
    __device__ __forceinline__ bool has_up(int d) const { return !(G.bc[d] == 1 && P.i[d] + 1 == G.n[d]); }
};

struct NbIn {
    int xm2, xm1, xp1, xp2, s1, s2;
    __device__ __forceinline__ NbIn(const Grid& G, const Idx3& P) {
        const int i = P.i[0], n = G.n[0];
        xm1 = i < 1 ? n - 1 : -1;
        xm2 = i < 2 ? n - 2 : -2;
        xp1 = i + 1 >= n ? 1 - n : 1;
        xp2 = i + 2 >= n ? 2 - n : 2;
        s1 = n;
        s2 = n * G.n[1];
    }
    // |k| <= 2
    __device__ __forceinline__ int off(int d, int k) const {
        const int x = k == 0 ? 0 : (k == 1 ? xp1 : (k == 2 ? xp2 : (k == -1 ? xm1 : xm2)));
        return d == 0 ? x : k * (d == 1 ? s1 : s2);
    }
    __device__ __forceinline__ double along(const double* __restrict__ uc, int c, int k) const {
        return uc[off(c, k)];
    }
    __device__ __forceinline__ double across(const double* __restrict__ uc, int, int d, int k) const {
        return uc[off(d, k)];
    }
    __device__ __forceinline__ double up(const double* __restrict__ f, int d) const { return f[off(d, 1)]; }
    __device__ __forceinline__ bool wall(int) const { return false; }
    __device__ __forceinline__ bool slot_along(int c, int k, int& o, bool& flip) const {
        o = off(c, k);
        flip = false;
        return true;
    }
    __device__ __forceinline__ bool slot_across(int, int d, int k, int& o, bool& flip) const {
        o = off(d, k);
        flip = false;
        return true;
    }
    __device__ __forceinline__ bool has_low(int) const { return true; }
    __device__ __forceinline__ bool has_up(int) const { return true; }
};

// whether every thread of this block of a cell_launch grid may use NbIn
template <int ND>
__device__ __forceinline__ bool inner_block(const Grid& G) {
    const int y0 = blockIdx.y * blockDim.y, y1 = y0 + blockDim.y - 1, z = blockIdx.z;
    bool in = G.bc[0] == 0 && y0 >= 2 && y1 + 2 < G.n[1];
    if (ND == 3) in = in && z >= 2 && z + 2 < G.n[2];
    return in;
}

// van Leer (1974) harmonic slope: 2ab/(a+b) if ab > 0 else 0.
__device__ __forceinline__ double vanleer(double a, double b) {
    double ab = a * b;
    return ab > 0.0 ? (2.0 * ab) / (a + b) : 0.0;
}

// Sign tests on the bit pattern (integer pipe; the flux kernels are bound by
// the FP64 pipe).  For every non-NaN x: nonneg(x) == (x >= 0.0) (both zeros
// count), positive(x) == (x > 0.0).
// Both on the two 32-bit words: as 64-bit tests of the whole pattern the
// compiler turned nonneg into an FP64 compare (DSETP) on the FP64 pipe.
__device__ __forceinline__ bool nonneg(double x) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    return (hi >= 0) | ((((unsigned)hi << 1) | lo) == 0u);
}
__device__ __forceinline__ bool is_zero(double x) {
    return (((unsigned)__double2hiint(x) << 1) | (unsigned)__double2loint(x)) == 0u;
}
__device__ __forceinline__ bool positive(double x) {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    return (hi > 0) | ((hi == 0) & (lo != 0u));
}

// The arithmetic of one thread's evaluation, on the FP64 pipe (FpOps:
// plain operators, which the compiler may fuse into FMAs) or on the integer
// pipes (IntOps: the reduced-range functions of emu64.cuh; products, differences
// (isub), halves and maxima are correctly rounded, reciprocals within 1/2 + 2^-4
// units in the last place, limited slopes and roots within 1/2 + 2^-3).
// The FP64 pipe of sm_103a issues one warp instruction per 64 cycles per
// scheduler, so the FP64-bound kernels move part of their arithmetic to the
// idle integer pipes; what a kernel writes with plain operators stays on the
// FP64 pipe.  IntOps collects one validity flag for the whole sequence (operands
// zero or of moderate exponent) instead of branching per operation, so a kernel
// checks it once and redoes the thread's work with FpOps where it failed; no
// branch splits the integer sequence, and the compiler can interleave its
// independent chains.
struct FpOps {
    __device__ __forceinline__ double mul(double a, double b) { return a * b; }
    __device__ __forceinline__ double root(double a) { return sqrt(a); }
    __device__ __forceinline__ double half(double a) { return 0.5 * a; }
    __device__ __forceinline__ double larger(double a, double b) { return fmax(a, b); }
    __device__ __forceinline__ double isub(double a, double b) { return a - b; }
    __device__ __forceinline__ bool valid() const { return true; }
    static constexpr bool checked = false;
};

struct IntOps {
    bool ok = true;
    __device__ __forceinline__ double mul(double a, double b) { return emu::mul_mid(a, b, ok); }
    __device__ __forceinline__ double recip(double d) { return emu::recip_mid(d, ok); }
    __device__ __forceinline__ double harm(double a, double b) { return emu::harm_mid(a, b, ok); }
    __device__ __forceinline__ double root(double a) { return emu::sqrt_mid(a, ok); }
    __device__ __forceinline__ double half(double a) { return emu::half_mid(a, ok); }
    __device__ __forceinline__ double larger(double a, double b) { return emu::max_nonneg(a, b); }   // a >= 0
    __device__ __forceinline__ double isub(double a, double b) { return emu::add_mid(a, emu::neg(b), ok); }
    __device__ __forceinline__ bool valid() const { return ok; }
    static constexpr bool checked = true;
};

// Float <-> double conversions on the integer pipe.  On sm_103a the
// conversion instructions run on the FP64 pipe (2 per cycle per SM), and a
// predicated-off instruction still occupies it, so these handle every
// input in integer arithmetic, with no FP64 instruction on any path, and
// give the bits of the conversion instructions (IEEE 754: the float->double
// conversion is exact, double->float rounds to nearest, ties to even; NaNs
// stay NaNs).

// (double)f
__device__ __forceinline__ double f2d_exact(float f) {
    const unsigned u = __float_as_uint(f);
    const unsigned sign = u & 0x80000000u, mag = u & 0x7fffffffu, m = u & 0x7fffffu;
    const unsigned e = mag >> 23;
    unsigned hi, lo;
    if (e - 1u < 254u) {                              // normal: rebias by 1023 - 127 = 896
        hi = sign | ((mag >> 3) + 0x38000000u);
        lo = u << 29;
    } else if (e == 255u) {                           // infinity or NaN (quiet)
        hi = sign | 0x7ff00000u | (m >> 3) | (m ? 0x00080000u : 0u);
        lo = m << 29;
    } else if (m == 0u) {                             // zero
        hi = sign;
        lo = 0u;
    } else {                                          // subnormal float: a normal double
        const int k = 31 - __clz(m);                  // leading bit of m (value m 2^-149)
        const unsigned long long t = ((unsigned long long)m << (52 - k)) & 0xfffffffffffffULL;
        hi = sign | ((unsigned)(k + 874) << 20) | (unsigned)(t >> 32);
        lo = (unsigned)t;
    }
    return __hiloint2double((int)hi, (int)lo);
}

// (float)x, rounded to nearest, ties to even
__device__ __forceinline__ float d2f_rn(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned sign = hi & 0x80000000u, e = (hi >> 20) & 0x7ffu;
    unsigned b;
    if (e - 897u <= 1150u - 897u) {                   // normal float result: keep 23 bits, round on 29
        const unsigned m23 = ((hi & 0xfffffu) << 3) | (lo >> 29);
        const unsigned rem = lo & 0x1fffffffu;
        b = (((e - 896u) << 23) | m23) + ((rem > 0x10000000u || (rem == 0x10000000u && (m23 & 1u))) ? 1u : 0u);
    } else if (e == 0x7ffu) {                         // infinity or NaN (quiet)
        const bool nan = (hi & 0xfffffu) | lo;
        b = 0x7f800000u | (nan ? 0x00400000u | ((hi & 0xfffffu) << 3) | (lo >> 29) : 0u);
    } else if (e > 1150u) {                           // beyond the float range: infinity
        b = 0x7f800000u;
    } else if (e >= 873u) {                           // subnormal float (or the smallest normal)
        const unsigned long long m53 = (1ULL << 52) | ((unsigned long long)(hi & 0xfffffu) << 32) | lo;
        const unsigned s = 926u - e;                  // 30 .. 53
        const unsigned long long v = m53 >> s, r = m53 & ((1ULL << s) - 1ULL), half = 1ULL << (s - 1u);
        b = (unsigned)v + ((r > half || (r == half && (v & 1ULL))) ? 1u : 0u);
    } else {                                          // below half the smallest subnormal: zero
        b = 0u;
    }
    return __uint_as_float(sign | b);
}

// between the basis precision and double
__device__ __forceinline__ double to_f64(double x) { return x; }
__device__ __forceinline__ double to_f64(float x) { return f2d_exact(x); }
template <typename T> __device__ __forceinline__ T from_f64(double x);
template <> __device__ __forceinline__ double from_f64<double>(double x) { return x; }
template <> __device__ __forceinline__ float from_f64<float>(double x) { return d2f_rn(x); }

// 1/d from the hardware approximation r0 (rcp.approx.ftz.f64, MUFU pipe)
// refined by one third-order step of the reciprocal iteration: with
// e = 1 - d r0 the exact reciprocal is r0 (1 + e + e^2 + e^3 / (1 - e)), so
// r = r0 + r0 (e + e^2) leaves a relative error of about e^3 (the series
// form of Newton-Raphson refinement, P. Markstein, IBM J. Res. Dev. 34
// (1990) 111-119, taken one term further).  Three fused multiply-adds
// instead of the four of two quadratic steps; the result is within one ulp
// of the correctly rounded 1/d (the error before the last rounding is far
// below half an ulp).  Valid for normal d whose reciprocal is normal (the
// approximation flushes subnormals); callers guarantee the range.
__device__ __forceinline__ double recip_nr(double d) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    const double e = fma(-d, r, 1.0);
    return fma(fma(e, e, e), r, r);
}

// r[i] = 1/d[i], i < K, with one reciprocal: Montgomery's simultaneous
// inversion (P. L. Montgomery, Math. Comp. 48 (1987) 243-264):
// prefix products p_i = d_0 ... d_i, one reciprocal 1/p_{K-1} (recip_nr),
// then going down r_i = p_{i-1} / p_i and 1/p_{i-1} = d_i / p_i.  It costs
// 3(K-1) multiplications instead of K-1 divisions; each result carries at
// most 3K + 1 roundings instead of one.  The prefix products stay in the
// normal range when every |d_i| lies in [2^-R, 2^R), R = 1000/K (exponent
// test on the high word, integer pipe); otherwise the thread divides K
// times.  For the FP64 pipe: with IntOps a reciprocal is one of its own
// (emu::recip_mid, about 30 integer instructions, fewer than the three products
// of about 36 that the batched inversion spends per element).
template <int K>
__device__ __forceinline__ void recip_all(const double (&d)[K], double (&r)[K]) {
    constexpr unsigned R = 1000u / K;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const unsigned e = ((unsigned)__double2hiint(d[i]) >> 20) & 0x7ffu;
        ok = ok & (e - (1023u - R) < 2u * R);
    }
    if (ok) {
        double p[K];
        p[0] = d[0];
#pragma unroll
        for (int i = 1; i < K; ++i) p[i] = p[i - 1] * d[i];
        double inv = recip_nr(p[K - 1]);
#pragma unroll
        for (int i = K - 1; i > 0; --i) {
            r[i] = inv * p[i - 1];
            inv = inv * d[i];
        }
        r[0] = inv;
    } else {
#pragma unroll
        for (int i = 0; i < K; ++i) r[i] = 1.0 / d[i];
    }
}

// Upwind reconstruction without divergent branches.  With q_near the cell
// on the upwind side of the face, q_far its other neighbour and q_other the
// cell across the face, the face value is
//     q_near + s/2,   s = vanleer(q_near - q_far, q_other - q_near).
// For the right-hand (negative speed) case this is q_R - s_R/2 exactly,
// because the two differences change sign, which is exact, and s/2 =
// ab/(a+b) exactly (scaling by two commutes with rounding).
struct Stencil { double near, far, other; };

// K face values.  With checked Ops each half slope ab/(a+b) is formed on the
// integer pipes with one rounding (emu::harm_mid, about 75 integer
// instructions), and the FP64 pipe keeps three operations per value: a, b and
// the addition to q_near.  (With the product ab and the reciprocal on the
// integer pipes and a + b and q + (ab) inv on the FP64 pipe it kept four and a
// third of a batched reciprocal.)  Otherwise the quotient is split as num/den
// (num = ab, den = a + b where the limiter is on, 0 and 1 where it is off),
// so that every thread divides and all reciprocals of the batch are formed
// together.
template <int K, class O>
__device__ __forceinline__ void upwind_values(const Stencil (&q)[K], double (&v)[K], O&& ops) {
    if constexpr (std::remove_reference_t<O>::checked) {
#pragma unroll
        for (int i = 0; i < K; ++i) v[i] = q[i].near + ops.harm(q[i].near - q[i].far, q[i].other - q[i].near);
    } else {
        double num[K], den[K], inv[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const double a = q[i].near - q[i].far, b = q[i].other - q[i].near, ab = a * b;
            const bool on = positive(ab);
            num[i] = on ? ab : 0.0;
            den[i] = on ? a + b : 1.0;
        }
        recip_all<K>(den, inv);
#pragma unroll
        for (int i = 0; i < K; ++i) v[i] = fma(num[i], inv[i], q[i].near);
    }
}

// Error-free transformations (Knuth's TwoSum, FMA-based TwoProduct) used by
// the float basis and the float preconditioner output: a dot product
// accumulated as an unevaluated pair (sum, err) is as accurate as one
// accumulated in twice the working precision (Ogita, Rump & Oishi,
// "Accurate sum and dot product", 2005), without touching the FP64 pipe
// inside the loop.
struct CompF {
    float s, e;
};

// (explicitly rounded intrinsics: the compiler must not contract these into FMAs)
__device__ __forceinline__ void comp_add(CompF& a, float p) {
    float t = __fadd_rn(a.s, p);
    float bp = __fsub_rn(t, a.s);
    a.e = __fadd_rn(a.e, __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(p, bp)));
    a.s = t;
}

__device__ __forceinline__ void comp_fma(CompF& a, float x, float y) {
    float p = __fmul_rn(x, y);
    float err = fmaf(x, y, -p);
    comp_add(a, p);
    a.e = __fadd_rn(a.e, err);
}

// Squares of float values of magnitude m stay normal floats when m lies in
// [2^-60, 2^60): a thread whose largest |x| lies outside that range redoes
// its sum of squares in double (a second loop, taken by no thread in
// practice); otherwise the compensated float sum is exact to about 2^-44 of
// the result.  The check runs once per thread, after the loop, so the loop
// itself has no FP64 instruction.
__device__ __forceinline__ bool sq_range_unsafe(float maxabs) {
    return maxabs >= 0x1p60f || (maxabs > 0.f && maxabs < 0x1p-60f);
}

template <typename T> struct Acc { typedef double type; };

// Block-wide sum of one double per thread; result valid in thread 0.
template <int BS>
__device__ __forceinline__ double block_sum(double v, double* sh) {
    const int t = threadIdx.x + blockDim.x * threadIdx.y;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    int lane = t & 31, w = t >> 5;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    v = (t < BS / 32) ? sh[t] : 0.0;
    if (w == 0) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;
}

template <int BS>
__device__ __forceinline__ double block_max(double v, double* sh) {
    const int t = threadIdx.x + blockDim.x * threadIdx.y;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    int lane = t & 31, w = t >> 5;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    v = (t < BS / 32) ? sh[t] : 0.0;
    if (w == 0) {
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    }
    __syncthreads();
    return v;
}

// Sums of NV values over the lanes of a warp, value i into lane i (and, for NV
// below 32, into every lane that is i modulo the next power of two).  Halving
// exchange: in each step a lane keeps half of its values and adds the
// partner's copies of them, P - 1 additions for P values instead of five per
// value.
template <int NV>
__device__ __forceinline__ double warp_sums(double (&v)[NV]) {
    constexpr int P = NV > 16 ? 32 : (NV > 8 ? 16 : (NV > 4 ? 8 : (NV > 2 ? 4 : (NV > 1 ? 2 : 1))));
    const int lane = (threadIdx.x + blockDim.x * threadIdx.y) & 31;
    double a[P];
#pragma unroll
    for (int i = 0; i < P; ++i) a[i] = i < NV ? v[i < NV ? i : 0] : 0.0;
#pragma unroll
    for (int w = P / 2; w >= 1; w /= 2) {
        const bool up = lane & w;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const double send = up ? a[i] : a[i + w], keep = up ? a[i + w] : a[i];
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
        }
    }
#pragma unroll
    for (int w = P; w < 32; w *= 2) a[0] += __shfl_xor_sync(0xffffffffu, a[0], w);
    return a[0];
}

// Partial sums of a block to out[0 .. NV-1] (BS threads; sh: BS/32 * NV doubles)
template <int BS, int NV>
__device__ __forceinline__ void block_sums(double (&v)[NV], double* sh, double* out) {
    const int t = threadIdx.x + blockDim.x * threadIdx.y, lane = t & 31, w = t >> 5;
    const double r = warp_sums<NV>(v);
    if (lane < NV) sh[w * NV + lane] = r;
    __syncthreads();
    if (t < NV) {
        double a = 0.0;
#pragma unroll
        for (int i = 0; i < BS / 32; ++i) a += sh[i * NV + t];
        out[t] = a;
    }
}

// True in every thread of the last block of the grid to arrive (of nblocks),
// after all blocks' earlier global writes became visible to it; the counter is
// left at zero for the next launch on the stream.
__device__ __forceinline__ bool last_block(unsigned* counter, unsigned nblocks) {
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        last = atomicAdd(counter, 1u) == nblocks - 1;
        if (last) *counter = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last;
}

template <typename T> __device__ __forceinline__ double to_d(T v) { return (double)v; }

}  // namespace jfnk
