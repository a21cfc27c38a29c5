// The coarse end of a V-cycle, or whole V-cycles on a small grid, in one thread
// block cluster.
//
// Below some ten thousand cells a level's kernels last as long as their
// launches, and a V-cycle has about ten of them per level.  Here the phases
// of all levels from some level down run in one kernel: x, the right-hand
// side, the residual and the coefficients live in the shared memory of the
// cluster's blocks, the neighbours' values of another block come through
// distributed shared memory, and a cluster barrier ends a phase.  Levels too
// small to share (level_shared) run on the cluster's first block alone, with
// block barriers, while the others wait.
//
// What bounds it is the length of a phase: a barrier, one round of
// shared-memory loads and a handful of multiply-adds, with few warps to hide
// anything.  So a half sweep takes its addresses from a table built once per
// launch and its coefficients from one record per cell (K below and above the
// cell per direction, D, M), padded so that 16-byte loads of a warp meet no
// bank twice; positions are taken apart only in the two transfer phases.
//
// Measured: a phase on the first block takes about 450 cycles in FP32 and 800
// in FP64, one with a cluster barrier 1,600 (with positions recomputed in
// every phase, coefficients in global memory and one code copy per phase it
// was 1,600 and 3,300).  Two V(2,2) cycles of the 64^2 FP64 sound system take
// 84 us, where the single-block kernel that this one replaces (data in global
// memory, one SM's two FP64 lanes) and the finest level's launches took
// 280 us; with conduction at 128^2 in FP64 about 150 us instead of 1,050.
//
// Every extent is a power of two, so positions are taken apart with shifts.  A
// level of 2^lc cells is dealt out in chunks of 2^lch consecutive cells in
// natural order; within a chunk the red cells come first: index
// colour 2^(lch-1) + (f / 2 mod 2^(lch-1)) of the cell at flat index f (the
// two cells f, f+1 of an even f are neighbours along the first direction with
// more than one cell, so one is red and one black).
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace jfnk {

constexpr int kClThreads = 512;
constexpr int kClMaxLevels = 16;
constexpr int kClSmemMax = 227 * 1024;

struct ClLevel {
    int n[3];
    int lx, ly, lc, lch;      // log2 of the x and y extents, of the cells and of a block's chunk
    int shared;               // dealt out over the cluster (else on its first block)
    int ox, ob, oc, on;       // byte offsets in shared memory: x, rhs, coefficient records, neighbour table
    const void *M, *K, *D;
};
struct ClArgs {
    ClLevel lv[kClMaxLevels];
    int nlev, nshared;        // levels; the first nshared of them are dealt out
    int orr;                  // byte offset of the residual scratch
    int bc[3];
    int nu1, nu2, cycles, started, tr;
    const void* rhs;          // of the first level
    void* x;
};

// Elements of a coefficient record: K (lower, upper) per direction and field,
// D, M, and padding to 4 mod 8 words, or 2 mod 4 where 8-byte loads do
template <typename T, int NF, int ND>
struct Rec {
    static constexpr int kD = NF * 2 * ND, kM = kD + NF * NF, kUsed = kM + NF * NF;
    static constexpr int words(int e) { return e * (int)sizeof(T) / 4; }
    static constexpr int pad(int e) { return words(e) % 8 == 4 || (NF == 1 && words(e) % 4 == 2) ? e : pad(e + 1); }
    static constexpr int kSize = pad(kUsed);
};

static int ilog2(long long v) {
    int l = 0;
    while ((1ll << l) < v) ++l;
    return l;
}

// Levels dealt out over the cluster: where a phase on the first block alone
// would last longer than one with a cluster barrier and remote loads (FP64), or
// where its shared memory would keep a larger level out of the cluster (two
// FP32 fields of 1,024 cells take 120 KB on one block).
static bool level_shared(long long ncell, int elt, int ctas) { return ctas > 1 && ncell > (elt == 8 ? 256 : 512); }

// Shared memory plan of levels[0 .. nlev-1]; bytes needed per block
template <typename T, int NF, int ND>
static size_t cluster_plan_t(const MGLevel* levels, int nlev, int ctas, ClArgs& A) {
    long long off = 0, res = 0;
    auto take = [&](long long bytes) {
        const long long o = off;
        off += (bytes + 15) / 16 * 16;
        return (int)o;
    };
    A.nlev = nlev;
    A.nshared = 0;
    for (int l = 0; l < nlev; ++l) {
        ClLevel& v = A.lv[l];
        for (int d = 0; d < 3; ++d) v.n[d] = levels[l].n[d];
        v.lx = ilog2(v.n[0]);
        v.ly = ilog2(v.n[1]);
        v.lc = ilog2(levels[l].ncell);
        v.shared = level_shared(levels[l].ncell, sizeof(T), ctas) ? 1 : 0;
        v.lch = v.shared ? v.lc - ilog2(ctas) : v.lc;
        if (v.shared) ++A.nshared;
        const long long ch = 1ll << v.lch;
        v.ox = take(NF * ch * sizeof(T));
        v.ob = take(NF * ch * sizeof(T));
        v.oc = take(Rec<T, NF, ND>::kSize * ch * sizeof(T));
        v.on = take(2 * ND * ch * 4);
        res = std::max(res, (long long)NF * ch);
        v.M = levels[l].M;
        v.K = levels[l].K;
        v.D = levels[l].D;
    }
    A.orr = take(res * sizeof(T));
    return (size_t)off;
}

template <typename T>
static size_t cluster_plan(const MGLevel* levels, int nlev, int nf, int nd, int ctas, ClArgs& A) {
    if (nf == 1)
        return nd == 3 ? cluster_plan_t<T, 1, 3>(levels, nlev, ctas, A) : cluster_plan_t<T, 1, 2>(levels, nlev, ctas, A);
    return nd == 3 ? cluster_plan_t<T, 2, 3>(levels, nlev, ctas, A) : cluster_plan_t<T, 2, 2>(levels, nlev, ctas, A);
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// address of another block's shared memory (32-bit shared window)
__device__ __forceinline__ unsigned map_rank(unsigned a, int rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// loads at an address of the cluster's (REMOTE) or of the own block's shared window
__device__ __forceinline__ float ld_remote(unsigned a, float) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ double ld_remote(unsigned a, double) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
template <bool REMOTE, typename T>
__device__ __forceinline__ T ld_sh(unsigned a, T t) {
    if constexpr (REMOTE) return ld_remote(a, t);
    else return *(const T*)__cvta_shared_to_generic(a);
}

template <typename T, int NF, int ND>
struct Cluster {
    using R = Rec<T, NF, ND>;
    const ClArgs& A;
    unsigned char* sm;
    unsigned sbase;           // the same as an address of the shared window
    int rank;

    __device__ __forceinline__ T* xp(const ClLevel& v, int i) const { return (T*)(sm + v.ox) + i * NF; }
    __device__ __forceinline__ T* bp(const ClLevel& v, int i) const { return (T*)(sm + v.ob) + i * NF; }
    __device__ __forceinline__ T* cp(const ClLevel& v, int i) const { return (T*)(sm + v.oc) + i * R::kSize; }
    __device__ __forceinline__ T* rp(int i) const { return (T*)(sm + A.orr) + i * NF; }

    struct Pos { int a, b, c; };
    __device__ __forceinline__ static Pos pos(const ClLevel& v, int f) {
        return Pos{f & (v.n[0] - 1), (f >> v.lx) & (v.n[1] - 1), f >> (v.lx + v.ly)};
    }
    __device__ __forceinline__ static int flat_of(const ClLevel& v, int a, int b, int c) {
        return (((c << v.ly) + b) << v.lx) + a;
    }
    // flat index of the cell with chunk index i of this block
    __device__ __forceinline__ int flat_at(const ClLevel& v, int i) const {
        if (v.lch == 0) return rank << v.lch;
        const int h = v.lch - 1, col = i >> h;
        const int f0 = 2 * ((rank << h) + (i & ((1 << h) - 1)));
        const Pos p = pos(v, f0);
        return f0 + (((p.a + p.b + p.c) & 1) != col);
    }
    __device__ __forceinline__ static int local_of(const ClLevel& v, int f, int par) {
        return v.lch == 0 ? 0 : (par << (v.lch - 1)) + ((f & ((1 << v.lch) - 1)) >> 1);
    }
    // index in the level's global arrays
    __device__ __forceinline__ static int gidx(const ClLevel& v, int f, int par) {
        return v.lx > 0 ? (par << (v.lc - 1)) + (f >> 1) : f;
    }
    // shared-window address of element i of a chunk array (byte offset o) that block `owner` holds
    __device__ __forceinline__ unsigned addr(int o, int i, int owner) const {
        const unsigned a = sbase + o + i * (NF * (int)sizeof(T));
        return owner == rank ? a : map_rank(a, owner);
    }

    // Records, neighbour table, and (top) x and rhs of the chunk of level v.  Of a
    // started level the red cells alone hold values: the black ones start at
    // zero here, as the first sweep adds zero times a cell that is its own
    // neighbour (a direction with a single cell).
    __device__ __forceinline__ void setup(const ClLevel& v, int i, bool top) const {
        const T *K = (const T*)v.K, *D = (const T*)v.D, *M = (const T*)v.M;
        const size_t nc = (size_t)1 << v.lc;
        const int f = flat_at(v, i);
        const Pos p = pos(v, f);
        const int par = (p.a + p.b + p.c) & 1, g = gidx(v, f, par);
        T* rec = cp(v, i);
        unsigned* nb = (unsigned*)(sm + v.on) + i * (2 * ND);
        T k[NF * 2 * ND], dm[2 * NF * NF];
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const int m = v.n[d] - 1;
            const int q = d == 0 ? p.a : (d == 1 ? p.b : p.c);
            const int up = (q + 1) & m, dn = (q - 1) & m;
            const int fu = flat_of(v, d == 0 ? up : p.a, d == 1 ? up : p.b, d == 2 ? up : p.c);
            const int fd = flat_of(v, d == 0 ? dn : p.a, d == 1 ? dn : p.b, d == 2 ? dn : p.c);
            // a direction with a single cell carries no flux: zero coefficients and the own cell
            const int np = m == 0 ? par : 1 - par;
            nb[2 * d] = addr(v.ox, local_of(v, fd, np), fd >> v.lch);
            nb[2 * d + 1] = addr(v.ox, local_of(v, fu, np), fu >> v.lch);
#pragma unroll
            for (int q2 = 0; q2 < NF; ++q2) {
                const T* Kd = K + (q2 * ND + d) * nc;
                k[(q2 * ND + d) * 2] = m == 0 ? (T)0 : Kd[g];
                k[(q2 * ND + d) * 2 + 1] = m == 0 ? (T)0 : Kd[gidx(v, fu, np)];
            }
        }
#pragma unroll
        for (int q = 0; q < NF * NF; ++q) {
            const int qt = (NF == 2 && A.tr && (q == 1 || q == 2)) ? 3 - q : q;
            dm[q] = D[qt * nc + g];
            dm[NF * NF + q] = M[qt * nc + g];
        }
        T xb[2 * NF];
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            xb[q] = top && !(A.started && par) ? ((const T*)A.x)[q * nc + g] : (T)0;
            xb[NF + q] = top ? ((const T*)A.rhs)[q * nc + g] : (T)0;
        }
#pragma unroll
        for (int q = 0; q < NF * 2 * ND; ++q) rec[q] = k[q];
#pragma unroll
        for (int q = 0; q < 2 * NF * NF; ++q) rec[R::kD + q] = dm[q];
#pragma unroll
        for (int q = 0; q < NF; ++q) {
            xp(v, i)[q] = xb[q];
            bp(v, i)[q] = xb[NF + q];
        }
    }

    __device__ __forceinline__ void block_times(const T* rec, const T (&w)[NF], T (&out)[NF]) const {
        if constexpr (NF == 1) {
            out[0] = rec[R::kD] * w[0];
        } else {
            out[0] = rec[R::kD] * w[0] + rec[R::kD + 1] * w[1];
            out[1] = rec[R::kD + 2] * w[0] + rec[R::kD + 3] * w[1];
        }
    }

    // half sweep of one colour
    template <bool SH>
    __device__ __forceinline__ void sweep(const ClLevel& v, int col) const {
        const int half = 1 << (v.lch - 1);
        for (int j = threadIdx.x; j < half; j += kClThreads) {
            const int i = (col ? half : 0) + j;
            const unsigned* nb = (const unsigned*)(sm + v.on) + i * (2 * ND);
            const T* rec = cp(v, i);
            // the faces of a direction first and rhs last: the sum over the faces
            // nearly cancels against the diagonal block, so its rounding counts
            T w[NF], o[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) w[f] = (T)0;
#pragma unroll
            for (int d = 0; d < ND; ++d) {
                const unsigned ad = nb[2 * d], au = nb[2 * d + 1];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const T* k = rec + (f * ND + d) * 2;
                    w[f] = w[f] + (k[0] * ld_sh<SH>(ad + f * (int)sizeof(T), (T)0) +
                                   k[1] * ld_sh<SH>(au + f * (int)sizeof(T), (T)0));
                }
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) w[f] = bp(v, i)[f] + w[f];
            block_times(rec, w, o);
#pragma unroll
            for (int f = 0; f < NF; ++f) xp(v, i)[f] = o[f];
        }
    }

    // residual into the scratch: of the red cells after pre-smoothing (the black
    // residuals are zero and not read), else of all cells
    template <bool SH>
    __device__ __forceinline__ void residual(const ClLevel& v) const {
        const int n = A.nu1 > 0 ? 1 << (v.lch - 1) : 1 << v.lch;
        for (int i = threadIdx.x; i < n; i += kClThreads) {
            const unsigned* nb = (const unsigned*)(sm + v.on) + i * (2 * ND);
            const T* rec = cp(v, i);
            T xo[NF], s[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                xo[f] = xp(v, i)[f];
                s[f] = (T)0;
            }
#pragma unroll
            for (int d = 0; d < ND; ++d) {
                const unsigned ad = nb[2 * d], au = nb[2 * d + 1];
#pragma unroll
                for (int f = 0; f < NF; ++f) {
                    const T* k = rec + (f * ND + d) * 2;
                    s[f] = s[f] + (k[1] * (ld_sh<SH>(au + f * (int)sizeof(T), (T)0) - xo[f]) -
                                   k[0] * (xo[f] - ld_sh<SH>(ad + f * (int)sizeof(T), (T)0)));
                }
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                T mx = rec[R::kM + f * NF] * xo[0];
                if constexpr (NF == 2) mx = mx + rec[R::kM + f * NF + 1] * xo[1];
                rp(i)[f] = bp(v, i)[f] - (mx - s[f]);
            }
        }
    }

    // Right-hand side of w from the residuals of v (mean of the children; a
    // scale that is a power of two) and, on red cells, the first half sweep of
    // w's zero start; on the last level the solution
    template <bool SH>
    __device__ __forceinline__ void restrict_to(const ClLevel& v, const ClLevel& w, bool last) const {
        if (!w.shared && rank != 0) return;
        const int cx = v.n[0] != w.n[0], cy = v.n[1] != w.n[1], cz = v.n[2] != w.n[2];
        const T scale = (T)1 / (T)((1 + cx) * (1 + cy) * (1 + cz));
        const int nw = 1 << w.lch;
        for (int i = threadIdx.x; i < nw; i += kClThreads) {
            const Pos p = pos(w, flat_at(w, i));
            const int base = flat_of(v, p.a << cx, p.b << cy, p.c << cz);
            T g[NF], o[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) g[f] = (T)0;
#pragma unroll
            for (int q = 0; q < (ND == 3 ? 8 : 4); ++q) {
                const int dx = q & 1, dy = (q >> 1) & 1, dz = q >> 2, par = (dx + dy + dz) & 1;
                if (dx > cx || dy > cy || dz > cz || (par && A.nu1 > 0)) continue;
                const int fi = base + dx + (((dz << v.ly) + dy) << v.lx);
                const unsigned a = addr(A.orr, local_of(v, fi, par), fi >> v.lch);
#pragma unroll
                for (int f = 0; f < NF; ++f) g[f] = g[f] + ld_sh<SH>(a + f * (int)sizeof(T), (T)0);
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                g[f] = scale * g[f];
                bp(w, i)[f] = g[f];
            }
            const bool start = last || (A.nu1 > 0 && i < nw >> 1);
            if (start) block_times(cp(w, i), g, o);
            if (start || A.nu1 == 0)
#pragma unroll
                for (int f = 0; f < NF; ++f) xp(w, i)[f] = start ? o[f] : (T)0;
        }
    }

    // x_v += P x_w on the red cells, or on all where no black half sweep
    // follows: 3/4 of the parent and 1/4 of the parent's neighbour on the
    // cell's side (periodic wrap; at a wall the parent itself), along x, then
    // y, then z
    template <bool SH>
    __device__ __forceinline__ void prolong(const ClLevel& v, const ClLevel& w) const {
        const T w0 = (T)0.75, w1 = (T)0.25;
        const int n = A.nu2 > 0 ? 1 << (v.lch - 1) : 1 << v.lch;
        for (int i = threadIdx.x; i < n; i += kClThreads) {
            const Pos p = pos(v, flat_at(v, i));
            const int q[3] = {p.a, p.b, p.c};
            int i0[3], i1[3];
            bool cd[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                cd[d] = v.n[d] != w.n[d];
                i0[d] = cd[d] ? q[d] >> 1 : q[d];
                int k = i0[d] + ((q[d] & 1) ? 1 : -1);
                if (A.bc[d] == 0) k = k & (w.n[d] - 1);
                else if (k < 0 || k >= w.n[d]) k = i0[d];
                i1[d] = cd[d] ? k : i0[d];
            }
            T u[NF];
            // value pairs along x, combined along y and z; a direction that is not
            // coarsened takes the cell itself
            T z[2][NF];
#pragma unroll
            for (int dz = 0; dz < (ND == 3 ? 2 : 1); ++dz) {
                if (dz && !cd[2]) break;
                T y[2][NF];
#pragma unroll
                for (int dy = 0; dy < 2; ++dy) {
                    if (dy && !cd[1]) break;
                    const int b = dy ? i1[1] : i0[1], c = dz ? i1[2] : i0[2];
                    const int f0 = flat_of(w, i0[0], b, c), f1 = flat_of(w, i1[0], b, c);
                    const unsigned a0 = addr(w.ox, local_of(w, f0, (i0[0] + b + c) & 1), f0 >> w.lch);
                    const unsigned a1 = addr(w.ox, local_of(w, f1, (i1[0] + b + c) & 1), f1 >> w.lch);
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        const T x0 = ld_sh<SH>(a0 + f * (int)sizeof(T), (T)0);
                        y[dy][f] = cd[0] ? w0 * x0 + w1 * ld_sh<SH>(a1 + f * (int)sizeof(T), (T)0) : x0;
                    }
                }
#pragma unroll
                for (int f = 0; f < NF; ++f) z[dz][f] = cd[1] ? w0 * y[0][f] + w1 * y[1][f] : y[0][f];
            }
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                u[f] = (ND == 3 && cd[2]) ? w0 * z[0][f] + w1 * z[ND == 3 ? 1 : 0][f] : z[0][f];
                xp(v, i)[f] = xp(v, i)[f] + u[f];
            }
        }
    }

    template <bool SH>
    __device__ __forceinline__ void sync() const {
        if (SH) cluster_sync();
        else __syncthreads();
    }
    // one code instance per half of the cycle: the phases are short enough that
    // fetching their instructions counts
    template <bool SH>
    __device__ __forceinline__ void descend(int l, bool started) const {
        const ClLevel& v = A.lv[l];
#pragma unroll 1
        for (int h = started ? 1 : 0; h < 2 * A.nu1; ++h) {
            sweep<SH>(v, h & 1);
            sync<SH>();
        }
        residual<SH>(v);
        sync<SH>();
        restrict_to<SH>(v, A.lv[l + 1], l + 2 == A.nlev);
    }
    template <bool SH>
    __device__ __forceinline__ void ascend(int l) const {
        const ClLevel& v = A.lv[l];
        prolong<SH>(v, A.lv[l + 1]);
        sync<SH>();
#pragma unroll 1
        for (int h = 1; h <= 2 * A.nu2; ++h) {
            sweep<SH>(v, h & 1);
            sync<SH>();
        }
    }

    __device__ __forceinline__ void run() const {
        const ClLevel& top = A.lv[0];
        // one loop over the cells of all levels, so that their loads overlap
        const int nl = rank == 0 ? A.nlev : A.nshared;
        for (int i = threadIdx.x, l = 0;; i += kClThreads) {
            while (l < nl && i >= 1 << A.lv[l].lch) i -= 1 << A.lv[l++].lch;
            if (l == nl) break;
            setup(A.lv[l], i, l == 0);
        }
        __syncthreads();
        if (A.nshared > 0) cluster_sync();
#pragma unroll 1
        for (int cyc = 0; cyc < A.cycles; ++cyc) {
            const bool st = cyc == 0 && A.started;
#pragma unroll 1
            for (int l = 0; l < A.nshared; ++l) {
                descend<true>(l, l > 0 || st);
                if (l + 1 < A.nshared) cluster_sync();
            }
            if (rank == 0) {                  // the others wait at the barrier below
                __syncthreads();
#pragma unroll 1
                for (int l = A.nshared; l + 1 < A.nlev; ++l) {
                    descend<false>(l, l > 0 || st);
                    __syncthreads();
                }
#pragma unroll 1
                for (int l = A.nlev - 2; l >= A.nshared; --l) ascend<false>(l);
            }
            if (A.nshared > 0) cluster_sync();
#pragma unroll 1
            for (int l = A.nshared - 1; l >= 0; --l) ascend<true>(l);
        }
        T* x = (T*)A.x;
        for (int i = threadIdx.x; i < 1 << top.lch; i += kClThreads) {
            const int f = flat_at(top, i);
            const int g = gidx(top, f, top.lch > 0 ? i >> (top.lch - 1) : 0);
#pragma unroll
            for (int q = 0; q < NF; ++q) x[((size_t)q << top.lc) + g] = xp(top, i)[q];
        }
    }
};

template <typename T, int NF, int ND>
__global__ void __launch_bounds__(kClThreads, 1) k_vcycle_cluster(const __grid_constant__ ClArgs A) {
    pdl_wait();
    extern __shared__ __align__(16) unsigned char raw[];
    Cluster<T, NF, ND> c{A, raw, (unsigned)__cvta_generic_to_shared(raw), (int)cluster_rank()};
    c.run();
}

template <typename T>
static const void* cluster_kernel(int nf, int nd) {
    if (nf == 1) return nd == 3 ? (const void*)k_vcycle_cluster<T, 1, 3> : (const void*)k_vcycle_cluster<T, 1, 2>;
    return nd == 3 ? (const void*)k_vcycle_cluster<T, 2, 3> : (const void*)k_vcycle_cluster<T, 2, 2>;
}

// Blocks of a cluster that the current device runs with all of their shared
// memory: 16 (non-portable) or 8, or 0 where it runs neither.
template <typename T>
static int query_cluster_ctas(const void* fn) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kClSmemMax) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    for (int ctas : {16, 8}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(ctas);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = kClSmemMax;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = ctas;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n > 0) return ctas;
        cudaGetLastError();
    }
    return 0;
}
// the same, asked once per kernel and device (0.2 ms)
template <typename T>
int vcycle_cluster_ctas(int nf, int nd) {
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices][4];          // 1 + the answer
    const void* fn = cluster_kernel<T>(nf, nd);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return query_cluster_ctas<T>(fn);
    std::atomic<int>& k = known[dev][(nf == 2 ? 2 : 0) + (nd == 3 ? 1 : 0)];
    int v = k.load();
    if (v == 0) {
        v = 1 + query_cluster_ctas<T>(fn);
        k.store(v);
    }
    return v - 1;
}
template int vcycle_cluster_ctas<double>(int, int);
template int vcycle_cluster_ctas<float>(int, int);

// Largest level that the cluster takes: beyond it a half sweep on its 16 SMs
// lasts longer than a launch of its own on all SMs (about 2.6 us in a stream).
// A half sweep took 0.8 us with 16,384 FP32 cells and 5 us with 65,536; in
// FP64 1.4 us with 4,096 two-field cells and 3.5-5 us with 16,384.  V(1,1) cycles
// with these limits and with a quarter of them: 17 and 24 us at 128^2 (FP32, one
// field), 37 and 51 at 64^2 (FP64, two fields).  Between one and four times the
// limits the cluster is still the faster one in places (FP32, one field, 32^3: 20
// against 27 us; FP64, two fields, 32 x 16 x 16: 47 against 53).
static long long cluster_max_cells(int nf, int elt) { return elt == 8 ? (nf == 1 ? 16384 : 4096) : 16384; }

template <typename T>
size_t vcycle_cluster_top(int nf, int nd, const std::vector<MGLevel>& levels, int ctas) {
    if (ctas == 0) return levels.size();
    ClArgs A;
    for (size_t l = 0; l + 1 < levels.size(); ++l) {
        const int nlev = (int)(levels.size() - l);
        if (nlev > kClMaxLevels || levels[l].ncell > cluster_max_cells(nf, sizeof(T))) continue;
        if (cluster_plan<T>(&levels[l], nlev, nf, nd, ctas, A) <= (size_t)kClSmemMax) return l;
    }
    return levels.size();
}
template size_t vcycle_cluster_top<double>(int, int, const std::vector<MGLevel>&, int);
template size_t vcycle_cluster_top<float>(int, int, const std::vector<MGLevel>&, int);

template <typename T>
void launch_vcycle_cluster(const Grid& G, int nf, const MGLevel* levels, int nlev, int nu1, int nu2, int cycles,
                           int started, int ctas, cudaStream_t s, int tr) {
    ClArgs A;
    const size_t bytes = cluster_plan<T>(levels, nlev, nf, G.ndim, ctas, A);
    for (int d = 0; d < 3; ++d) A.bc[d] = G.bc[d];
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.cycles = cycles;
    A.started = started && nu1 > 0;
    A.tr = tr;
    A.rhs = levels[0].rhs;
    A.x = levels[0].x;
    const int n = A.nshared > 0 ? ctas : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;     // see launch_k
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    void* args[] = {&A};
    ++g_launch_count;
    cudaLaunchKernelExC(&cfg, cluster_kernel<T>(nf, G.ndim), args);
}
template void launch_vcycle_cluster<double>(const Grid&, int, const MGLevel*, int, int, int, int, int, int,
                                            cudaStream_t, int);
template void launch_vcycle_cluster<float>(const Grid&, int, const MGLevel*, int, int, int, int, int, int,
                                           cudaStream_t, int);

}  // namespace jfnk
