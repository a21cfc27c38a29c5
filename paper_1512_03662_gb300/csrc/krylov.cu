// GMRES kernels (paper Sect. 4.1, Eq. forcing_term; restarted GMRES of Saad &
// Schultz 1986 with classical Gram-Schmidt):
//   * multi-dot: h_i = <v_i, w> for all basis vectors in ONE pass over w,
//     accumulated in double whatever the storage type;
//   * AXPY + norm: w -= sum_i h_i s_i v_i and ||w||^2 in the same pass;
//   * lazy normalisation: v_{j+1} keeps the unnormalised w, its scale
//     s_{j+1} = 1/||w|| is applied by every reader, which saves a pass;
//   * the second stages of the reductions, the Hessenberg column and its Givens
//     rotation run in the last block of the kernel before them, the triangular
//     solve in one thread (m <= 64); the host only reads the residual estimate.
// Reductions are two-stage with a fixed block count and a fixed summation
// order, so results are bit-reproducible from run to run.
#include "common.cuh"
#include "kernels.h"

namespace jfnk {

// Grid of a grid-stride reduction: as many blocks as are resident on all
// SMs at once (one wave: no tail wave, every SM equally loaded), capped at
// kMaxRedBlocks.  Fixed per kernel and device, so the summation order and
// the results stay reproducible.
static int red_grid(const void* fn) {
    int dev = 0, nsm = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, kBlock, 0);
    long long g = (long long)(nsm > 0 ? nsm : 1) * (occ > 0 ? occ : 1);
    return (int)(g < kMaxRedBlocks ? g : kMaxRedBlocks);
}

// one cached grid per kernel (the kernel is the template argument, so each
// instantiation has its own thread-safe static)
template <auto FN>
static int cached_grid() {
    static const int g = red_grid((const void*)FN);
    return g;
}

__global__ void k_finalize(const double* partials, int n, int stride, double* scal, int slot, int op) {
    pdl_wait();
    __shared__ double sh[32];
    double v = (op == 2) ? 0.0 : 0.0;
    bool nan = false;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double x = partials[(long long)i * stride];
        if (!(x == x)) nan = true;
        if (op == 2) v = fmax(v, x); else v += x;
    }
    double r = (op == 2) ? block_max<1024>(v, sh) : block_sum<1024>(v, sh);
    int anynan = __syncthreads_or(nan);
    if (threadIdx.x == 0) {
        if (anynan) r = __longlong_as_double(0x7ff8000000000000ULL);
        scal[slot] = (op == 0) ? sqrt(r) : r;
    }
}

// first stage for many partials: block b reduces its share in place, to
// partials[b * share] (a NaN makes the result one, a maximum too)
__global__ void k_prefinalize(double* partials, int n, int share, int op) {
    pdl_wait();
    __shared__ double sh[32];
    double* p = partials + (long long)blockIdx.x * share;
    const int m = min(share, n - (int)blockIdx.x * share);
    double v = 0.0;
    bool nan = false;
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const double x = p[i];
        if (!(x == x)) nan = true;
        if (op == 2) v = fmax(v, x);
        else v += x;
    }
    double r = (op == 2) ? block_max<256>(v, sh) : block_sum<256>(v, sh);
    const int anynan = __syncthreads_or(nan);
    if (threadIdx.x == 0) p[0] = anynan ? __longlong_as_double(0x7ff8000000000000ULL) : r;
}

// A cell kernel leaves one partial per 128 cells: 131,072 at 256^3, which one
// block's two FP64 lanes added in 117 us.  From kStageMin on, 128 blocks add
// their shares first.
void launch_finalize(double* partials, int n, double* scal, int slot, int op, cudaStream_t s) {
    constexpr int kStageMin = 8192, kStageBlocks = 128;
    int stride = 1;
    if (n >= kStageMin) {
        stride = (n + kStageBlocks - 1) / kStageBlocks;
        const int blocks = (n + stride - 1) / stride;
        ++g_launch_count;
        launch_k(k_prefinalize, blocks, 256, 0, s, partials, n, stride, op);
        n = blocks;
    }
    ++g_launch_count;
    launch_k(k_finalize, 1, 1024, 0, s, partials, n, stride, scal, slot, op);
}

__global__ void k_delta(double* scal, double lambda, int pert) {
    pdl_wait();
    const double zn = scal[kSlotZnorm];
    if (pert == 0) {
        set_delta(scal, zn, lambda);
        return;
    }
    const double uv = scal[kSlotTmp];
    const double sgn = uv >= 0.0 ? 1.0 : -1.0;
    const double d = lambda * (1e-12 / lambda + fabs(uv) / (zn * zn)) * sgn;
    scal[kSlotDelta] = d;
    scal[kSlotInvDelta] = 1.0 / d;
}

void launch_delta(double* scal, double lambda, int pert, cudaStream_t s) { launch_k(k_delta, 1, 1, 0, s, scal, lambda, pert); }

// partial sums of x_i^2: in double for a double x; for a float x as a
// compensated float pair per thread (no FP64 instruction per element),
// converted to double once per thread, or redone in double by a thread whose
// values are too large or too small for float squares (sq_range_unsafe)
template <typename T>
__global__ void k_norm2(const T* x, long long n, double* partials) {
    pdl_wait();
    __shared__ double sh[32];
    double acc = 0.0;
    CompF accf = {0.f, 0.f};
    float mx = 0.f;
    const long long i0 = blockIdx.x * (long long)blockDim.x + threadIdx.x, st = (long long)gridDim.x * blockDim.x;
    for (long long i = i0; i < n; i += st) {
        if (sizeof(T) == 8) {
            const double v = (double)x[i];
            acc += v * v;
        } else {
            const float v = (float)x[i];
            comp_fma(accf, v, v);
            mx = fmaxf(mx, fabsf(v));
        }
    }
    if (sizeof(T) != 8) {
        if (sq_range_unsafe(mx)) {
            for (long long i = i0; i < n; i += st) {
                const double v = (double)x[i];
                acc += v * v;
            }
        } else {
            acc = (double)accf.s + (double)accf.e;
        }
    }
    double s = block_sum<kBlock>(acc, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

template <typename T>
void launch_norm2_partials(const T* x, long long n, double* partials, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_norm2<T>, kRedBlocks, kBlock, 0, s, x, n, partials);
}
template void launch_norm2_partials<double>(const double*, long long, double*, cudaStream_t);
template void launch_norm2_partials<float>(const float*, long long, double*, cudaStream_t);

// partial sums of (a_i * ainv_i) * b_i  (used for x^ . z with x^ = X R^-1)
template <typename T>
__global__ void k_dot(const double* a, const double* ainv, const T* b,
                      long long n, double* partials) {
    pdl_wait();
    __shared__ double sh[32];
    double acc = 0.0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        acc += (a[i] * ainv[i]) * (double)b[i];
    double s = block_sum<kBlock>(acc, sh);
    if (threadIdx.x == 0) partials[blockIdx.x] = s;
}

template <typename T>
void launch_dot_partials(const double* a, const double* ainv, const T* b, long long n, double* partials,
                         cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_dot<T>, kRedBlocks, kBlock, 0, s, a, ainv, b, n, partials);
}
template void launch_dot_partials<double>(const double*, const double*, const double*, long long, double*, cudaStream_t);
template void launch_dot_partials<float>(const double*, const double*, const float*, long long, double*, cudaStream_t);

// End of a multi-dot: the block's partial sums of v_i . w to partials[blk * NV + i],
// and hcol[i] = vscale[i] times their sum over the blocks by the last block,
// one warp per value.  (A launch of its own for the second stage cost 5 us,
// and a block reduction per value, two barriers and ten dependent FP64
// additions each, up to 30 us on the small grids.)
template <int NV>
__device__ __forceinline__ void finish_dots(double (&acc)[NV], double* sh, const GsState& S, double* hcol) {
    block_sums<kBlock, NV>(acc, sh, S.partials + (long long)blockIdx.x * NV);
    if (!last_block(S.counter, gridDim.x)) return;
    const int lane = threadIdx.x & 31;
    for (int i = threadIdx.x >> 5; i < NV; i += kBlock / 32) {
        double v = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(S.partials + (long long)b * NV + i);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) hcol[i] = v * S.vscale[i];
    }
}

// one pass over w: sums of v_i * w
template <typename T, int NV>
__global__ void k_multidot(const T* V, long long ld, const T* w, long long n,
                           GsState S, double* hcol) {
    pdl_wait();
    __shared__ double sh[kBlock / 32 * NV];
    double acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double wk = (double)w[k];
#pragma unroll
        for (int i = 0; i < NV; ++i) acc[i] += (double)V[i * ld + k] * wk;
    }
    finish_dots<NV>(acc, sh, S, hcol);
}

// float basis: compensated FP32 accumulation per thread, double per block
template <int NV>
__global__ void k_multidot_f32(const float* V, long long ld, const float* w, long long n,
                               GsState S, double* hcol) {
    pdl_wait();
    __shared__ double sh[kBlock / 32 * NV];
    CompF acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = CompF{0.f, 0.f};
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        float wk = w[k];
#pragma unroll
        for (int i = 0; i < NV; ++i) comp_fma(acc[i], V[i * ld + k], wk);
    }
    double sums[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) sums[i] = (double)acc[i].s + (double)acc[i].e;
    finish_dots<NV>(sums, sh, S, hcol);
}

// The same with 16-byte loads: each thread takes four consecutive elements
// per step, which keeps enough bytes in flight per SM to cover HBM latency
// when the basis is short (one load instruction per vector per four
// elements).  Needs ld % 4 == 0 and 16-byte aligned V and w; the n % 4 tail
// is summed element by element.
template <int NV>
__global__ void __launch_bounds__(kBlock) k_multidot_f32v(const float* V, long long ld,
                                                          const float* w, long long n,
                                                          GsState S, double* hcol) {
    pdl_wait();
    __shared__ double sh[kBlock / 32 * NV];
    CompF acc[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) acc[i] = CompF{0.f, 0.f};
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n4 = n >> 2;
    const float4* w4 = reinterpret_cast<const float4*>(w);
    for (long long k = t0; k < n4; k += stride) {
        const float4 wk = w4[k];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const float4 v = reinterpret_cast<const float4*>(V + i * ld)[k];
            comp_fma(acc[i], v.x, wk.x);
            comp_fma(acc[i], v.y, wk.y);
            comp_fma(acc[i], v.z, wk.z);
            comp_fma(acc[i], v.w, wk.w);
        }
    }
    for (long long k = 4 * n4 + t0; k < n; k += stride) {
        const float wk = w[k];
#pragma unroll
        for (int i = 0; i < NV; ++i) comp_fma(acc[i], V[i * ld + k], wk);
    }
    double sums[NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) sums[i] = (double)acc[i].s + (double)acc[i].e;
    finish_dots<NV>(sums, sh, S, hcol);
}

// generic fallback for any count: groups of up to 8 vectors, one launch each
template <typename T>
__global__ void k_multidot_group(const T* V, long long ld, int ni, const T* w, long long n,
                                 GsState S, double* hcol) {
    pdl_wait();
    __shared__ double sh[kBlock / 32 * 8], out[8];
    double acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double wk = (double)w[k];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (i < ni) acc[i] += (double)V[i * ld + k] * wk;
    }
    block_sums<kBlock, 8>(acc, sh, out);
    __syncthreads();
    if (threadIdx.x < 8) S.partials[(long long)blockIdx.x * 8 + threadIdx.x] = out[threadIdx.x];
    if (!last_block(S.counter, gridDim.x)) return;
    const int lane = threadIdx.x & 31, i = threadIdx.x >> 5;
    if (i >= ni) return;
    double v = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(S.partials + (long long)b * 8 + i);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) hcol[i] = v * S.vscale[i];
}

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Blocks of a reduction over n elements, `per` per thread and step: one wave,
// but no more than have work (the last block adds one partial per block).
static int red_blocks(int wave, long long n, int per) {
    const long long need = (n + (long long)kBlock * per - 1) / ((long long)kBlock * per);
    return (int)(need < wave ? (need > 0 ? need : 1) : wave);
}

template <typename T>
void launch_multidot(const T* V, long long ld, int nv, const T* w, long long n, const GsState& S, double* hcol,
                     cudaStream_t s) {
    if (sizeof(T) == 4 && nv <= 32) {
        const float* Vf = (const float*)V;
        const float* wf = (const float*)w;
        const bool vec = ld % 4 == 0 && aligned16(V) && aligned16(w);
        ++g_launch_count;
        switch (nv) {
#define CASEF(N)                                                                                   \
    case N:                                                                                        \
        if (vec)                                                                                   \
            launch_k(k_multidot_f32v<N>, red_blocks(cached_grid<k_multidot_f32v<N>>(), n, 4), kBlock, 0, s, \
                     Vf, ld, wf, n, S, hcol);                                                      \
        else                                                                                       \
            launch_k(k_multidot_f32<N>, red_blocks(cached_grid<k_multidot_f32<N>>(), n, 1), kBlock, 0, s, Vf, \
                     ld, wf, n, S, hcol);                                                          \
        return;
            CASEF(1) CASEF(2) CASEF(3) CASEF(4) CASEF(5) CASEF(6) CASEF(7) CASEF(8)
            CASEF(9) CASEF(10) CASEF(11) CASEF(12) CASEF(13) CASEF(14) CASEF(15) CASEF(16)
            CASEF(17) CASEF(18) CASEF(19) CASEF(20) CASEF(21) CASEF(22) CASEF(23) CASEF(24)
            CASEF(25) CASEF(26) CASEF(27) CASEF(28) CASEF(29) CASEF(30) CASEF(31) CASEF(32)
#undef CASEF
        }
    }
    switch (nv) {
#define CASE(N)                                                                                    \
    case N:                                                                                        \
        ++g_launch_count;                                                                          \
        launch_k(k_multidot<T, N>, red_blocks(cached_grid<k_multidot<T, N>>(), n, 1), kBlock, 0, s, V, ld, w, n, S, hcol); \
        return;
        CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8)
        CASE(9) CASE(10) CASE(11) CASE(12) CASE(13) CASE(14) CASE(15) CASE(16)
#undef CASE
        default:
            for (int i0 = 0; i0 < nv; i0 += 8) {
                const int ni = nv - i0 < 8 ? nv - i0 : 8;
                GsState Si = S;
                Si.vscale = S.vscale + i0;
                ++g_launch_count;
                launch_k(k_multidot_group<T>, red_blocks(cached_grid<k_multidot_group<T>>(), n, 1), kBlock, 0, s,
                         V + i0 * ld, ld, ni, w, n, Si, hcol + i0);
            }
    }
}
template void launch_multidot<double>(const double*, long long, int, const double*, long long, const GsState&, double*,
                                      cudaStream_t);
template void launch_multidot<float>(const float*, long long, int, const float*, long long, const GsState&, double*,
                                     cudaStream_t);

// what ends a Gram-Schmidt pass: column < 0 the norm only (see launch_axpy_norm)
struct GsFinish {
    int column;
    const double* more;
    int col_scale_slot;
};

// End of a GMRES iteration, by one block; nrm = |w| in thread 0.
//   Subdiagonal entry h_{j+1,j} = |w|, lazy scale 1/|w|.  With w = delta J^ z
// (kModeJvD) the pass ran on delta times the true vector: every coefficient and
// the norm carry the factor delta, and the normalised v_{j+1} is the same, so
// only the column is rescaled.
//   Givens: apply the previous rotations to column j, form rotation j, update
// g; scal[kSlotRes] = |g_{j+1}|.  One thread's chain on operands staged in
// shared memory.
__device__ __forceinline__ void gs_end(double nrm, const double* hcol, const GsState& S, const GsFinish& F) {
    __shared__ double hs[64], c[64], d[64];
    const int j = F.column;
    const bool scaled = F.col_scale_slot >= 0;
    const double f = scaled ? S.scal[F.col_scale_slot] : 1.0;
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
        const double h = F.more ? hcol[i] + F.more[i] : hcol[i];
        hs[i] = scaled ? h * f : h;
        if (i < j) {
            c[i] = S.cs[i];
            d[i] = S.sn[i];
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    S.vscale[j + 1] = nrm > 0.0 ? 1.0 / nrm : 0.0;
    double* h = S.H + (long long)j * S.ldh;
    double x = hs[0];
    for (int i = 0; i < j; ++i) {
        const double y = hs[i + 1];
        h[i] = c[i] * x + d[i] * y;
        x = -d[i] * x + c[i] * y;
    }
    const double b = scaled ? nrm * f : nrm;
    const double den = sqrt(x * x + b * b);
    double cj = 1.0, sj = 0.0;
    if (den != 0.0) { cj = x / den; sj = b / den; }
    S.cs[j] = cj;
    S.sn[j] = sj;
    h[j] = cj * x + sj * b;
    h[j + 1] = 0.0;
    const double gj = S.g[j], gn = -sj * gj;
    S.g[j + 1] = gn;
    S.g[j] = cj * gj;
    S.scal[kSlotRes] = fabs(gn);
}

// end of the AXPY: the last block adds the partial sums of |w|^2
__device__ __forceinline__ void finish_axpy(double sum, double* sh, const double* hcol, const GsState& S,
                                            const GsFinish& F) {
    const double t = block_sum<kBlock>(sum, sh);
    if (threadIdx.x == 0) S.partials[blockIdx.x] = t;
    if (!last_block(S.counter, gridDim.x)) return;
    double a = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kBlock) a += __ldcg(S.partials + b);
    const double nrm = sqrt(block_sum<kBlock>(a, sh));
    if (threadIdx.x == 0) S.scal[kSlotTmp] = nrm;
    if (F.column >= 0) gs_end(nrm, hcol, S, F);
}

__global__ void k_gs_end(GsState S, GsFinish F, const double* hcol) {
    pdl_wait();
    gs_end(S.scal[kSlotTmp], hcol, S, F);
}

void launch_gs_end(const GsState& S, int column, const double* hcol, int col_scale_slot, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_gs_end, 1, 64, 0, s, S, GsFinish{column, nullptr, col_scale_slot}, hcol);
}

// w -= sum_i (h_i s_i) v_i ; partial ||w||^2
template <typename T, int NV>
__global__ void k_axpy_norm(T* w, const T* V, long long ld, const double* hcol,
                            long long n, GsState S, GsFinish F) {
    pdl_wait();
    __shared__ double sh[32];
    __shared__ double coef[64];
    if (threadIdx.x < NV) coef[threadIdx.x] = hcol[threadIdx.x] * S.vscale[threadIdx.x];
    __syncthreads();
    double acc = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double x = (double)w[k];
#pragma unroll
        for (int i = 0; i < NV; ++i) x -= coef[i] * (double)V[i * ld + k];
        T xs = (T)x;
        w[k] = xs;
        double xd = (double)xs;
        acc += xd * xd;
    }
    finish_axpy(acc, sh, hcol, S, F);
}

template <typename T>
__global__ void k_axpy_norm_dyn(T* w, const T* V, long long ld, int nv,
                                const double* hcol,
                            long long n, GsState S, GsFinish F) {
    pdl_wait();
    __shared__ double sh[32];
    __shared__ double coef[64];
    if (threadIdx.x < nv) coef[threadIdx.x] = hcol[threadIdx.x] * S.vscale[threadIdx.x];
    __syncthreads();
    double acc = 0.0;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        double x = (double)w[k];
        for (int i = 0; i < nv; ++i) x -= coef[i] * (double)V[i * ld + k];
        T xs = (T)x;
        w[k] = xs;
        double xd = (double)xs;
        acc += xd * xd;
    }
    finish_axpy(acc, sh, hcol, S, F);
}

// float basis: w -= sum_i c_i v_i with c_i split into float hi + lo parts and
// the sum kept as a compensated pair; ||w||^2 of the rounded result, compensated.
template <int NV>
__global__ void k_axpy_norm_f32(float* w, const float* V, long long ld,
                                const double* hcol,
                            long long n, GsState S, GsFinish F) {
    pdl_wait();
    __shared__ double sh[32];
    __shared__ float chi[32], clo[32];
    if (threadIdx.x < NV) {
        double c = -(hcol[threadIdx.x] * S.vscale[threadIdx.x]);
        float h = (float)c;
        chi[threadIdx.x] = h;
        clo[threadIdx.x] = (float)(c - (double)h);
    }
    __syncthreads();
    CompF nrm{0.f, 0.f};
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n; k += (long long)gridDim.x * blockDim.x) {
        CompF x{w[k], 0.f};
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            float v = V[i * ld + k];
            comp_fma(x, chi[i], v);
            x.e = fmaf(clo[i], v, x.e);
        }
        float xs = x.s + x.e;
        w[k] = xs;
        comp_fma(nrm, xs, xs);
    }
    finish_axpy((double)nrm.s + (double)nrm.e, sh, hcol, S, F);
}

// The same with 16-byte loads and stores (four consecutive elements per
// thread and step); needs ld % 4 == 0 and 16-byte aligned w and V.
template <int NV>
__global__ void __launch_bounds__(kBlock) k_axpy_norm_f32v(float* w, const float* V,
                                                           long long ld, const double* hcol,
                            long long n, GsState S, GsFinish F) {
    pdl_wait();
    __shared__ double sh[32];
    __shared__ float chi[32], clo[32];
    if (threadIdx.x < NV) {
        double c = -(hcol[threadIdx.x] * S.vscale[threadIdx.x]);
        float h = (float)c;
        chi[threadIdx.x] = h;
        clo[threadIdx.x] = (float)(c - (double)h);
    }
    __syncthreads();
    CompF nrm{0.f, 0.f};
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n4 = n >> 2;
    float4* w4 = reinterpret_cast<float4*>(w);
    for (long long k = t0; k < n4; k += stride) {
        const float4 wk = w4[k];
        CompF x0{wk.x, 0.f}, x1{wk.y, 0.f}, x2{wk.z, 0.f}, x3{wk.w, 0.f};
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const float4 v = reinterpret_cast<const float4*>(V + i * ld)[k];
            const float ch = chi[i], cl = clo[i];
            comp_fma(x0, ch, v.x);
            x0.e = fmaf(cl, v.x, x0.e);
            comp_fma(x1, ch, v.y);
            x1.e = fmaf(cl, v.y, x1.e);
            comp_fma(x2, ch, v.z);
            x2.e = fmaf(cl, v.z, x2.e);
            comp_fma(x3, ch, v.w);
            x3.e = fmaf(cl, v.w, x3.e);
        }
        float4 o;
        o.x = x0.s + x0.e;
        o.y = x1.s + x1.e;
        o.z = x2.s + x2.e;
        o.w = x3.s + x3.e;
        w4[k] = o;
        comp_fma(nrm, o.x, o.x);
        comp_fma(nrm, o.y, o.y);
        comp_fma(nrm, o.z, o.z);
        comp_fma(nrm, o.w, o.w);
    }
    for (long long k = 4 * n4 + t0; k < n; k += stride) {
        CompF x{w[k], 0.f};
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            float v = V[i * ld + k];
            comp_fma(x, chi[i], v);
            x.e = fmaf(clo[i], v, x.e);
        }
        float xs = x.s + x.e;
        w[k] = xs;
        comp_fma(nrm, xs, xs);
    }
    finish_axpy((double)nrm.s + (double)nrm.e, sh, hcol, S, F);
}

template <typename T>
void launch_axpy_norm(T* w, const T* V, long long ld, int nv, const double* hcol, long long n, const GsState& S,
                      int column, const double* more, int col_scale_slot, cudaStream_t s) {
    const GsFinish F = {column, more, col_scale_slot};
    ++g_launch_count;
    if (sizeof(T) == 4 && nv <= 32) {
        float* wf = (float*)w;
        const float* Vf = (const float*)V;
        const bool vec = ld % 4 == 0 && aligned16(V) && aligned16(w);
        switch (nv) {
#define CASEF(N)                                                                                   \
    case N:                                                                                        \
        if (vec)                                                                                   \
            launch_k(k_axpy_norm_f32v<N>, red_blocks(cached_grid<k_axpy_norm_f32v<N>>(), n, 4), kBlock, 0, s, \
                     wf, Vf, ld, hcol, n, S, F);                                                   \
        else                                                                                       \
            launch_k(k_axpy_norm_f32<N>, red_blocks(cached_grid<k_axpy_norm_f32<N>>(), n, 1), kBlock, 0, s, wf, \
                     Vf, ld, hcol, n, S, F);                                                       \
        return;
            CASEF(1) CASEF(2) CASEF(3) CASEF(4) CASEF(5) CASEF(6) CASEF(7) CASEF(8)
            CASEF(9) CASEF(10) CASEF(11) CASEF(12) CASEF(13) CASEF(14) CASEF(15) CASEF(16)
            CASEF(17) CASEF(18) CASEF(19) CASEF(20) CASEF(21) CASEF(22) CASEF(23) CASEF(24)
            CASEF(25) CASEF(26) CASEF(27) CASEF(28) CASEF(29) CASEF(30) CASEF(31) CASEF(32)
#undef CASEF
        }
    }
    switch (nv) {
#define CASE(N)                                                                                    \
    case N:                                                                                        \
        launch_k(k_axpy_norm<T, N>, red_blocks(cached_grid<k_axpy_norm<T, N>>(), n, 1), kBlock, 0, s, w, V, ld, \
                 hcol, n, S, F);                                                                   \
        return;
        CASE(1) CASE(2) CASE(3) CASE(4) CASE(5) CASE(6) CASE(7) CASE(8)
        CASE(9) CASE(10) CASE(11) CASE(12) CASE(13) CASE(14) CASE(15) CASE(16)
#undef CASE
        default:
            launch_k(k_axpy_norm_dyn<T>, red_blocks(cached_grid<k_axpy_norm_dyn<T>>(), n, 1), kBlock, 0, s, w, V, ld, nv,
                     hcol, n, S, F);
    }
}
template void launch_axpy_norm<double>(double*, const double*, long long, int, const double*, long long,
                                       const GsState&, int, const double*, int, cudaStream_t);
template void launch_axpy_norm<float>(float*, const float*, long long, int, const double*, long long, const GsState&,
                                      int, const double*, int, cudaStream_t);

__global__ void k_backsolve(const double* H, int ldh, int k, const double* g, double* y) {
    pdl_wait();
    for (int i = k - 1; i >= 0; --i) {
        double s = g[i];
        for (int l = i + 1; l < k; ++l) s -= H[(long long)l * ldh + i] * y[l];
        y[i] = s / H[(long long)i * ldh + i];
    }
}

void launch_backsolve(const double* H, int ldh, int k, const double* g, double* y, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_backsolve, 1, 1, 0, s, H, ldh, k, g, y);
}

// x += sum_{i<k} y_i Z_i
template <typename T>
__global__ void k_update(double* x, const T* Z, long long ld, int k,
                         const double* y, long long n) {
    pdl_wait();
    __shared__ double ys[64];
    if (threadIdx.x < k) ys[threadIdx.x] = y[threadIdx.x];
    __syncthreads();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        double v = x[e];
        for (int i = 0; i < k; ++i) v = v + ys[i] * (double)Z[i * ld + e];
        x[e] = v;
    }
}

// The same for a float basis: the products and their sum run on the FP32
// pipe as an unevaluated pair (TwoProduct, TwoSum; each y_i split into two
// floats), four elements per thread with 16-byte loads.  In double, the k
// FMAs per element bound this pass by the FP64 pipe (k up to 30 at 84
// million unknowns).  Columns of Z start on 16-byte boundaries (ld is a
// multiple of 64) and x is 256-byte aligned; the last n mod 4 elements take
// the scalar loop.
__global__ void __launch_bounds__(kBlock) k_update_f32v(double* x, const float* Z,
                                                        long long ld, int k, const double* y,
                                                        long long n) {
    pdl_wait();
    __shared__ float yh[64], yl[64];
    if (threadIdx.x < k) {
        const double c = y[threadIdx.x];
        const float h = (float)c;
        yh[threadIdx.x] = h;
        yl[threadIdx.x] = (float)(c - (double)h);
    }
    __syncthreads();
    const long long t0 = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long n4 = n >> 2;
    for (long long q = t0; q < n4; q += stride) {
        CompF a0{0.f, 0.f}, a1{0.f, 0.f}, a2{0.f, 0.f}, a3{0.f, 0.f};
#pragma unroll 4
        for (int i = 0; i < k; ++i) {
            const float4 v = reinterpret_cast<const float4*>(Z + i * ld)[q];
            const float h = yh[i], l = yl[i];
            comp_fma(a0, h, v.x);
            a0.e = fmaf(l, v.x, a0.e);
            comp_fma(a1, h, v.y);
            a1.e = fmaf(l, v.y, a1.e);
            comp_fma(a2, h, v.z);
            a2.e = fmaf(l, v.z, a2.e);
            comp_fma(a3, h, v.w);
            a3.e = fmaf(l, v.w, a3.e);
        }
        double2* xp = reinterpret_cast<double2*>(x) + 2 * q;
        double2 lo = xp[0], hi = xp[1];
        lo.x += (double)a0.s + (double)a0.e;
        lo.y += (double)a1.s + (double)a1.e;
        hi.x += (double)a2.s + (double)a2.e;
        hi.y += (double)a3.s + (double)a3.e;
        xp[0] = lo;
        xp[1] = hi;
    }
    for (long long e = 4 * n4 + t0; e < n; e += stride) {
        CompF a{0.f, 0.f};
        for (int i = 0; i < k; ++i) {
            const float z = Z[i * ld + e];
            comp_fma(a, yh[i], z);
            a.e = fmaf(yl[i], z, a.e);
        }
        x[e] += (double)a.s + (double)a.e;
    }
}

template <typename T>
void launch_update(double* x, const T* Z, long long ld, int k, const double* y, long long n, cudaStream_t s) {
    ++g_launch_count;
    if (sizeof(T) == 4 && ld % 4 == 0) {
        const int g = cached_grid<k_update_f32v>();
        launch_k(k_update_f32v, g, kBlock, 0, s, x, (const float*)Z, ld, k, y, n);
    } else {
        launch_k(k_update<T>, kRedBlocks, kBlock, 0, s, x, Z, ld, k, y, n);
    }
}
template void launch_update<double>(double*, const double*, long long, int, const double*, long long, cudaStream_t);
template void launch_update<float>(double*, const float*, long long, int, const double*, long long, cudaStream_t);

// dst = src * (alpha, or scal[slot], or 1/scal[slot])
template <typename TS, typename TD>
__global__ void k_scale_copy(const TS* src, double alpha, const double* scal, int slot, int invert,
                             TD* dst, long long n) {
    pdl_wait();
    double a = alpha;
    if (slot >= 0) a = invert ? 1.0 / scal[slot] : scal[slot];
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        dst[e] = (TD)((double)src[e] * a);
}

template <typename TS, typename TD>
void launch_scale_copy(const TS* src, double alpha, const double* scal, int slot, int invert, TD* dst, long long n,
                       cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_scale_copy<TS, TD>, kRedBlocks, kBlock, 0, s, src, alpha, scal, slot, invert, dst, n);
}
template void launch_scale_copy<double, double>(const double*, double, const double*, int, int, double*, long long, cudaStream_t);
template void launch_scale_copy<double, float>(const double*, double, const double*, int, int, float*, long long, cudaStream_t);
template void launch_scale_copy<float, float>(const float*, double, const double*, int, int, float*, long long, cudaStream_t);
template void launch_scale_copy<float, double>(const float*, double, const double*, int, int, double*, long long, cudaStream_t);

// X += R dxh ; partial max |dxh| (NaN propagates)
__global__ void k_newton_update(double* X, const double* R, const double* dxh,
                                long long n, double* partials) {
    pdl_wait();
    __shared__ double sh[32];
    double m = 0.0;
    bool nan = false;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        double d = dxh[e];
        X[e] = X[e] + R[e] * d;
        double a = fabs(d);
        if (!(a == a)) nan = true;
        m = fmax(m, a);
    }
    double r = block_max<kBlock>(m, sh);
    int anynan = __syncthreads_or(nan);
    if (threadIdx.x == 0) partials[blockIdx.x] = anynan ? __longlong_as_double(0x7ff8000000000000ULL) : r;
}

void launch_newton_update(double* X, const double* R, const double* dxh, long long n, double* partials,
                          cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_newton_update, kRedBlocks, kBlock, 0, s, X, R, dxh, n, partials);
}

template <typename T>
__global__ void k_zero(T* x, long long n) {
    pdl_wait();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
        x[e] = (T)0;
}

template <typename T>
void launch_zero(T* x, long long n, cudaStream_t s) { launch_k(k_zero<T>, kRedBlocks, kBlock, 0, s, x, n); }
template void launch_zero<double>(double*, long long, cudaStream_t);
template void launch_zero<float>(float*, long long, cudaStream_t);

// r = b - r with b = -(G0 - b^n) L^-1 (the Newton right-hand side, rebuilt in
// double for a GMRES restart); r holds J^ x on entry
template <typename T>
__global__ void k_restart_residual(T* r, const double* G0, const double* bn,
                                   const double* Linv, long long n) {
    pdl_wait();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        double b = -((G0[e] - bn[e]) * Linv[e]);
        r[e] = (T)(b - (double)r[e]);
    }
}

template <typename T>
void launch_restart_residual(T* r, const double* G0, const double* bn, const double* Linv, long long n,
                             cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_restart_residual<T>, kRedBlocks, kBlock, 0, s, r, G0, bn, Linv, n);
}
template void launch_restart_residual<double>(double*, const double*, const double*, const double*, long long,
                                              cudaStream_t);
template void launch_restart_residual<float>(float*, const double*, const double*, const double*, long long,
                                             cudaStream_t);

// start of a GMRES cycle: g = (beta, 0, ...), vscale[0] = 1/beta
__global__ void k_init_cycle(double* scal, double* g, double* vscale, int m) {
    pdl_wait();
    double beta = scal[kSlotBeta];
    for (int i = 0; i <= m; ++i) g[i] = 0.0;
    g[0] = beta;
    vscale[0] = beta > 0.0 ? 1.0 / beta : 0.0;
}

void launch_init_cycle(double* scal, double* g, double* vscale, int m, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_init_cycle, 1, 1, 0, s, scal, g, vscale, m);
}

// P = L^-1/dt, Q = theta L^-1, C = L^-1 G(X) of the Jacobian-free assemble;
// entries from u_begin on (the momentum rows, whose conserved value the
// assemble forms as 2 rho_f u) take P = L^-1/(2 dt)
__global__ void k_jv_coeffs(const double* Linv, const double* G0, double idt, double idt_h,
                            double theta, double* P, double* Q, double* C,
                            long long n, long long u_begin) {
    pdl_wait();
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const double li = Linv[e];
        P[e] = (e < u_begin ? idt : idt_h) * li;
        Q[e] = theta * li;
        C[e] = G0[e] * li;
    }
}

void launch_jv_coeffs(const double* Linv, const double* G0, double dt, double theta, double* P, double* Q, double* C,
                      long long n, long long u_begin, cudaStream_t s) {
    ++g_launch_count;
    launch_k(k_jv_coeffs, kRedBlocks, kBlock, 0, s, Linv, G0, 1.0 / dt, 0.5 / dt, theta, P, Q, C, n, u_begin);
}

}  // namespace jfnk
