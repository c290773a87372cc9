// FP64 Lanczos eigensolver on the GPU around the H_eff matvec (the eigensolver of the
// two-site DMRG step, Section II-C / III; Lanczos is the fixed-iteration alternative to
// the Davidson routine of Algorithm 1).
//
// Every vector operation runs in FP64 on the device and the loop never synchronises with
// the host.  Per iteration k, the matvec and one cooperative kernel (lz_step_kernel):
//   w = H v_k                       (heff_apply_prepared; any precision, FP64 vectors)
//   a = v_k . (w - beta_{k-1} v_{k-1}),  w -= beta_{k-1} v_{k-1} + a v_k
//                                   (the three-term recurrence, with ||w||^2 after it)
//   h = V^T w, w -= V h             (classical Gram-Schmidt against v_0..v_k: the full
//                                    reorthogonalisation, with ||w||^2 after it)
//   h2 = V^T w, w -= V h2           (a second pass, only when the first removed more than half
//                                    of ||w||^2: the criterion of Daniel, Gragg, Kaufman and
//                                    Stewart (1976); "twice is enough")
//   alpha_k = a + h_k (+ h2_k), beta_k = ||w||, v_{k+1} = w / beta_k
// The recurrence goes first so that the Gram-Schmidt pass acts on a vector already
// orthogonal to V up to the basis' own small loss of orthogonality: a pass applied to
// H v_k itself would carry that loss, times ||H v_k|| / beta_k, into v_{k+1} (large once
// the start vector is nearly an eigenvector, as in the later sweeps of DMRG).
// then the lowest eigenpair of the (n x n) tridiagonal matrix is found on the device
// (bisection + inverse iteration), and the Ritz vector x = sum_j s_j v_j is formed and
// normalised.  If beta_k falls below 1e-13 |alpha_k| the Krylov space is invariant: the
// remaining iterations become no-ops and the eigenproblem uses the k + 1 vectors built.
// Reductions are two-stage with a fixed order, so results are deterministic.
//
// One step's vector work was twelve launches whose kernels ran 3-16 us each; at m = 1024 (n =
// 406k) they took 120 us of a 216 us step.  In one kernel the phases meet at grid barriers (about
// 2 us each) and w stays in shared memory between them.
#include <cuda_runtime.h>

#include <cmath>

#include "barrier.cuh"
#include "internal.h"

using heff::fail;

namespace heff {
namespace {

constexpr int RT = 256;          // threads per reduction block
constexpr int RB = 456;          // reduction blocks (partial sums per vector): 3 per SM on 152 SMs
constexpr int VT = 8;            // vectors per multi-dot pass

constexpr int NVMAX = 128;       // basis vectors of one Lanczos workspace, at most

// State in the Lanczos workspace (doubles): [0] n_eff (as double), [1] active flag,
// [2] theta, [3] residual estimate, [8..8+NMAX) alpha, [8+NMAX..) beta; then s (NMAX), partial
// sums (RB blocks x (NVMAX + 2)), the grid barrier's words, and the vectors.
struct LzLayout {
    int nmax;
    int64_t n;
    size_t off_state, off_s, off_part, off_bar, off_V, bytes;
};

LzLayout lz_layout(int64_t n, int n_iter) {
    LzLayout l{};
    l.nmax = n_iter + 1;
    l.n = n;
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    size_t o = 0;
    l.off_state = o; o = al(o + sizeof(double) * (8 + 2 * (size_t)l.nmax));
    l.off_s = o;     o = al(o + sizeof(double) * (size_t)l.nmax);
    l.off_part = o;  o = al(o + sizeof(double) * (size_t)RB * (NVMAX + 2));
    l.off_bar = o;   o = al(o + 3 * sizeof(unsigned int));
    l.off_V = o;     o = al(o + sizeof(double) * (size_t)(l.nmax + 1) * (size_t)n);   // V + w
    l.bytes = o;
    return l;
}

struct Lz {
    double* state;   // n_eff, active, theta, resid, -, ..., alpha[nmax], beta[nmax]
    double* s;       // eigenvector of the tridiagonal matrix
    double* part;    // partial sums, [quantity][block]
    unsigned int* bar;   // grid barrier: counter, -, error
    double* V;       // (nmax) basis vectors, then w
    int64_t n;
    int nmax;
    __host__ __device__ double* w() const { return V + (int64_t)nmax * n; }
};

__device__ __forceinline__ double block_sum(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) sh[w] = v;
    __syncthreads();
    v = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    if (w == 0)
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    __syncthreads();
    return v;
}

// partial[b * VT + t] = sum over block b's chunk of V[j0 + t] . w, t < nv
__global__ void __launch_bounds__(RT) multidot_kernel(const double* __restrict__ V, const double* __restrict__ w,
                                                      int64_t n, int j0, int nv, double* __restrict__ part,
                                                      const double* __restrict__ state) {
    __shared__ double sh[RT / 32];
    if (state[1] == 0.0) return;
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t beg = (int64_t)blockIdx.x * chunk, end = beg + chunk < n ? beg + chunk : n;
    double acc[VT];
#pragma unroll
    for (int t = 0; t < VT; ++t) acc[t] = 0.0;
    // two elements per iteration: 2 (nv + 1) loads in flight per thread
    int64_t i = beg + threadIdx.x;
    for (; i + RT < end; i += 2 * RT) {
        const double w0 = w[i], w1 = w[i + RT];
        double v0[VT], v1[VT];
#pragma unroll
        for (int t = 0; t < VT; ++t) {
            v0[t] = t < nv ? V[(int64_t)(j0 + t) * n + i] : 0.0;
            v1[t] = t < nv ? V[(int64_t)(j0 + t) * n + i + RT] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < VT; ++t) acc[t] = fma(v1[t], w1, fma(v0[t], w0, acc[t]));
    }
    for (; i < end; i += RT) {
        const double wi = w[i];
#pragma unroll
        for (int t = 0; t < VT; ++t)
            if (t < nv) acc[t] = fma(V[(int64_t)(j0 + t) * n + i], wi, acc[t]);
    }
#pragma unroll
    for (int t = 0; t < VT; ++t) {
        if (t >= nv) break;                          // block-uniform
        double s = block_sum(acc[t], sh);
        if (threadIdx.x == 0) part[blockIdx.x * VT + t] = s;
    }
}

// out[j0 + t] = (accumulate ? out : 0) + sum_b partial[b * VT + t]
__global__ void finish_dots_kernel(const double* __restrict__ part, int nb, int j0, int nv, double* out,
                                   int accumulate, const double* __restrict__ state) {
    __shared__ double sh[RT / 32];
    if (state[1] == 0.0) return;
    for (int t = 0; t < nv; ++t) {
        double v = 0.0;
        for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[b * VT + t];
        v = block_sum(v, sh);
        if (threadIdx.x == 0) out[j0 + t] = accumulate ? out[j0 + t] + v : v;
    }
}

// y[i] = (beta_y * y[i]) + sign * sum_{j < nv} c[j] V[j][i]   (c from device memory)
__global__ void __launch_bounds__(RT) combine_kernel(const double* __restrict__ V, int64_t n, int nv,
                                                     const double* __restrict__ c, double sign, double beta_y,
                                                     double* __restrict__ y, const double* __restrict__ state) {
    __shared__ double cs[128];
    if (state[1] == 0.0) return;
    for (int j = threadIdx.x; j < nv; j += blockDim.x) cs[j] = c[j];
    __syncthreads();
    // two elements per iteration (their loads in flight together), then the remainder
    const int64_t stride = (int64_t)gridDim.x * RT;
    int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x;
    for (; i + stride < n; i += 2 * stride) {
        double a0 = 0.0, a1 = 0.0;
#pragma unroll 8
        for (int j = 0; j < nv; ++j) {
            a0 = fma(cs[j], V[(int64_t)j * n + i], a0);
            a1 = fma(cs[j], V[(int64_t)j * n + i + stride], a1);
        }
        y[i] = (beta_y == 0.0 ? 0.0 : beta_y * y[i]) + sign * a0;
        y[i + stride] = (beta_y == 0.0 ? 0.0 : beta_y * y[i + stride]) + sign * a1;
    }
    for (; i < n; i += stride) {
        double a = 0.0;
#pragma unroll 8
        for (int j = 0; j < nv; ++j) a = fma(cs[j], V[(int64_t)j * n + i], a);
        y[i] = (beta_y == 0.0 ? 0.0 : beta_y * y[i]) + sign * a;
    }
}

// sum of squares of x into part (stage 1)
__global__ void __launch_bounds__(RT) sumsq_kernel(const double* __restrict__ x, int64_t n, double* part) {
    __shared__ double sh[RT / 32];
    double a = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT)
        a = fma(x[i], x[i], a);
    a = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x * VT] = a;
}

// dst = src / sqrt(sum part); mode 0: initial vector (sets active and n_eff = 0); mode 2:
// plain; mode 3: plain, only while active
__global__ void __launch_bounds__(RT) normalize_kernel(const double* __restrict__ part, int nb,
                                                       const double* __restrict__ src, double* __restrict__ dst,
                                                       int64_t n, double* state, int mode) {
    __shared__ double sh[RT / 32];
    __shared__ double nrm;
    if (mode == 3 && state[1] == 0.0) return;
    double v = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[b * VT];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) nrm = sqrt(v);
    __syncthreads();
    const double r = nrm;
    if (mode == 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        state[0] = 0.0;
        state[1] = r > 0.0 ? 1.0 : 0.0;
    }
    if (!(r > 0.0)) return;
    const double inv = 1.0 / r;
    for (int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT) dst[i] = src[i] * inv;
}

// ---------------------------------------------------------------- Lanczos step
// The cooperative kernels run at most one block of LT threads per SM; block b owns the
// elements [b chunk, (b + 1) chunk) of every vector, and its piece of w lives in shared memory
// when it fits (LW_MAX doubles), else in place.
constexpr int LTS = 512, LTL = 1024;     // threads of a block: short and long vectors
constexpr int LW_MAX = 25600;
// elements per block from which it has LTL threads: twice the loads in flight (m = 4096, 39k elements a block,
// 30 steps: 34.5 ms with 512 threads, 28.3 with 1024; m = 1024, 2.7k elements, 20 steps: 2.376 and
// 2.360), while fewer elements leave the added warps only reductions (m = 48, 20 steps: 0.70 and 0.76)
constexpr int LT_WIDE = 1280;

struct LzArgs {
    Lz z;
    const double* x0;       // start vector (lz_start)
    double* x_out;          // Ritz vector (lz_finish)
    double* result;
    int64_t chunk;
    int k, w_shared;
    int* apply_err;         // the matvec workspace's error flag, raised with the barrier's
};

struct LzBlock {
    double* h;              // [NVMAX + 1] sums over all blocks, shared memory
    double* red;            // [2 * LTL / 32]
    int64_t beg;
    int len;
};

// Sum over the block, for thread 0 (a warp's FP64 addition takes 16 cycles of the SM's FP64 unit:
// only one warp adds the warps' sums).
template <int LT>
__device__ __forceinline__ double lz_block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        v = threadIdx.x < LT / 32 ? red[threadIdx.x] : 0.0;
        for (int o = LT / 64; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    __syncthreads();
    return v;
}

__device__ __forceinline__ bool lz_barrier(const LzArgs& a) {
    if (gridDim.x == 1) {
        __syncthreads();
        return true;
    }
    const bool ok = grid_barrier(a.z.bar, gridDim.x, reinterpret_cast<int*>(a.z.bar + 2));
    if (!ok && threadIdx.x == 0) atomicExch(a.apply_err, 1);
    return ok;
}

// out[j] = sum over the blocks of part[j0 + j][block], j < nv: one warp per quantity, every block
// the same sums in the same order.
template <int LT>
__device__ __forceinline__ void lz_gather(const LzArgs& a, int j0, int nv, double* out) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int j = warp; j < nv; j += (LT / 32)) {
        double v = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) v += __ldcg(a.z.part + (int64_t)(j0 + j) * RB + b);
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) out[j] = v;
    }
    __syncthreads();
}

// part[j][this block] = V_j . w over the block's elements, j < nv, and part[nv] = w . w.  A warp
// takes one vector over one of `seg` pieces of the chunk (all warps busy also for few vectors).
template <int LT>
__device__ __forceinline__ void lz_dots(const LzArgs& a, const LzBlock& b, const double* w, int nv) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = nv + 1, seg = q >= (LT / 32) ? 1 : (LT / 32) / q;
    const int piece = ((b.len + seg - 1) / seg + 31) & ~31;
    for (int item = warp; item < q * seg; item += (LT / 32)) {
        const int j = item / seg, s = item % seg;
        const double* v = j < nv ? a.z.V + (int64_t)j * a.z.n + b.beg : w;
        const int end = (s + 1) * piece < b.len ? (s + 1) * piece : b.len;
        double acc = 0.0;
        int i = s * piece + lane;
        for (; i + 7 * 32 < end; i += 8 * 32) {
            double u[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) u[e] = v[i + 32 * e];
#pragma unroll
            for (int e = 0; e < 8; ++e) acc = fma(u[e], w[i + 32 * e], acc);
        }
        for (; i < end; i += 32) acc = fma(v[i], w[i], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) {
            if (seg == 1) a.z.part[(int64_t)j * RB + blockIdx.x] = acc;
            else b.red[item] = acc;
        }
    }
    if (seg > 1) {
        __syncthreads();
        if ((int)threadIdx.x < q) {
            double s = 0.0;
            for (int e = 0; e < seg; ++e) s += b.red[threadIdx.x * seg + e];
            a.z.part[(int64_t)threadIdx.x * RB + blockIdx.x] = s;
        }
    }
}

// w -= sum_{j < nv} h_j V_j over the block's elements; returns the block's new w . w
template <int LT>
__device__ __forceinline__ double lz_subtract(const LzArgs& a, const LzBlock& b, double* w, int nv) {
    double sq = 0.0;
    for (int i = threadIdx.x; i < b.len; i += LT) {
        const double* v = a.z.V + b.beg + i;
        double s = 0.0;
#pragma unroll 8
        for (int j = 0; j < nv; ++j) s = fma(b.h[j], v[(int64_t)j * a.z.n], s);
        const double y = w[i] - s;
        w[i] = y;
        sq = fma(y, y, sq);
    }
    return lz_block_sum<LT>(sq, b.red);
}

__device__ __forceinline__ LzBlock lz_block(const LzArgs& a, double* h, double* red) {
    LzBlock b{h, red, (int64_t)blockIdx.x * a.chunk, 0};
    const int64_t left = a.z.n - b.beg;
    b.len = (int)(left < a.chunk ? (left > 0 ? left : 0) : a.chunk);
    return b;
}

// One Lanczos step on w = H v_k (in the workspace): recurrence, one or two Gram-Schmidt passes,
// alpha_k, beta_k and v_{k+1}.
template <int LT>
__global__ void __launch_bounds__(LT, 1) lz_step_kernel(LzArgs a) {
    extern __shared__ double dyn[];
    __shared__ double h[NVMAX + 1], red[2 * LTL / 32];
    double* state = a.z.state;
    if (state[1] == 0.0) return;                       // the same for every block: no barrier is left open
    const LzBlock b = lz_block(a, h, red);
    const int k = a.k, nmax = a.z.nmax;
    double* wg = a.z.w() + b.beg;
    double* w = a.w_shared ? dyn : wg;
    const double* vk = a.z.V + (int64_t)k * a.z.n + b.beg;
    const double* vp = vk - a.z.n;
    const double beta = k > 0 ? state[8 + nmax + k - 1] : 0.0;
    // x = w - beta v_{k-1}, a = v_k . x
    double acc = 0.0;
    for (int i = threadIdx.x; i < b.len; i += LT) {
        const double x = k > 0 ? wg[i] - beta * vp[i] : wg[i];
        w[i] = x;
        acc = fma(vk[i], x, acc);
    }
    // slots NVMAX (||w||^2 after a pass) and NVMAX + 1 (a) are their own: no block still reads a
    // slot that another writes, with one barrier per sum
    acc = lz_block_sum<LT>(acc, red);
    if (threadIdx.x == 0) a.z.part[(int64_t)(NVMAX + 1) * RB + blockIdx.x] = acc;
    if (!lz_barrier(a)) return;
    lz_gather<LT>(a, NVMAX + 1, 1, h);
    double alpha = h[0];
    for (int i = threadIdx.x; i < b.len; i += LT) w[i] -= alpha * vk[i];
    __syncthreads();
    // Gram-Schmidt against v_0 .. v_k; again when less than half of ||w||^2 is left
    double sq = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        lz_dots<LT>(a, b, w, k + 1);
        if (!lz_barrier(a)) return;
        lz_gather<LT>(a, 0, k + 2, h);
        const double before = h[k + 1];
        alpha += h[k];
        const double mine = lz_subtract<LT>(a, b, w, k + 1);
        if (threadIdx.x == 0) a.z.part[(int64_t)NVMAX * RB + blockIdx.x] = mine;
        if (!lz_barrier(a)) return;
        lz_gather<LT>(a, NVMAX, 1, h);
        sq = h[0];
        __syncthreads();
        if (!(sq < 0.5 * before)) break;
    }
    const double r = sqrt(sq);
    // an invariant Krylov space (beta_k <= 1e-13 |alpha_k|) ends the iteration
    const bool go = r > 1e-13 * fabs(alpha) && r > 1e-300;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state[8 + k] = alpha;
        state[8 + nmax + k] = r;
        state[0] = (double)(k + 1);
        if (!go) state[1] = 0.0;
    }
    if (!go) return;
    const double inv = 1.0 / r;
    double* vn = a.z.V + (int64_t)(k + 1) * a.z.n + b.beg;
    for (int i = threadIdx.x; i < b.len; i += LT) vn[i] = w[i] * inv;
}

// v_0 = x0 / ||x0||; a zero x0 leaves the iteration inactive
template <int LT>
__global__ void __launch_bounds__(LT, 1) lz_start_kernel(LzArgs a) {
    __shared__ double h[NVMAX + 1], red[2 * LTL / 32];
    const LzBlock b = lz_block(a, h, red);
    const double* x = a.x0 + b.beg;
    double acc = 0.0;
    for (int i = threadIdx.x; i < b.len; i += LT) acc = fma(x[i], x[i], acc);
    acc = lz_block_sum<LT>(acc, red);
    if (threadIdx.x == 0) a.z.part[blockIdx.x] = acc;
    if (!lz_barrier(a)) return;
    lz_gather<LT>(a, 0, 1, h);
    const double r = sqrt(h[0]);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.z.state[0] = 0.0;
        a.z.state[1] = r > 0.0 ? 1.0 : 0.0;
    }
    if (!(r > 0.0)) return;
    const double inv = 1.0 / r;
    double* v = a.z.V + b.beg;
    for (int i = threadIdx.x; i < b.len; i += LT) v[i] = x[i] * inv;
}

// Lowest eigenpair of the n x n tridiagonal matrix T (diagonal al, off-diagonal be, shared
// memory), in FP64 by one warp: the eigenvalue by multisection on the Sturm sequence (the leading
// principal minors p_i of T - x I change sign when an eigenvalue lies below x), the lanes at 32
// points of the bracket; the eigenvector by inverse iteration, T - theta I factored once by Gaussian
// elimination with partial pivoting.  Chains of FP64 operations set the time, and every warp that
// joins slows the others (a warp's FP64 instruction holds the SM's FP64 unit for 16 cycles): the
// minors need three multiply-adds a row and no division (rescaled when they leave 2^+-300), and
// the factors are kept over the iterations (20 x 20: 265 us with divisions and arrays in global
// memory, 30 us now).  Returns theta to lane 0; s gets the eigenvector; work: 5 arrays of NVMAX.
__device__ double lz_tridiag(const double* al, const double* be, int n, double* s, double* work) {
    const int lane = threadIdx.x;
    double *f = work, *dd = work + NVMAX, *du = work + 2 * NVMAX, *du2 = work + 3 * NVMAX, *b2 = work + 4 * NVMAX;
    double lo = al[0], hi = al[0];
    for (int i = lane; i < n; i += 32) {
        const double r = (i > 0 ? fabs(be[i - 1]) : 0.0) + (i + 1 < n ? fabs(be[i]) : 0.0);
        lo = fmin(lo, al[i] - r);
        hi = fmax(hi, al[i] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const double scale = fmax(fabs(lo), fabs(hi)) + 1e-300;
    const double inv = 1.0 / scale;
    // squares of the scaled off-diagonals; b2[0] = 0
    for (int i = lane; i < n; i += 32) {
        const double e = i > 0 ? be[i - 1] * inv : 0.0;
        b2[i] = e * e;
    }
    __syncwarp();
    // whether an eigenvalue lies below x.  The scaled entries are at most 1 (x at most 1): a row
    // changes the minors by at most a factor of 4
    auto below = [&](double x) {
        double p0 = 0.0, p1 = 1.0;
        bool neg = false;
        for (int i = 0; i < n; ++i) {
            const double p2 = fma((al[i] - x) * inv, p1, -(b2[i] * p0));
            // a vanishing minor counts with the sign opposite to its predecessor's
            neg = neg || p2 == 0.0 || (__double2hiint(p2) ^ __double2hiint(p1)) < 0;
            p0 = p1;
            p1 = p2;
            const int e = (__double2hiint(p1) >> 20) & 0x7ff;
            if (e < 1023 - 300 || e > 1023 + 300) {
                const int g = 1023 - e < 500 ? 1023 - e : 500;      // both times 2^g
                const double m = __hiloint2double((g + 1023) << 20, 0);
                p0 *= m;
                p1 *= m;
            }
        }
        return neg;
    };
    // the lowest eigenvalue stays in (lo, hi]
    for (int it = 0; it < 60 && hi - lo > 4e-16 * scale; ++it) {
        const double step = (hi - lo) / 33.0;
        const double x = lane == 31 ? hi - 0.5 * step : lo + (lane + 1) * step;
        const unsigned m = __ballot_sync(0xffffffffu, below(x));
        const int k = m ? __ffs(m) - 1 : 32;          // first point with an eigenvalue below it
        const double xk = __shfl_sync(0xffffffffu, x, k < 32 ? k : 31);
        const double xk1 = __shfl_sync(0xffffffffu, x, k > 0 ? (k < 32 ? k - 1 : 31) : 0);
        if (k < 32) hi = xk;
        if (k > 0) lo = xk1;
    }
    const double theta = 0.5 * (lo + hi);
    // P (T - theta I) = L U: multipliers and row exchanges, U with two super-diagonals.  A pivot
    // below tiny (theta is an eigenvalue to rounding, so one pivot is ~0) is replaced by +-tiny
    __shared__ unsigned char swap[NVMAX];
    const double tiny = 1e-15 * scale;
    if (lane == 0) {
        double d = al[0] - theta, u = n > 1 ? be[0] : 0.0;        // row i of the elimination
        for (int i = 0; i + 1 < n; ++i) {
            const double l = be[i], dn = al[i + 1] - theta, un = i + 2 < n ? be[i + 1] : 0.0;
            if (fabs(d) >= fabs(l)) {                 // no exchange
                if (fabs(d) < tiny) d = d < 0.0 ? -tiny : tiny;
                const double m = l / d;
                f[i] = m; swap[i] = 0;
                dd[i] = d; du[i] = u; du2[i] = 0.0;
                d = dn - m * u;
                u = un;
            } else {                                  // rows i and i + 1 exchanged
                const double m = d / l;
                f[i] = m; swap[i] = 1;
                dd[i] = l; du[i] = dn; du2[i] = un;
                d = u - m * dn;
                u = -m * un;
            }
        }
        if (fabs(d) < tiny) d = d < 0.0 ? -tiny : tiny;
        dd[n - 1] = d;
        du[n - 1] = du2[n - 1] = 0.0;
    }
    __syncwarp();
    const double s0 = 1.0 / sqrt((double)n);
    for (int i = lane; i < n; i += 32) {
        dd[i] = 1.0 / dd[i];
        s[i] = s0;
    }
    __syncwarp();
    for (int iter = 0; iter < 4; ++iter) {
        if (lane == 0) {
            double y = s[0];
            for (int i = 0; i + 1 < n; ++i) {
                const double z = s[i + 1];
                s[i] = swap[i] ? z : y;
                y = swap[i] ? y - f[i] * z : z - f[i] * y;
            }
            s[n - 1] = y;
            double x1 = 0.0, x2 = 0.0;
            for (int i = n - 1; i >= 0; --i) {
                const double x = (s[i] - du[i] * x1 - du2[i] * x2) * dd[i];
                s[i] = x;
                x2 = x1;
                x1 = x;
            }
        }
        __syncwarp();
        // scale by the largest entry, then by the norm: the large solution does not overflow
        double mx = 0.0, nr = 0.0;
        for (int i = lane; i < n; i += 32) mx = fmax(mx, fabs(s[i]));
        for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        if (!(mx > 0.0) || !isfinite(mx)) {           // cannot happen with the guards; keep e_0
            for (int i = lane; i < n; i += 32) s[i] = i == 0 ? 1.0 : 0.0;
            __syncwarp();
            break;
        }
        const double im = 1.0 / mx;
        for (int i = lane; i < n; i += 32) nr = fma(s[i] * im, s[i] * im, nr);
        for (int o = 16; o > 0; o >>= 1) nr += __shfl_xor_sync(0xffffffffu, nr, o);
        nr = im / sqrt(nr);
        for (int i = lane; i < n; i += 32) s[i] *= nr;
        __syncwarp();
    }
    if (lane == 0) {
        // fix the sign (largest component positive) for reproducible Ritz vectors
        int im = 0;
        for (int i = 1; i < n; ++i) if (fabs(s[i]) > fabs(s[im])) im = i;
        if (s[im] < 0)
            for (int i = 0; i < n; ++i) s[i] = -s[i];
    }
    __syncwarp();
    return theta;
}

// The lowest Ritz pair: theta, the residual estimate |beta_{n-1} s_{n-1}|, x = V s normalised, and
// the result record.
template <int LT>
__global__ void __launch_bounds__(LT, 1) lz_finish_kernel(LzArgs a) {
    __shared__ double h[NVMAX + 1], red[2 * LTL / 32], al[NVMAX], be[NVMAX], work[5 * NVMAX];
    const LzBlock b = lz_block(a, h, red);
    double* state = a.z.state;
    const int n = (int)state[0], nmax = a.z.nmax;
    if (blockIdx.x == 0) {
        if (n > 0) {
            for (int i = threadIdx.x; i < n; i += LT) {
                al[i] = state[8 + i];
                be[i] = state[8 + nmax + i];
            }
            __syncthreads();
            if (threadIdx.x < 32) {
                const double theta = lz_tridiag(al, be, n, h, work);
                for (int i = threadIdx.x; i < n; i += 32) a.z.s[i] = h[i];
                if (threadIdx.x == 0) {
                    state[2] = theta;
                    state[3] = fabs(be[n - 1] * h[n - 1]);
                }
            }
        } else if (threadIdx.x == 0) {                // a zero start vector: no Krylov space
            state[2] = 0.0;
            state[3] = 0.0;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < 3 + 2 * nmax; i += LT)
            a.result[i] = i < 2 ? state[2 + i] : (i == 2 ? (double)n : state[8 + i - 3]);
    }
    if (!lz_barrier(a)) return;
    for (int j = threadIdx.x; j < n; j += LT) h[j] = __ldcg(a.z.s + j);
    __syncthreads();
    double* x = a.x_out + b.beg;
    double acc = 0.0;
    for (int i = threadIdx.x; i < b.len; i += LT) {
        const double* v = a.z.V + b.beg + i;
        double s = 0.0;
#pragma unroll 8
        for (int j = 0; j < n; ++j) s = fma(h[j], v[(int64_t)j * a.z.n], s);
        x[i] = s;
        acc = fma(s, s, acc);
    }
    acc = lz_block_sum<LT>(acc, red);
    if (threadIdx.x == 0) a.z.part[blockIdx.x] = acc;
    if (!lz_barrier(a)) return;
    lz_gather<LT>(a, 0, 1, h);
    const double r = sqrt(h[0]);
    if (!(r > 0.0)) return;
    const double inv = 1.0 / r;
    for (int i = threadIdx.x; i < b.len; i += LT) x[i] *= inv;
}

// ---------------------------------------------------------------- Davidson (Algorithm 1)
// State (doubles): [0] vectors in use, [1] active, [2] lambda, [3] ||q||, [4] ||q|| before
// the Gram-Schmidt passes, [5] tol.

// M[i][j] = M[j][i] = h[j], j <= i
__global__ void dav_set_m_kernel(double* M, const double* h, int i, int maxv, const double* state) {
    if (state[1] == 0.0) return;
    for (int j = threadIdx.x; j <= i; j += blockDim.x) {
        M[i * maxv + j] = h[j];
        M[j * maxv + i] = h[j];
    }
}

// Lowest eigenpair of the leading m x m block of the symmetric M (one thread, cyclic
// Jacobi rotations in FP64 until the off-diagonal mass is below 1e-30 of the total):
// lambda -> state[2], eigenvector (largest component positive) -> s.
__global__ void dav_eig_kernel(const double* M, double* E, double* s, double* state, int m, int maxv) {
    if (threadIdx.x != 0 || blockIdx.x != 0 || state[1] == 0.0) return;
    double* A = E;                    // m x m working copy
    double* Q = E + maxv * maxv;      // accumulated rotations
    for (int r = 0; r < m; ++r)
        for (int c = 0; c < m; ++c) {
            A[r * m + c] = M[r * maxv + c];
            Q[r * m + c] = r == c ? 1.0 : 0.0;
        }
    for (int sweep = 0; sweep < 60; ++sweep) {
        double off = 0.0, tot = 0.0;
        for (int r = 0; r < m; ++r)
            for (int c = 0; c < m; ++c) {
                const double v = A[r * m + c] * A[r * m + c];
                tot += v;
                if (r != c) off += v;
            }
        if (!(off > 1e-30 * tot)) break;
        for (int p = 0; p < m; ++p)
            for (int q = p + 1; q < m; ++q) {
                const double apq = A[p * m + q];
                if (apq == 0.0) continue;
                const double zeta = (A[q * m + q] - A[p * m + p]) / (2.0 * apq);
                const double t = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                const double c = 1.0 / sqrt(1.0 + t * t), sn = c * t;
                for (int k = 0; k < m; ++k) {           // columns p, q
                    const double akp = A[k * m + p], akq = A[k * m + q];
                    A[k * m + p] = c * akp - sn * akq;
                    A[k * m + q] = sn * akp + c * akq;
                }
                for (int k = 0; k < m; ++k) {           // rows p, q
                    const double apk = A[p * m + k], aqk = A[q * m + k];
                    A[p * m + k] = c * apk - sn * aqk;
                    A[q * m + k] = sn * apk + c * aqk;
                }
                for (int k = 0; k < m; ++k) {
                    const double qkp = Q[k * m + p], qkq = Q[k * m + q];
                    Q[k * m + p] = c * qkp - sn * qkq;
                    Q[k * m + q] = sn * qkp + c * qkq;
                }
            }
    }
    int lo = 0;
    for (int r = 1; r < m; ++r) if (A[r * m + r] < A[lo * m + lo]) lo = r;
    int im = 0;
    for (int r = 1; r < m; ++r) if (fabs(Q[r * m + lo]) > fabs(Q[im * m + lo])) im = r;
    const double sg = Q[im * m + lo] < 0.0 ? -1.0 : 1.0;
    for (int r = 0; r < maxv; ++r) s[r] = r < m ? sg * Q[r * m + lo] : 0.0;
    state[2] = A[lo * m + lo];
    state[0] = (double)m;
}

// q -= lambda x
__global__ void __launch_bounds__(RT) dav_shift_kernel(double* __restrict__ q, const double* __restrict__ x,
                                                       int64_t n, const double* __restrict__ state) {
    if (state[1] == 0.0) return;
    const double lam = state[2];
    for (int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT) q[i] -= lam * x[i];
}

// ||q|| -> state[3]; stop (active = 0) when ||q|| < tol max(1, |lambda|) or the subspace is
// full, else remember ||q|| in state[4]
__global__ void dav_check_kernel(const double* __restrict__ part, int nb, double* state, int last) {
    __shared__ double sh[RT / 32];
    if (state[1] == 0.0) return;
    double v = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[b * VT];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) {
        const double r = sqrt(v);
        state[3] = r;
        state[4] = r;
        if (last || !(r >= state[5] * fmax(1.0, fabs(state[2])))) state[1] = 0.0;
    }
}

// Randomisation (Algorithm 1's remedy for a failed reorthogonalisation): if Gram-Schmidt
// left less than 1e-12 of ||q||, replace q by the caller's random vector
__global__ void __launch_bounds__(RT) dav_random_kernel(const double* __restrict__ part, int nb,
                                                        double* __restrict__ q, const double* __restrict__ rnd,
                                                        int64_t n, const double* __restrict__ state) {
    __shared__ double sh[RT / 32];
    __shared__ int swap;
    if (state[1] == 0.0) return;
    double v = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[b * VT];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) swap = !(sqrt(v) >= 1e-12 * state[4]);
    __syncthreads();
    if (!swap) return;
    for (int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT) q[i] = rnd[i];
}

int grid_for(int64_t n) {
    int64_t g = (n + RT - 1) / RT;
    return (int)(g < 4096 ? (g > 0 ? g : 1) : 4096);
}

}  // namespace
}  // namespace heff

using namespace heff;

extern "C" int heff_lanczos_workspace_size(const heff_plan* plan, int32_t n_iter, size_t* bytes) {
    clear_error();
    if (!plan || !bytes || n_iter < 1 || n_iter > 126)
        return fail(HEFF_ERR_INVALID_ARG, "heff_lanczos_workspace_size: bad arguments (n_iter 1..126)");
    *bytes = lz_layout(plan->nelem_x, n_iter).bytes;
    return HEFF_OK;
}

namespace heff {
namespace {

Lz lz_view(const LzLayout& lay, void* lz_ws, int64_t n) {
    char* base = static_cast<char*>(lz_ws);
    return Lz{reinterpret_cast<double*>(base + lay.off_state), reinterpret_cast<double*>(base + lay.off_s),
              reinterpret_cast<double*>(base + lay.off_part), reinterpret_cast<unsigned int*>(base + lay.off_bar),
              reinterpret_cast<double*>(base + lay.off_V), n, lay.nmax};
}

// n_iter Lanczos steps from x0 on operators already prepared in apply_ws; x0 may alias x_out
// (it is only read into the first basis vector).
int lanczos_core(heff_plan* plan, const double* x0, int32_t n_iter, double* x_out, double* result,
                 void* apply_ws, size_t apply_ws_bytes, const Lz& z, cudaStream_t st) {
    const int64_t n = z.n;
    // a block per SM, each with at least 1024 elements (two per thread)
    int64_t blocks = (n + 1023) / 1024;
    const int most = plan->num_sms < RB ? plan->num_sms : RB;
    if (blocks > most) blocks = most;
    LzArgs a{z, x0, x_out, result, (n + blocks - 1) / blocks, 0, 0,
             reinterpret_cast<int*>(static_cast<char*>(apply_ws) + plan->off_flags)};
    a.w_shared = a.chunk <= LW_MAX;
    const size_t smem = a.w_shared ? (size_t)a.chunk * sizeof(double) : 0;
    const bool wide = a.chunk >= LT_WIDE;
    const unsigned threads = wide ? LTL : LTS;
    static PerDevice done[2];
    if (int rc = raise_smem_limit(done[wide], wide ? (const void*)lz_step_kernel<LTL> : (const void*)lz_step_kernel<LTS>,
                                  LW_MAX * (int)sizeof(double)))
        return rc;
    cudaError_t e = cudaMemsetAsync(z.bar, 0, 3 * sizeof(unsigned int), st);
    void* args[] = {&a};
    auto launch = [&](const void* kernel, size_t bytes) {
        if (e == cudaSuccess)
            e = cudaLaunchCooperativeKernel(kernel, dim3((unsigned)blocks), dim3(threads), args, bytes, st);
        count_launches(1);
    };
    launch((const void*)(wide ? lz_start_kernel<LTL> : lz_start_kernel<LTS>), 0);
    for (int k = 0; k < n_iter && e == cudaSuccess; ++k) {
        // w = H v_k (skipped work is harmless after breakdown: the result is not used)
        int rc = heff_apply_prepared(plan, z.V + (int64_t)k * n, z.w(), apply_ws, apply_ws_bytes, st);
        if (rc) return rc;
        a.k = k;
        launch((const void*)(wide ? lz_step_kernel<LTL> : lz_step_kernel<LTS>), smem);
    }
    launch((const void*)(wide ? lz_finish_kernel<LTL> : lz_finish_kernel<LTS>), 0);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "heff_lanczos: %s", cudaGetErrorString(e));
    return HEFF_OK;
}

}  // namespace
}  // namespace heff

extern "C" int heff_lanczos(heff_plan* plan, const void* L, const void* W1, const void* W2, const void* R,
                            const double* x0, int32_t n_iter, double* x_out, double* result,
                            void* apply_ws, size_t apply_ws_bytes, void* lz_ws, size_t lz_ws_bytes,
                            void* stream) {
    clear_error();
    if (!plan || !L || !W1 || !W2 || !R || !x0 || !x_out || !result || !lz_ws)
        return fail(HEFF_ERR_INVALID_ARG, "heff_lanczos: null argument");
    if (plan->opts.io_dtype != HEFF_DTYPE_F64)
        return fail(HEFF_ERR_UNSUPPORTED, "heff_lanczos needs a plan with HEFF_DTYPE_F64 tensors");
    if (n_iter < 1 || n_iter > 126) return fail(HEFF_ERR_INVALID_ARG, "n_iter must be 1..126");
    if (plan->nelem_x == 0) return fail(HEFF_ERR_INVALID_ARG, "heff_lanczos: the two-site space is empty");
    const LzLayout lay = lz_layout(plan->nelem_x, n_iter);
    if (lz_ws_bytes < lay.bytes || reinterpret_cast<uintptr_t>(lz_ws) % 256)
        return fail(HEFF_ERR_WORKSPACE, "Lanczos workspace of %zu bytes, needs %zu (256-byte aligned)",
                    lz_ws_bytes, lay.bytes);
    int rc = heff_prepare(plan, L, W1, W2, R, apply_ws, apply_ws_bytes, stream);
    if (rc) return rc;
    return lanczos_core(plan, x0, n_iter, x_out, result, apply_ws, apply_ws_bytes,
                        lz_view(lay, lz_ws, plan->nelem_x), static_cast<cudaStream_t>(stream));
}

// ---------------------------------------------------------------- ground state to a tolerance
namespace heff {
namespace {

// part[b] = sum over block b's chunk of x[i] * y[i]  (mode 0), or of (y[i] - E x[i])^2 with
// E = *e_dev (mode 1); two-stage with a fixed order, like the Lanczos reductions
__global__ void __launch_bounds__(RT) rq_part_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                                     int64_t n, const double* __restrict__ e_dev, int mode,
                                                     double* __restrict__ part) {
    __shared__ double sh[RT / 32];
    const double E = mode ? *e_dev : 0.0;
    double a = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * RT + threadIdx.x; i < n; i += (int64_t)gridDim.x * RT) {
        if (mode == 0) {
            a = fma(x[i], y[i], a);
        } else {
            const double r = y[i] - E * x[i];
            a = fma(r, r, a);
        }
    }
    a = block_sum(a, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = a;
}

__global__ void rq_finish_kernel(const double* __restrict__ part, int nb, double* out) {
    __shared__ double sh[RT / 32];
    double v = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) v += part[b];
    v = block_sum(v, sh);
    if (threadIdx.x == 0) *out = v;
}

// ground-state workspace: the Lanczos workspace, then the cycle's result and 4 scalars
size_t gs_result_off(const LzLayout& lay) { return lay.bytes; }
size_t gs_bytes(const LzLayout& lay) {
    return lay.bytes + (sizeof(double) * (3 + 2 * (size_t)lay.nmax + 8) + 255) / 256 * 256;
}

}  // namespace
}  // namespace heff

extern "C" int heff_ground_state_workspace_size(const heff_plan* plan, int32_t n_iter, size_t* bytes) {
    clear_error();
    if (!plan || !bytes || n_iter < 1 || n_iter > 126)
        return fail(HEFF_ERR_INVALID_ARG, "heff_ground_state_workspace_size: bad arguments (n_iter 1..126)");
    *bytes = gs_bytes(lz_layout(plan->nelem_x, n_iter));
    return HEFF_OK;
}

extern "C" int heff_ground_state(heff_plan* plan, heff_plan* plan64, const void* L, const void* W1,
                                 const void* W2, const void* R, const double* x0, int32_t n_iter,
                                 int32_t max_cycles, double tol, double* x_out, double* result,
                                 void* apply_ws, size_t apply_ws_bytes, void* apply_ws64, size_t apply_ws64_bytes,
                                 void* gs_ws, size_t gs_ws_bytes, void* stream) {
    clear_error();
    if (!plan || !L || !W1 || !W2 || !R || !x0 || !x_out || !result || !gs_ws)
        return fail(HEFF_ERR_INVALID_ARG, "heff_ground_state: null argument");
    if (plan->opts.io_dtype != HEFF_DTYPE_F64)
        return fail(HEFF_ERR_UNSUPPORTED, "heff_ground_state needs a plan with HEFF_DTYPE_F64 tensors");
    if (n_iter < 1 || n_iter > 126 || max_cycles < 1 || !(tol >= 0.0))
        return fail(HEFF_ERR_INVALID_ARG, "heff_ground_state: n_iter 1..126, max_cycles >= 1, tol >= 0");
    if (plan->nelem_x == 0) return fail(HEFF_ERR_INVALID_ARG, "heff_ground_state: the two-site space is empty");
    // the FP64 Rayleigh quotient: plan64, or the plan itself when it is the FP64 path
    heff_plan* p64 = plan64 ? plan64 : (plan->opts.precision == HEFF_PREC_FP64 ? plan : nullptr);
    void* ws64 = plan64 ? apply_ws64 : apply_ws;
    const size_t ws64_bytes = plan64 ? apply_ws64_bytes : apply_ws_bytes;
    if (p64) {
        if (p64->opts.precision != HEFF_PREC_FP64 || p64->opts.io_dtype != HEFF_DTYPE_F64 ||
            p64->nelem_x != plan->nelem_x)
            return fail(HEFF_ERR_INVALID_ARG, "heff_ground_state: plan64 must be an FP64 plan of the same layouts");
        if (plan64 && !apply_ws64) return fail(HEFF_ERR_INVALID_ARG, "heff_ground_state: null apply_ws64");
    }
    const LzLayout lay = lz_layout(plan->nelem_x, n_iter);
    if (gs_ws_bytes < gs_bytes(lay) || reinterpret_cast<uintptr_t>(gs_ws) % 256)
        return fail(HEFF_ERR_WORKSPACE, "ground-state workspace of %zu bytes, needs %zu (256-byte aligned)",
                    gs_ws_bytes, gs_bytes(lay));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const Lz z = lz_view(lay, gs_ws, plan->nelem_x);
    double* res = reinterpret_cast<double*>(static_cast<char*>(gs_ws) + gs_result_off(lay));
    double* scal = res + 3 + 2 * lay.nmax;          // [0] x.y, [1] |y - E x|^2
    int rc = heff_prepare(plan, L, W1, W2, R, apply_ws, apply_ws_bytes, stream);
    if (rc) return rc;
    double theta = 0.0, est = 0.0;
    int cycles = 0;
    const double* start = x0;
    for (; cycles < max_cycles;) {
        if ((rc = lanczos_core(plan, start, n_iter, x_out, res, apply_ws, apply_ws_bytes, z, st))) return rc;
        ++cycles;
        start = x_out;                                // the next cycle restarts from the Ritz vector
        double h[2];
        cudaError_t e = cudaMemcpyAsync(h, res, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "heff_ground_state: %s", cudaGetErrorString(e));
        theta = h[0];
        est = h[1] / (fabs(theta) > 0.0 ? fabs(theta) : 1.0);
        if (!(est > tol)) break;
    }
    result[0] = theta;
    result[1] = theta;
    result[2] = est;
    result[3] = cycles;
    result[4] = (double)cycles * n_iter;
    result[5] = -1.0;
    if (p64) {
        // E = <x|K|x> (x is normalised) with an FP64 apply, and ||K x - E x|| / |E|
        if (p64 != plan && (rc = heff_prepare(p64, L, W1, W2, R, ws64, ws64_bytes, stream))) return rc;
        double* y = z.w();
        if ((rc = heff_apply_prepared(p64, x_out, y, ws64, ws64_bytes, stream))) return rc;
        const int64_t n = z.n;
        rq_part_kernel<<<RB, RT, 0, st>>>(x_out, y, n, nullptr, 0, z.part);
        rq_finish_kernel<<<1, RT, 0, st>>>(z.part, RB, scal);
        rq_part_kernel<<<RB, RT, 0, st>>>(x_out, y, n, scal, 1, z.part);
        rq_finish_kernel<<<1, RT, 0, st>>>(z.part, RB, scal + 1);
        count_launches(4);
        double h[2];
        cudaError_t e = cudaMemcpyAsync(h, scal, sizeof(h), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "heff_ground_state: %s", cudaGetErrorString(e));
        result[0] = h[0];
        result[5] = sqrt(h[1]) / (fabs(h[0]) > 0.0 ? fabs(h[0]) : 1.0);
    }
    return HEFF_OK;
}

// ---------------------------------------------------------------- Davidson host side
namespace heff {
namespace {

struct DavLayout {
    int maxv;
    size_t off_state, off_M, off_E, off_s, off_h, off_part, off_V, off_VA, off_q, bytes;
};

DavLayout dav_layout(int64_t n, int maxv) {
    DavLayout l{};
    l.maxv = maxv;
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    size_t o = 0;
    l.off_state = o; o = al(o + sizeof(double) * 16);
    l.off_M = o;     o = al(o + sizeof(double) * (size_t)maxv * maxv);
    l.off_E = o;     o = al(o + sizeof(double) * 2 * (size_t)maxv * maxv);
    l.off_s = o;     o = al(o + sizeof(double) * (size_t)maxv);
    l.off_h = o;     o = al(o + sizeof(double) * (size_t)maxv);
    l.off_part = o;  o = al(o + sizeof(double) * (size_t)RB * VT);
    l.off_V = o;     o = al(o + sizeof(double) * (size_t)maxv * (size_t)n);
    l.off_VA = o;    o = al(o + sizeof(double) * (size_t)maxv * (size_t)n);
    l.off_q = o;     o = al(o + sizeof(double) * (size_t)n);
    l.bytes = o;
    return l;
}

__global__ void dav_init_state_kernel(double* state, double tol) {
    if (threadIdx.x == 0) state[5] = tol;
}

}  // namespace
}  // namespace heff

extern "C" int heff_davidson_workspace_size(const heff_plan* plan, int32_t max_vecs, size_t* bytes) {
    clear_error();
    if (!plan || !bytes || max_vecs < 1 || max_vecs > 64)
        return fail(HEFF_ERR_INVALID_ARG, "heff_davidson_workspace_size: bad arguments (max_vecs 1..64)");
    *bytes = dav_layout(plan->nelem_x, max_vecs).bytes;
    return HEFF_OK;
}

extern "C" int heff_davidson(heff_plan* plan, const void* L, const void* W1, const void* W2, const void* R,
                             const double* x0, const double* rnd, int32_t max_vecs, double tol, double* x_out,
                             double* result, void* apply_ws, size_t apply_ws_bytes, void* dav_ws,
                             size_t dav_ws_bytes, void* stream) {
    clear_error();
    if (!plan || !L || !W1 || !W2 || !R || !x0 || !rnd || !x_out || !result || !dav_ws)
        return fail(HEFF_ERR_INVALID_ARG, "heff_davidson: null argument");
    if (plan->opts.io_dtype != HEFF_DTYPE_F64)
        return fail(HEFF_ERR_UNSUPPORTED, "heff_davidson needs a plan with HEFF_DTYPE_F64 tensors");
    if (max_vecs < 1 || max_vecs > 64) return fail(HEFF_ERR_INVALID_ARG, "max_vecs must be 1..64");
    if (plan->nelem_x == 0) return fail(HEFF_ERR_INVALID_ARG, "heff_davidson: the two-site space is empty");
    if (!(tol >= 0.0)) return fail(HEFF_ERR_INVALID_ARG, "tol must be >= 0");
    const DavLayout lay = dav_layout(plan->nelem_x, max_vecs);
    if (dav_ws_bytes < lay.bytes || reinterpret_cast<uintptr_t>(dav_ws) % 256)
        return fail(HEFF_ERR_WORKSPACE, "Davidson workspace of %zu bytes, needs %zu (256-byte aligned)",
                    dav_ws_bytes, lay.bytes);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* base = static_cast<char*>(dav_ws);
    double* state = reinterpret_cast<double*>(base + lay.off_state);
    double* M = reinterpret_cast<double*>(base + lay.off_M);
    double* E = reinterpret_cast<double*>(base + lay.off_E);
    double* s = reinterpret_cast<double*>(base + lay.off_s);
    double* h = reinterpret_cast<double*>(base + lay.off_h);
    double* part = reinterpret_cast<double*>(base + lay.off_part);
    double* V = reinterpret_cast<double*>(base + lay.off_V);
    double* VA = reinterpret_cast<double*>(base + lay.off_VA);
    double* q = reinterpret_cast<double*>(base + lay.off_q);
    const int64_t n = plan->nelem_x;
    const int G = grid_for(n);
    const int GN = G < 1024 ? G : 1024;      // normalize: every block re-sums the RB partials
    int rc = heff_prepare(plan, L, W1, W2, R, apply_ws, apply_ws_bytes, stream);
    if (rc) return rc;
    dav_init_state_kernel<<<1, 32, 0, st>>>(state, tol);
    // v_0 = x0 / ||x0|| (sets active when x0 != 0), v^A_0 = A v_0
    sumsq_kernel<<<RB, RT, 0, st>>>(x0, n, part);
    normalize_kernel<<<GN, RT, 0, st>>>(part, RB, x0, V, n, state, 0);
    count_launches(3);
    if ((rc = heff_apply_prepared(plan, V, VA, apply_ws, apply_ws_bytes, stream))) return rc;
    auto gram_schmidt = [&](int nv) {          // q -= V (V^T q) over v_0 .. v_{nv-1}
        for (int j0 = 0; j0 < nv; j0 += VT) {
            const int k = nv - j0 < VT ? nv - j0 : VT;
            multidot_kernel<<<RB, RT, 0, st>>>(V, q, n, j0, k, part, state);
            finish_dots_kernel<<<1, RT, 0, st>>>(part, RB, j0, k, h, 0, state);
            count_launches(2);
        }
        combine_kernel<<<G, RT, 0, st>>>(V, n, nv, h, -1.0, 1.0, q, state);
        count_launches(1);
    };
    for (int i = 0; i < max_vecs; ++i) {
        double* vi = V + (int64_t)i * n;
        // m_ij = (v^A_j)^T v_i, j <= i
        for (int j0 = 0; j0 <= i; j0 += VT) {
            const int k = i + 1 - j0 < VT ? i + 1 - j0 : VT;
            multidot_kernel<<<RB, RT, 0, st>>>(VA, vi, n, j0, k, part, state);
            finish_dots_kernel<<<1, RT, 0, st>>>(part, RB, j0, k, h, 0, state);
            count_launches(2);
        }
        dav_set_m_kernel<<<1, 64, 0, st>>>(M, h, i, max_vecs, state);
        dav_eig_kernel<<<1, 32, 0, st>>>(M, E, s, state, i + 1, max_vecs);
        // x = V s, q = V^A s - lambda x, ||q||
        combine_kernel<<<G, RT, 0, st>>>(V, n, i + 1, s, 1.0, 0.0, x_out, state);
        combine_kernel<<<G, RT, 0, st>>>(VA, n, i + 1, s, 1.0, 0.0, q, state);
        dav_shift_kernel<<<G, RT, 0, st>>>(q, x_out, n, state);
        sumsq_kernel<<<RB, RT, 0, st>>>(q, n, part);
        dav_check_kernel<<<1, RT, 0, st>>>(part, RB, state, i + 1 == max_vecs);
        count_launches(7);
        if (i + 1 == max_vecs) break;
        // orthogonalise q against v_0..v_i (two classical Gram-Schmidt passes), randomise if
        // nothing is left, orthogonalise again, normalise into v_{i+1}, v^A_{i+1} = A v_{i+1}
        gram_schmidt(i + 1);
        gram_schmidt(i + 1);
        sumsq_kernel<<<RB, RT, 0, st>>>(q, n, part);
        dav_random_kernel<<<G, RT, 0, st>>>(part, RB, q, rnd, n, state);
        count_launches(2);
        gram_schmidt(i + 1);
        gram_schmidt(i + 1);
        double* vn = V + (int64_t)(i + 1) * n;
        sumsq_kernel<<<RB, RT, 0, st>>>(q, n, part);
        normalize_kernel<<<GN, RT, 0, st>>>(part, RB, q, vn, n, state, 3);
        count_launches(2);
        if ((rc = heff_apply_prepared(plan, vn, VA + (int64_t)(i + 1) * n, apply_ws, apply_ws_bytes, stream)))
            return rc;
    }
    sumsq_kernel<<<RB, RT, 0, st>>>(x_out, n, part);
    normalize_kernel<<<GN, RT, 0, st>>>(part, RB, x_out, x_out, n, state, 2);
    count_launches(2);
    // result: [lambda, ||q||, vectors used]
    cudaMemcpyAsync(result, state + 2, sizeof(double) * 2, cudaMemcpyDeviceToDevice, st);
    cudaMemcpyAsync(result + 2, state, sizeof(double), cudaMemcpyDeviceToDevice, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "heff_davidson: %s", cudaGetErrorString(e));
    return HEFF_OK;
}
