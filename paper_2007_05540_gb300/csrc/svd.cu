// Block SVD split of the two-site tensor with truncation, FP64 on the GPU (Section IV:
// the tensor is "wrapped" into a matrix with rows (a, s1) and columns (s2, b), one dense
// block per charge Q; Fig. 1e: the factors are split and the singular values absorbed in
// the sweep direction; Section II-C: singular values below a cutoff are removed).
//
// Each charge block M_Q (rows (s1, i, a), columns (s2, j, b)) is decomposed by one-sided
// Jacobi rotations (Hestenes): the columns of J = M_Q (or M_Q^T when M_Q is wide) are made
// mutually orthogonal by plane rotations applied in a round-robin order, so every round
// rotates k/2 disjoint column pairs in parallel (one thread block per pair, all sectors in
// one launch); V accumulates the rotations.  On convergence the column norms are the singular
// values.  The truncation rule runs on the host on the singular values; the kept singular
// triplets are then written into the caller's left (a, s1, c) and right (c, s2, b) tensors.
//
// Precision: the GB300's FP64 rate is low, and a full FP64 Jacobi run needs ~18 sweeps of
// ~12 r k^2 flops.  The sweeps therefore start on an FP32 copy (J32, V32) until the
// columns are orthogonal to FP32 accuracy (block sweeps: pairs of 16-column blocks, each
// rotated by one Jacobi sweep on its 32 x 32 Gram matrix, see svd_block_sweep_kernel); V32 is made orthonormal in FP64 by two
// Newton-Schulz steps (V <- V (3 I - V^T V) / 2, each squaring the orthogonality error),
// J <- J V in FP64, and FP64 Jacobi sweeps, accumulating into V, finish the
// decomposition (quadratic convergence from the preconditioned start: 2-3 sweeps).  The
// result is the FP64 one-sided Jacobi SVD of J; the FP32 phase only supplies the start.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <new>
#include <numeric>
#include <tuple>

#include "barrier.cuh"
#include "internal.h"

using heff::fail;

namespace {

struct SvdSector {           // device-side description of one charge block
    int64_t j_off, v_off;    // column-major J (r x k) and V (k x k) in the workspace
    int64_t g_off, w_off;    // FP64 scratch: G (k x k), W (r x k)
    int64_t j32_off, v32_off;    // FP32 copies (offsets in floats from the FP32 region)
    int32_t r, k;            // rows, columns of J (k <= r)
    int32_t transposed;      // 1 when J = M_Q^T
    int32_t s_off;           // first singular value of this sector in the s array
};

struct WriteEntry {          // one output block element range: dst block <- kept vectors
    int64_t dst_off;         // output block offset
    int32_t rows, cols;      // output block shape
    int32_t sec;             // sector
    int32_t vec_row0;        // first row inside the left (or right) singular vectors
    int32_t kept_off;        // offset into the kept-index list of this sector
    int32_t left;            // 1: left tensor A[(a), c] ; 0: right tensor B[c, (b)]
};

}  // namespace

struct heff_svd {
    int nq = 1;
    std::vector<std::vector<int32_t>> Q;       // sector charges
    std::vector<SvdSector> sec;
    // per sector: row groups (i, s1) with row offsets, column groups (s2, j)
    std::vector<std::vector<std::tuple<int, int, int32_t>>> rows, cols;    // (sector idx, phys, offset)
    std::vector<std::vector<int64_t>> xoff;    // per sector: x block offsets [row group][col group]
    std::vector<int32_t> mrows, ncols;         // M_Q shape
    int64_t ws_doubles = 0;
    // byte offset of the sweeps' words: convergence measures and counts (16), the sectors' pair offsets, the grid
    // barrier and its error word (3), the sectors' block-pair offsets
    size_t off_words = 0;
    size_t ws_bytes = 0;
    int64_t s_total = 0;
    std::vector<double> s;                     // singular values (per sector, unsorted)
    std::vector<std::vector<int32_t>> kept;    // per sector: kept column indices of J, s descending
    double norm = 0, discarded = 0;
    SvdSector* d_sec = nullptr;
    size_t off_f32 = 0;                        // byte offset of the FP32 region
    heff::BList gram, vg, jv;                  // G = V^T V, W = V G, W = J V (all sectors)
    bool lists_uploaded = false;
    int fp32_sweeps = 0, fp64_sweeps = 0;
    std::vector<int> pair_off;                 // prefix sums of the sectors' pair counts
    int max_k = 0;
    bool computed = false;
    int alpha_nsec = 0, beta_nsec = 0;
    std::vector<int32_t> alpha_dims, beta_dims;
};

namespace {

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Blocks per tensor block of the kernels that copy between the tensors and J, V: bound by latency, and a tensor of
// few blocks leaves most SMs idle with one each (m = 512, 70 tensor blocks: 26 and 40 us).  Eight is from that size
// alone.
constexpr int COPY_SPLIT = 8;

// scatter x blocks into column-major J (or J^T layout for wide sectors)
__global__ void svd_load_kernel(const SvdSector* __restrict__ secs, const int64_t* __restrict__ tab, int ntab,
                                const double* __restrict__ x, double* __restrict__ ws) {
    // tab: per x block: [sector, x_off, m_rows, n_cols, row0 in M, col0 in M]
    for (int b = blockIdx.x; b < ntab; b += gridDim.x) {
        const int64_t* t = tab + 6 * b;
        const SvdSector s = secs[t[0]];
        const int64_t xo = t[1];
        const int mr = (int)t[2], nc = (int)t[3], r0 = (int)t[4], c0 = (int)t[5];
        double* J = ws + s.j_off;
        for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < mr * nc; e += gridDim.y * blockDim.x) {
            const int a = e / nc, c = e % nc;
            const int R = r0 + a, Cc = c0 + c;         // position in M_Q
            const double v = x[xo + e];
            if (!s.transposed) J[(int64_t)Cc * s.r + R] = v;     // J = M: column Cc, row R
            else J[(int64_t)R * s.r + Cc] = v;                    // J = M^T: column R, row Cc
        }
    }
}


// J32 = float(J), V32 = I
__global__ void svd_to_f32_kernel(const SvdSector* __restrict__ secs, const double* __restrict__ ws,
                                  float* __restrict__ f32) {
    const SvdSector s = secs[blockIdx.y];
    const int64_t nj = (int64_t)s.r * s.k, nv = (int64_t)s.k * s.k;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nj + nv; e += (int64_t)gridDim.x * blockDim.x) {
        if (e < nj) f32[s.j32_off + e] = (float)ws[s.j_off + e];
        else {
            const int64_t v = e - nj;
            f32[s.v32_off + v] = (v % (s.k + 1) == 0) ? 1.f : 0.f;
        }
    }
}

// V = double(V32)
__global__ void svd_v_to_f64_kernel(const SvdSector* __restrict__ secs, const float* __restrict__ f32,
                                    double* __restrict__ ws) {
    const SvdSector s = secs[blockIdx.y];
    const int64_t nv = (int64_t)s.k * s.k;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nv; e += (int64_t)gridDim.x * blockDim.x)
        ws[s.v_off + e] = (double)f32[s.v32_off + e];
}

// G = V^T V - 1: what is left of the identity is all of one size (products with G itself would round to its ones)
__global__ void svd_residual_kernel(const SvdSector* __restrict__ secs, double* __restrict__ ws) {
    const SvdSector s = secs[blockIdx.y];
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < s.k; e += gridDim.x * blockDim.x)
        ws[s.g_off + (int64_t)e * (s.k + 1)] -= 1.0;
}

// Newton-Schulz combine: V (3 - V^T V) / 2 = V + W, with W = -0.5 V (V^T V - 1) already formed
__global__ void svd_ns_kernel(const SvdSector* __restrict__ secs, double* __restrict__ ws) {
    const SvdSector s = secs[blockIdx.y];
    const int64_t nv = (int64_t)s.k * s.k;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nv; e += (int64_t)gridDim.x * blockDim.x)
        ws[s.v_off + e] += ws[s.w_off + e];
}

// J = W (the product J V)
__global__ void svd_copy_w_kernel(const SvdSector* __restrict__ secs, double* __restrict__ ws) {
    const SvdSector s = secs[blockIdx.y];
    const int64_t nj = (int64_t)s.r * s.k;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nj; e += (int64_t)gridDim.x * blockDim.x)
        ws[s.j_off + e] = ws[s.w_off + e];
}

// A sweep (all rounds) inside one cooperative launch: the warps of the grid take the
// (sector, pair) items of a round from a flattened list (pair_off: prefix sums of each
// sector's pair count), rotate, and meet at a grid barrier before the next round.  The
// barrier is a counter word in global memory; its wait is bounded (about a
// second), after which the kernel sets err and returns.  The phase's further sweeps follow in the same launch.
//
// Column norms are carried instead of recomputed per pair (as in the standard one-sided
// Jacobi codes): the sweep starts by computing every column's squared norm into nrm
// (indexed like the singular values, s_off + column), and a rotation by tan(theta) = t of
// columns with squared norms a, b and inner product g leaves exactly a - t g and b + t g
// (the rotation zeroes the inner product).  A pair then needs one dot product instead of
// three.  The updates change a norm by t g, tiny once the columns are nearly orthogonal, and
// the norms are recomputed at the start of every sweep, so the rounding drift stays at a
// few ulps of the column's norm.
//
// Bound by the latency of a round (grid barrier 2 us, a trip to L2, the dot product's and the angle's chains),
// which FP64 work lengthens where several pairs share an SM's FP64 unit (two lanes a clock: a warp's
// instruction holds it 16 cycles).  So the pairs go to blocks first and warps second, which spreads them over every SM
// (472 pairs on 59 SMs: 2.45 ms a sweep); the first SVD_PIECES * 32 rows of both columns of J and V are
// loaded at once and stay in registers from the dot product to the rotation; and a rotation takes three
// multiply-adds per element pair, as the shears u -= p v, v += s u, u -= p v with p = tan(theta / 2), or
// two where the cosine rounds to one, instead of two products and two multiply-adds; and an angle takes one
// division: 0.82 ms a sweep (942 columns in 19 sectors; 0.11 ms of it is FP64 multiply-adds at 0.6 T/s).  The
// shears have determinant one whatever p and s round to; with a cosine that rounds to one the columns grew
// with every rotation (sum of s^2 over |x|^2 - 1 at m = 512: 1.2e-14, now 6e-16).
constexpr int SVD_SWEEP_NT = 256;
constexpr int SVD_PIECES = 16;
using heff::grid_barrier;

// The sweeps of a phase are one launch: they end when a sweep's largest off-diagonal measure is below stop.
struct Sweeps {
    int limit;
    float stop;
    int* seen;                   // [3]: a sweep's largest measure (float bits), zero before the launch
    int* count;                  // sweeps run
};

// Whether to run another sweep after number `sweep`, in which this block saw `mine` (float bits, >= 0).  A
// slot is cleared while the sweep before it runs, two barriers after it was last read.
__device__ __forceinline__ bool sweep_goes_on(const Sweeps& sw, int sweep, int mine, unsigned int* bar, int* err) {
    if (threadIdx.x == 0) {
        atomicMax(sw.seen + sweep % 3, mine);
        if (blockIdx.x == 0) {
            sw.seen[(sweep + 1) % 3] = 0;
            *sw.count = sweep + 1;
        }
    }
    if (!grid_barrier(bar, gridDim.x, err)) return false;
    return !(__int_as_float(*(volatile int*)(sw.seen + sweep % 3)) < sw.stop);
}

struct Rotation {
    double p, s;                 // tan(theta / 2), sin(theta)
};

// |g| / sqrt(a b) for a, b > 0.  It steers the sweeps, so FP32 will do: the three numbers, over the larger
// square's power of two, get their FP32 forms from their upper words, 20 bits of mantissa each, without an
// FP64 instruction (a root and a division in FP64 cost as much as rotating 180 rows).
__device__ __forceinline__ float off_diagonal(double g, double a, double b) {
    const int ha = __double2hiint(a), hb = __double2hiint(b), hg = __double2hiint(g) & 0x7fffffff;
    const int e = max(ha, hb) >> 20;                     // biased exponent of the larger square
    auto scaled = [&](int h) {
        const int x = (h >> 20) - e + 127;
        return x > 0 && x < 255 ? __int_as_float((x << 23) | ((h & 0xfffff) << 3)) : 0.f;
    };
    const float ab = scaled(ha) * scaled(hb);
    if (e > 64 && e < 2047 && ab > 1e-36f) return scaled(hg) * rsqrtf(ab);
    return (float)(fabs(g) / sqrt(a * b));
}

// tan(theta) of the rotation that makes columns of squared norms a, b and inner product g orthogonal, and
// its shears.  With w = 2 g / (b - a) = tan(2 theta) under 1e-3 by the first terms of their series in w (the
// next are under 3e-19): one division instead of three and two roots.
__device__ __forceinline__ double rotation(double g, double a, double b, Rotation& r) {
    const double d = b - a, g2 = 2.0 * g;
    if (fabs(g2) < 1e-3 * fabs(d)) {
        const double w = g2 / d, w2 = w * w;
        r.p = w * fma(w2, fma(w2, 23.0 / 512.0, -5.0 / 64.0), 0.25);
        r.s = w * fma(w2, fma(w2, 31.0 / 256.0, -3.0 / 16.0), 0.5);
        return w * fma(w2, fma(w2, 0.0625, -0.125), 0.5);
    }
    const double zeta = d / g2;
    const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
    const double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
    r.p = s / (1.0 + c);
    r.s = s;
    return t;
}

template <bool TINY>
__device__ __forceinline__ void rotate(const Rotation& r, double& u, double& v) {
    if (TINY) {
        const double u0 = u;
        u = fma(-r.s, v, u0);
        v = fma(r.s, u0, v);
    } else {
        u = fma(-r.p, v, u);
        v = fma(r.s, u, v);
        u = fma(-r.p, v, u);
    }
}

// Rotates the columns cp, cq of n rows, whose first SVD_PIECES * 32 rows are in u, v.
template <bool TINY>
__device__ __forceinline__ void rotate_columns(const Rotation& rot, double* cp, double* cq, int n, int lane,
                                               double (&u)[SVD_PIECES], double (&v)[SVD_PIECES]) {
#pragma unroll
    for (int t = 0; t < SVD_PIECES; ++t)
        if (32 * t < n) {                                // uniform: no FP64 work past the last row
            rotate<TINY>(rot, u[t], v[t]);
            const int i = lane + 32 * t;
            if (i < n) {
                cp[i] = u[t];
                cq[i] = v[t];
            }
        }
    for (int i0 = lane + 32 * SVD_PIECES; i0 < n; i0 += 32 * 4) {
        double a[4], b[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = i0 + 32 * t;
            a[t] = i < n ? cp[i] : 0.0;
            b[t] = i < n ? cq[i] : 0.0;
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const int i = i0 + 32 * t;
            if (i < n) {
                rotate<TINY>(rot, a[t], b[t]);
                cp[i] = a[t];
                cq[i] = b[t];
            }
        }
    }
}

__global__ void __launch_bounds__(SVD_SWEEP_NT, 1) svd_sweep_kernel(const SvdSector* __restrict__ secs, int nsec,
                                                                 const int* __restrict__ pair_off, int kk_all,
                                                                 double* __restrict__ base, double* __restrict__ nrm,
                                                                 int ncols_all, Sweeps sw,
                                                                 unsigned int* __restrict__ bar, int* __restrict__ err) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    constexpr int warps = SVD_SWEEP_NT / 32;
    const int gw = w * gridDim.x + blockIdx.x, nw = gridDim.x * warps;
    const int npairs = pair_off[nsec];
    // (a warp's first item is the same in every round: its sector is looked up once, since a barrier
    // empties L1 and each step of the search then waits for L2)
    SvdSector s{};
    int pair = 0;
    auto find = [&](int item) {
        int lo = 0, hi = nsec;                           // sector: pair_off[lo] <= item < pair_off[lo + 1]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pair_off[mid] <= item) lo = mid; else hi = mid;
        }
        s = secs[lo];
        pair = item - pair_off[lo];
    };
    const bool several = npairs > nw;
    if (gw < npairs) find(gw);
    __shared__ int mx;
    for (int sweep = 0; sweep < sw.limit; ++sweep) {
    if (threadIdx.x == 0) mx = 0;
    float mymax = 0.f;
    // squared column norms (one warp per column; the sectors' s_off are prefix sums of k)
    for (int item = gw; item < ncols_all; item += nw) {
        int lo = 0, hi = nsec;                           // sector: s_off[lo] <= item < s_off[lo + 1]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (secs[mid].s_off <= item) lo = mid; else hi = mid;
        }
        const SvdSector cs = secs[lo];
        const int n = cs.r;
        const double* c = base + cs.j_off + (int64_t)(item - cs.s_off) * n;
        double a = 0;
        for (int i0 = lane; i0 < n; i0 += 32 * 8) {
            double u[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) u[t] = i0 + 32 * t < n ? c[i0 + 32 * t] : 0.0;
#pragma unroll
            for (int t = 0; t < 8; ++t) a = fma(u[t], u[t], a);
        }
        a = warp_sum(a);
        if (lane == 0) nrm[item] = a;
    }
    if (!grid_barrier(bar, gridDim.x, err)) return;
    for (int round = 0; round < kk_all - 1; ++round) {
        for (int item = gw; item < npairs; item += nw) {
            if (several) find(item);
            const int kk = s.k + (s.k & 1);
            if (round >= kk - 1) continue;
            auto pos = [&](int j) { return j == 0 ? 0 : 1 + (j - 1 + round) % (kk - 1); };
            int p = pos(pair), q = pos(kk - 1 - pair);
            if (p >= s.k || q >= s.k) continue;          // pair with the dummy column
            if (p > q) { const int t = p; p = q; q = t; }
            double* cp = base + s.j_off + (int64_t)p * s.r;
            double* cq = base + s.j_off + (int64_t)q * s.r;
            double* vp = base + s.v_off + (int64_t)p * s.k;
            double* vq = base + s.v_off + (int64_t)q * s.k;
            double* np = nrm + s.s_off + p;
            double* nq = nrm + s.s_off + q;
            const double a = *np, b = *nq;
            double u[SVD_PIECES], v[SVD_PIECES], x[SVD_PIECES], y[SVD_PIECES];
#pragma unroll
            for (int t = 0; t < SVD_PIECES; ++t) {
                const int i = lane + 32 * t;
                u[t] = i < s.r ? cp[i] : 0.0;
                v[t] = i < s.r ? cq[i] : 0.0;
            }
#pragma unroll
            for (int t = 0; t < SVD_PIECES; ++t) {
                const int i = lane + 32 * t;
                x[t] = i < s.k ? vp[i] : 0.0;
                y[t] = i < s.k ? vq[i] : 0.0;
            }
            double g4[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
            for (int t = 0; t < SVD_PIECES; ++t)
                if (32 * t < s.r) g4[t & 3] = fma(u[t], v[t], g4[t & 3]);
            for (int i0 = lane + 32 * SVD_PIECES; i0 < s.r; i0 += 32 * 4) {
                double c[4], d[4];
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int i = i0 + 32 * t;
                    c[t] = i < s.r ? cp[i] : 0.0;
                    d[t] = i < s.r ? cq[i] : 0.0;
                }
#pragma unroll
                for (int t = 0; t < 4; ++t) g4[t] = fma(c[t], d[t], g4[t]);
            }
            const double g = warp_sum((g4[0] + g4[1]) + (g4[2] + g4[3]));
            if (g == 0.0 || a == 0.0 || b == 0.0) continue;
            const float meas = off_diagonal(g, a, b);
            mymax = fmaxf(mymax, meas);
            if (meas < 1e-15f) continue;
            Rotation rot;
            const double t = rotation(g, a, b, rot);
            if (lane == 0) {                             // the rotated columns' squared norms
                *np = a - t * g;
                *nq = b + t * g;
            }
            if (fabs(t) < 7.4505805969238281e-9) {       // 2^-27: the cosine, 1 - t^2 / 2, rounds to 1
                rotate_columns<true>(rot, cp, cq, s.r, lane, u, v);
                rotate_columns<true>(rot, vp, vq, s.k, lane, x, y);
            } else {
                rotate_columns<false>(rot, cp, cq, s.r, lane, u, v);
                rotate_columns<false>(rot, vp, vq, s.k, lane, x, y);
            }
        }
        if (!grid_barrier(bar, gridDim.x, err)) return;
    }
    for (int o = 16; o > 0; o >>= 1) mymax = fmaxf(mymax, __shfl_xor_sync(0xffffffffu, mymax, o));
    if (lane == 0) atomicMax(&mx, __float_as_int(mymax));
    __syncthreads();
    if (!sweep_goes_on(sw, sweep, mx, bar, err)) return;
    }
}

// Block one-sided Jacobi sweep for the FP32 preconditioning phase.  The columns of each
// sector are grouped into blocks of SVD_BW; a round pairs the blocks round-robin (a block
// left without a partner, or the only block, is processed alone), and one thread block
// takes one block pair: it forms the Gram matrix G = P^T P of the pair's <= 2 SVD_BW columns
// (its columns in shared memory), runs one cyclic Jacobi sweep on G (disjoint
// rotations in parallel; each is the rotation the one-sided method would apply to that
// column pair), accumulates the rotations in W, and updates the columns of J and V by
// P <- P W.  One round per block pair instead of one per column pair: ~SVD_BW times fewer
// grid barriers per sweep, and the work is in small dense products.  The sweep's
// measure is the largest off-diagonal ratio |G_ab| / sqrt(G_aa G_bb).
//
// Bound by the latency of its steps (a pair of 216 + 179 rows, cycles a round: Gram matrix 5300, rotations
// 10400, update 8700, copies 2200, barrier 6000).  A sweep of m = 512 (942 columns in 19 sectors) went from
// 371 to 195 us: 31 rounds of rotations from 24000 cycles to 10400, the rest from columns resident in shared
// memory and 16-byte loads.
constexpr int SVD_BW = 16, SVD_PC = 2 * SVD_BW;
#ifndef SVD_TR_ROWS
#define SVD_TR_ROWS 128
#endif
constexpr int SVD_TR = SVD_TR_ROWS;

// row pitches: of G even, for 8-byte loads, with the 2 x 2 blocks on the diagonal in different banks; of W for
// 16-byte loads
constexpr int SVD_GLD = SVD_PC + 2, SVD_WLD = SVD_PC + 4;

// cosine and sine of the rotation that zeroes gab, in FP32 (the block sweeps only precondition).  The rounds
// of a block pair wait for one another through this chain, so it is written with two dependent reciprocal
// roots and no division.
__device__ __forceinline__ float2 pair_rotation(float gab, float gaa, float gbb) {
    // |gab| against 1e-7 of the columns' norms
    float n;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(n) : "f"(gaa * gbb));
    const bool turn = gab != 0.f && gaa > 0.f && gbb > 0.f && fabsf(gab) > 1e-7f * n;
    // scaled by a power of two so that the larger square lies in [1, 2)
    // (to [2, 4) at the top of the range, where the reciprocal would be subnormal)
    const float scale = __int_as_float(max(0x7f000000 - (__float_as_int(fmaxf(gaa, gbb)) & 0x7f800000), 0x00800000));
    const float d = (gbb - gaa) * scale, g = gab * scale;
    // cos(2 theta) = |d| / h, sin(2 theta) = 2 g / h, h^2 = d^2 + 4 g^2, |theta| <= pi / 4
    const float rh = rsqrtf(fmaf(d, d, 4.f * g * g));
    const float c2 = fmaf(0.5f * fabsf(d), rh, 0.5f), rc = rsqrtf(c2);
    float c = c2 * rc, sn = copysignf(1.f, d) * (g * rh * rc);
    // The approximate roots leave c^2 + s^2 a few ulps from one, always to the same side, and a column goes
    // through k rotations a sweep: a Newton step to unit length.  (Without it V32 was too far from orthonormal
    // for the two Newton-Schulz steps at k = 2450: V^T V - 1 ended at 8e-11, with it at 1e-14.)
    const float e = 0.5f * fmaf(-sn, sn, fmaf(-c, c, 1.f));
    c = fmaf(c, e, c);
    sn = fmaf(sn, e, sn);
    return turn ? make_float2(c, sn) : make_float2(1.f, 0.f);
}

__device__ __forceinline__ int rr_pos(int j, int round, int n) { return j == 0 ? 0 : 1 + (j - 1 + round) % (n - 1); }

#ifndef SVD_BT_THREADS
#define SVD_BT_THREADS 512
#endif
constexpr int SVD_BT = SVD_BT_THREADS;    // threads of a block-pair CTA
// RES: the pair's columns of J and V are copied to shared memory once (rows_j + rows_v rows of SVD_TLD
// floats), V's while G is formed and turned; else they pass through one tile of SVD_TR rows, twice for J.
// (row pitch: 8 rows of four consecutive columns lie in 32 different banks)
constexpr int SVD_TLD = SVD_PC + 4;
constexpr size_t SVD_RES_BYTES = 208 << 10;          // with 18 KB of static shared memory within the SM's 227
template <bool RES>
__global__ void __launch_bounds__(SVD_BT) svd_block_sweep_kernel(const SvdSector* __restrict__ secs, int nsec,
                                                              const int* __restrict__ bpair_off, int nbb_all,
                                                              float* __restrict__ base, Sweeps sw,
                                                              unsigned int* __restrict__ bar, int* __restrict__ err,
                                                              int rows_j) {
    extern __shared__ __align__(16) float dyn[];
    float* const sj = dyn;
    float* const sv = RES ? dyn + (int64_t)rows_j * SVD_TLD : dyn;
    __shared__ __align__(16) float G[2][SVD_PC][SVD_GLD], W[2][SVD_PC][SVD_WLD];
    __shared__ int col[SVD_PC];
    __shared__ int bmax;
    const int tid = threadIdx.x;
    const int npairs = bpair_off[nsec];
    SvdSector sc{};
    int pair = 0;
    auto find = [&](int item) {                          // bpair_off[lo] <= item < bpair_off[lo + 1]
        int lo = 0, hi = nsec;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (bpair_off[mid] <= item) lo = mid; else hi = mid;
        }
        sc = secs[lo];
        pair = item - bpair_off[lo];
    };
    const bool several = npairs > (int)gridDim.x;        // (a block's only item is looked up once)
    if ((int)blockIdx.x < npairs) find(blockIdx.x);
    for (int sweep = 0; sweep < sw.limit; ++sweep) {
    if (tid == 0) bmax = 0;                              // (the pairs synchronise before they use it)
    for (int round = 0; round < nbb_all - 1; ++round) {
        for (int item = blockIdx.x; item < npairs; item += gridDim.x) {
            if (several) find(item);
            const int nb = (sc.k + SVD_BW - 1) / SVD_BW, nbb = nb + (nb & 1);
            if (round >= (nbb > 1 ? nbb - 1 : 1)) continue;                 // block-uniform
            int bp = nbb > 1 ? rr_pos(pair, round, nbb) : 0;
            int bq = nbb > 1 ? rr_pos(nbb - 1 - pair, round, nbb) : nbb;
            if (bp >= nb) { const int t = bp; bp = bq; bq = t; }              // the real block first
            if (bp >= nb) continue;
            const int np = min(SVD_BW, sc.k - bp * SVD_BW);
            const int nq = bq < nb ? min(SVD_BW, sc.k - bq * SVD_BW) : 0;
            const int nc = np + nq;
            if (tid < SVD_PC) col[tid] = tid < np ? bp * SVD_BW + tid : (tid < nc ? bq * SVD_BW + tid - np : -1);
            float* J = base + sc.j32_off;
            float* V = base + sc.v32_off;
            __syncthreads();
            // (a column that is not there, and the rows up to the next multiple of 8, are zeros)
            auto copy_columns = [&](float* dst, const float* M, int rows) {
                const int a = 4 * ((tid >> 5) & 7) + ((tid >> 3) & 3), cidx = col[a];
                const float* src = M + (int64_t)max(cidx, 0) * rows;
#pragma unroll 4
                for (int rr = 8 * (tid >> 8) + (tid & 7); rr < (rows + 7) / 8 * 8; rr += 16) {
                    const bool in = cidx >= 0 && rr < rows;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(dst + rr * SVD_TLD + a)),
                                 "l"(in ? src + rr : src), "r"(in ? 4 : 0)
                                 : "memory");
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            if (RES) {
                copy_columns(sj, J, sc.r);
                copy_columns(sv, V, sc.k);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
                __syncthreads();
            }
            // 1. G = P^T P, register-tiled: thread t takes the 4 x 4 block blk = t / 8 of G
            //    (rows 4 (blk / 8) .., columns 4 (blk % 8) ..) over the tile rows g, g + 8, ...
            //    (g = t % 8), and the 8 partial sums of a block (8 consecutive lanes) are added
            //    by shuffles: two 16-byte shared-memory loads per 16 FMAs
            static_assert(SVD_PC == 32 && SVD_BT == 512 && SVD_TR % 8 == 0, "Gram tiling assumes 32 columns");
            const int gblk = tid >> 3, gg = tid & 7;
            const int ga0 = 4 * (gblk >> 3), gb0 = 4 * (gblk & 7);
            float acc[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
            // tiles of SVD_TR rows; the next tile's loads are issued into registers before the
            // current tile is used, so their latency overlaps the arithmetic
            constexpr int TE = SVD_TR * SVD_PC / SVD_BT;                    // tile elements per thread
            float nxt[TE];
            auto load_tile = [&](const float* M, int rows, int r0) {
#pragma unroll
                for (int u = 0; u < TE; ++u) {
                    const int e = tid + SVD_BT * u, a = ((e >> 3) & 3) + 4 * ((e >> 5) & 7), rr = (e & 7) + 8 * (e >> 8);
                    const int cidx = col[a];
                    nxt[u] = (cidx >= 0 && r0 + rr < rows) ? M[(int64_t)cidx * rows + r0 + rr] : 0.f;
                }
            };
            auto stage_tile = [&]() {
#pragma unroll
                for (int u = 0; u < TE; ++u) {
                    const int e = tid + SVD_BT * u, a = ((e >> 3) & 3) + 4 * ((e >> 5) & 7), rr = (e & 7) + 8 * (e >> 8);
                    sj[rr * SVD_TLD + a] = nxt[u];
                }
            };
            if (!RES) load_tile(J, sc.r, 0);
            for (int r0 = 0; r0 < sc.r; r0 += SVD_TR) {
                if (!RES) {
                    stage_tile();
                    __syncthreads();
                    if (r0 + SVD_TR < sc.r) load_tile(J, sc.r, r0 + SVD_TR);
                }
                const float* tile = RES ? sj + r0 * SVD_TLD : sj;
                const int end = RES ? min(SVD_TR, (sc.r - r0 + 7) / 8 * 8) : SVD_TR;
#pragma unroll 4
                for (int rr = gg; rr < end; rr += 8) {
                    const float4 fa = *reinterpret_cast<const float4*>(tile + rr * SVD_TLD + ga0);
                    const float4 fb = *reinterpret_cast<const float4*>(tile + rr * SVD_TLD + gb0);
                    const float xa[4] = {fa.x, fa.y, fa.z, fa.w}, xb[4] = {fb.x, fb.y, fb.z, fb.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(xa[i], xb[j], acc[i][j]);
                }
                if (!RES) __syncthreads();
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) acc[i][j] += __shfl_xor_sync(0xffffffffu, acc[i][j], o);
            if (gg == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int a = ga0 + i, b = gb0 + j;
                        G[0][a][b] = a == b && a >= nc ? 1.f : acc[i][j];          // (an absent column: 1)
                    }
            }
            for (int e = tid; e < SVD_PC * SVD_PC; e += SVD_BT) W[0][e / SVD_PC][e % SVD_PC] = (e / SVD_PC == e % SVD_PC);
            __syncthreads();
            // off-diagonal measure before the rotations (thread t: row t / 16, columns 2 (t % 16) + u)
            {
                const int ga = tid / (SVD_PC / 2), gbp = (tid % (SVD_PC / 2)) * 2;
                float m = 0.f;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int b = gbp + u;
                    if (ga < b && b < nc) {
                        const float d = sqrtf(G[0][ga][ga] * G[0][b][b]);
                        if (d > 0.f) m = fmaxf(m, fabsf(G[0][ga][b]) / d);
                    }
                }
                for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if ((tid & 31) == 0) atomicMax(&bmax, __float_as_int(m));
            }
            // 2. one cyclic Jacobi sweep on G: SVD_PC - 1 rounds of SVD_PC / 2 disjoint rotations, each waiting
            //    for the one before.  The columns move instead of the pairs: pair j always lies in the places
            //    2 j, 2 j + 1, and a round writes what it turned to the places of the next (the tournament's
            //    step; after all rounds every column is back), so no address changes from round to round.
            //    Each lane l works out the rotation of pair l % 16; thread (i, j) of the first half takes
            //    the 2 x 2 block of the pairs i and j from one copy of G to the other, the second half two
            //    rows each of W.
            {
                const int j = tid & 15, i = (tid >> 4) & 15;
                // tournament position t (pairs t, 31 - t) <-> place; the column at position t moves to t - 1
                auto place = [](int t) { return t < 16 ? 2 * t : 2 * (SVD_PC - 1 - t) + 1; };
                auto next = [&](int t) { return place(t == 0 ? 0 : (t == 1 ? SVD_PC - 1 : t - 1)); };
                const int na = next(j), nb2 = next(SVD_PC - 1 - j);
                if (tid < 256) {
                    const int nc2 = next(i), nd = next(SVD_PC - 1 - i);
                    const int rd_j = 2 * j * SVD_GLD + 2 * j, rd_b = 2 * i * SVD_GLD + 2 * j;
                    const int wca = nc2 * SVD_GLD + na, wcb = nc2 * SVD_GLD + nb2;
                    const int wda = nd * SVD_GLD + na, wdb = nd * SVD_GLD + nb2;
                    auto step = [&](const float* Gc, float* Gn) {
                        const float2 g0 = *reinterpret_cast<const float2*>(Gc + rd_j);
                        const float gbb = Gc[rd_j + SVD_GLD + 1];
                        const float2 cv = *reinterpret_cast<const float2*>(Gc + rd_b);
                        const float2 dv = *reinterpret_cast<const float2*>(Gc + rd_b + SVD_GLD);
                        const float2 cs = pair_rotation(g0.y, g0.x, gbb);
                        const float rx = __shfl_sync(0xffffffffu, cs.x, i), ry = __shfl_sync(0xffffffffu, cs.y, i);
                        const float p0 = cs.x * cv.x - cs.y * cv.y, p1 = cs.y * cv.x + cs.x * cv.y;      // columns
                        const float q0 = cs.x * dv.x - cs.y * dv.y, q1 = cs.y * dv.x + cs.x * dv.y;
                        Gn[wca] = rx * p0 - ry * q0;                                                    // rows
                        Gn[wcb] = rx * p1 - ry * q1;
                        Gn[wda] = ry * p0 + rx * q0;
                        Gn[wdb] = ry * p1 + rx * q1;
                    };
                    for (int jr = 0; jr < SVD_PC - 2; jr += 2) {
                        step(&G[0][0][0], &G[1][0][0]);
                        __syncthreads();
                        step(&G[1][0][0], &G[0][0][0]);
                        __syncthreads();
                    }
                } else {
                    const int rd_j = 2 * j * SVD_GLD + 2 * j;
                    auto step = [&](const float* Gc, const float* Wc, float* Wn) {
                        const float2 g0 = *reinterpret_cast<const float2*>(Gc + rd_j);
                        const float gbb = Gc[rd_j + SVD_GLD + 1];
                        const float2 u = *reinterpret_cast<const float2*>(Wc + i * SVD_WLD + 2 * j);
                        const float2 v = *reinterpret_cast<const float2*>(Wc + (i + 16) * SVD_WLD + 2 * j);
                        const float2 cs = pair_rotation(g0.y, g0.x, gbb);
                        Wn[i * SVD_WLD + na] = cs.x * u.x - cs.y * u.y;
                        Wn[i * SVD_WLD + nb2] = cs.y * u.x + cs.x * u.y;
                        Wn[(i + 16) * SVD_WLD + na] = cs.x * v.x - cs.y * v.y;
                        Wn[(i + 16) * SVD_WLD + nb2] = cs.y * v.x + cs.x * v.y;
                    };
                    for (int jr = 0; jr < SVD_PC - 2; jr += 2) {
                        step(&G[0][0][0], &W[0][0][0], &W[1][0][0]);
                        __syncthreads();
                        step(&G[1][0][0], &W[1][0][0], &W[0][0][0]);
                        __syncthreads();
                    }
                    step(&G[0][0][0], &W[0][0][0], &W[1][0][0]);
                }
            }
            if (RES) asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();
            // 3. P <- P W for the columns of J (r rows) and of V (k rows): a warp takes eight output columns of
            //    32 UR rows, UR rows a lane: 2 UR + 8 (broadcast) 16-byte shared-memory loads per 32 UR FMAs
            //    of four inner columns, coalesced column stores
            constexpr int UR = RES ? 2 : 1;
            const int ul = tid & 31, uw = tid >> 5;
            auto update = [&](const float* tile, float* M, int rows, int r0, int c8) {
                // rows r0 .. of M (tile: their first), output columns c8 .. c8 + 7
                float o[UR][8];
#pragma unroll
                for (int u = 0; u < UR; ++u)
#pragma unroll
                    for (int c = 0; c < 8; ++c) o[u][c] = 0.f;
#pragma unroll 2
                for (int b4 = 0; b4 < SVD_PC; b4 += 4) {
                    float t[UR][4];
#pragma unroll
                    for (int u = 0; u < UR; ++u) {
                        const float4 f = *reinterpret_cast<const float4*>(tile + (ul + 32 * u) * SVD_TLD + b4);
                        t[u][0] = f.x; t[u][1] = f.y; t[u][2] = f.z; t[u][3] = f.w;
                    }
#pragma unroll
                    for (int bb = 0; bb < 4; ++bb) {
                        const float4 wa = *reinterpret_cast<const float4*>(&W[1][b4 + bb][c8]);
                        const float4 wb = *reinterpret_cast<const float4*>(&W[1][b4 + bb][c8 + 4]);
                        const float wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
                        for (int u = 0; u < UR; ++u)
#pragma unroll
                            for (int c = 0; c < 8; ++c) o[u][c] = fmaf(t[u][bb], wv[c], o[u][c]);
                    }
                }
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int cidx = col[c8 + c];
                    if (cidx < 0) continue;
#pragma unroll
                    for (int u = 0; u < UR; ++u)
                        if (r0 + ul + 32 * u < rows) M[(int64_t)cidx * rows + r0 + ul + 32 * u] = o[u][c];
                }
            };
            if (RES) {
                const int nj = (sc.r + 63) / 64, nv = (sc.k + 63) / 64;
                for (int unit = uw; unit < 4 * (nj + nv); unit += SVD_BT / 32) {
                    const int g = unit >> 2, c8 = 8 * (unit & 3);
                    if (g < nj) update(sj + 64 * g * SVD_TLD, J, sc.r, 64 * g, c8);
                    else update(sv + 64 * (g - nj) * SVD_TLD, V, sc.k, 64 * (g - nj), c8);
                }
            } else {
                static_assert(SVD_TR == 128 && SVD_BT == 512, "one unit of 32 rows and 8 columns per warp");
                for (int pass = 0; pass < 2; ++pass) {
                    float* M = pass == 0 ? J : V;
                    const int rows = pass == 0 ? sc.r : sc.k;
                    load_tile(M, rows, 0);
                    for (int r0 = 0; r0 < rows; r0 += SVD_TR) {
                        stage_tile();
                        __syncthreads();
                        if (r0 + SVD_TR < rows) load_tile(M, rows, r0 + SVD_TR);
                        const int rr = 32 * (uw >> 2);
                        if (r0 + rr < rows) update(sj + rr * SVD_TLD, M, rows, r0 + rr, 8 * (uw & 3));
                        __syncthreads();
                    }
                }
            }
            __syncthreads();
        }
        if (!grid_barrier(bar, gridDim.x, err)) return;
    }
    if (!sweep_goes_on(sw, sweep, bmax, bar, err)) return;
    }
}

// column norms of J = singular values
__global__ void svd_norms_kernel(const SvdSector* __restrict__ secs, const double* __restrict__ ws,
                                 double* __restrict__ sv) {
    const SvdSector s = secs[blockIdx.y];
    const int col = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (col >= s.k) return;
    const double* c = ws + s.j_off + (int64_t)col * s.r;
    double a = 0;
    for (int i = lane; i < s.r; i += 32) a = fma(c[i], c[i], a);
    a = warp_sum(a);
    if (lane == 0) sv[s.s_off + col] = sqrt(a);
}

// Write kept singular triplets.  Left vectors of M: columns of J / s (not transposed) or of
// V (transposed); right vectors: columns of V (not transposed) or J / s (transposed).
// A block (i, s1, c): element (a, k) = left[row0 + a, kept_k] * (absorb left ? s : 1)
// B block (c, s2, j): element (k, b) = right[col0 + b, kept_k] * (absorb right ? s : 1)
__global__ void svd_write_kernel(const SvdSector* __restrict__ secs, const WriteEntry* __restrict__ ent,
                                 const int32_t* __restrict__ kept, const double* __restrict__ ws,
                                 const double* __restrict__ sv, double* __restrict__ A, double* __restrict__ B,
                                 int absorb_right) {
    const WriteEntry e = ent[blockIdx.x];
    const SvdSector s = secs[e.sec];
    const double* J = ws + s.j_off;
    const double* V = ws + s.v_off;
    for (int idx = blockIdx.y * blockDim.x + threadIdx.x; idx < e.rows * e.cols; idx += gridDim.y * blockDim.x) {
        const int r = idx / e.cols, c = idx % e.cols;
        double v;
        if (e.left) {
            const int kc = kept[e.kept_off + c];                // J column index
            const double sk = sv[s.s_off + kc];
            const int row = e.vec_row0 + r;                      // row of M
            const double u = s.transposed ? V[(int64_t)kc * s.k + row] : J[(int64_t)kc * s.r + row] / sk;
            v = absorb_right ? u : u * sk;
            A[e.dst_off + idx] = v;
        } else {
            const int kc = kept[e.kept_off + r];
            const double sk = sv[s.s_off + kc];
            const int col = e.vec_row0 + c;                      // column of M
            const double w = s.transposed ? J[(int64_t)kc * s.r + col] / sk : V[(int64_t)kc * s.k + col];
            v = absorb_right ? w * sk : w;
            B[e.dst_off + idx] = v;
        }
    }
}

// One block meets the sweeps' grid barrier set up for two blocks (bar: counter, -, its error word): its wait must
// give up, and the workspace's flag is raised.
__global__ void barrier_selftest_kernel(unsigned int* bar, int* flag) {
    if (!grid_barrier(bar, 2u, reinterpret_cast<int*>(bar + 2)) && threadIdx.x == 0) atomicExch(flag, 1);
}

}  // namespace

void heff::svd_barrier_selftest(unsigned int* bar, int* flag, void* stream) {
    barrier_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(bar, flag);
}

extern "C" int heff_svd_create(const heff_layout* x, heff_svd** out) {
    heff::clear_error();
    if (!x || !out) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_create: null argument");
    *out = nullptr;
    if (x->idx.size() != 4) return fail(HEFF_ERR_CHARGE_MISMATCH, "x must have order 4");
    const heff::IndexDesc &al = x->idx[0], &p1 = x->idx[1], &p2 = x->idx[2], &be = x->idx[3];
    heff_svd* S = new (std::nothrow) heff_svd();
    if (!S) return fail(HEFF_ERR_OOM, "out of host memory");
    S->nq = x->nq;
    S->alpha_dims = al.dims;
    S->beta_dims = be.dims;
    try {
        std::map<std::vector<int32_t>, int> qid;
        std::vector<std::map<std::pair<int, int>, int32_t>> rpos, cpos;
        // sectors from the x blocks: Q = q(a) + q(s1)
        for (size_t b = 0; b < x->offsets.size(); ++b) {
            const int i = x->keys[b * 4], s1 = x->keys[b * 4 + 1], s2 = x->keys[b * 4 + 2], j = x->keys[b * 4 + 3];
            std::vector<int32_t> q = al.q(i);
            for (int c = 0; c < x->nq; ++c) q[c] += p1.charges[s1 * x->nq + c];
            auto it = qid.find(q);
            int id;
            if (it == qid.end()) {
                id = (int)S->Q.size();
                qid[q] = id;
                S->Q.push_back(q);
                S->rows.emplace_back();
                S->cols.emplace_back();
                rpos.emplace_back();
                cpos.emplace_back();
            } else {
                id = it->second;
            }
            if (!rpos[id].count({i, s1})) { rpos[id][{i, s1}] = 0; S->rows[id].push_back({i, s1, 0}); }
            if (!cpos[id].count({s2, j})) { cpos[id][{s2, j}] = 0; S->cols[id].push_back({s2, j, 0}); }
            (void)p2;
        }
        const int nsec = (int)S->Q.size();
        S->mrows.assign(nsec, 0);
        S->ncols.assign(nsec, 0);
        int64_t o = 0, so = 0, o32 = 0;
        for (int q = 0; q < nsec; ++q) {
            std::sort(S->rows[q].begin(), S->rows[q].end());
            std::sort(S->cols[q].begin(), S->cols[q].end());
            int32_t r = 0;
            for (auto& t : S->rows[q]) { std::get<2>(t) = r; rpos[q][{std::get<0>(t), std::get<1>(t)}] = r; r += al.dims[std::get<0>(t)]; }
            int32_t c = 0;
            for (auto& t : S->cols[q]) { std::get<2>(t) = c; cpos[q][{std::get<0>(t), std::get<1>(t)}] = c; c += be.dims[std::get<1>(t)]; }
            S->mrows[q] = r;
            S->ncols[q] = c;
            SvdSector sc{};
            sc.transposed = c > r;
            sc.r = sc.transposed ? c : r;
            sc.k = sc.transposed ? r : c;
            sc.j_off = o; o += (int64_t)sc.r * sc.k;
            sc.v_off = o; o += (int64_t)sc.k * sc.k;
            sc.g_off = o; o += (int64_t)sc.k * sc.k;
            sc.w_off = o; o += (int64_t)sc.r * sc.k;
            sc.j32_off = o32; o32 += (int64_t)sc.r * sc.k;
            sc.v32_off = o32; o32 += (int64_t)sc.k * sc.k;
            sc.s_off = (int32_t)so; so += sc.k;
            S->sec.push_back(sc);
            // FP64 GEMMs on column-major matrices, as row-major products of transposes:
            // G[i][j] = sum_l V[l,i] V[l,j]
            {
                heff::BProd p{};
                p.a_off = sc.v_off; p.a_rs = sc.k; p.a_cs = 1;
                p.b_off = sc.v_off; p.b_rs = 1; p.b_cs = sc.k;
                p.K = sc.k; p.c1 = -1; p.c2 = -1;
                S->gram.add_block(sc.g_off, sc.k, sc.k, sc.k, {p});
            }
            // W = V G (column-major W[i,j] = row j, column i of W^T): W^T[j][i] = sum_l G[l,j] V[i,l]
            {
                heff::BProd p{};
                p.a_off = sc.g_off; p.a_rs = sc.k; p.a_cs = 1;
                p.b_off = sc.v_off; p.b_rs = sc.k; p.b_cs = 1;
                p.K = sc.k; p.c1 = -1; p.c2 = -1;
                S->vg.add_block(sc.w_off, sc.k, sc.k, sc.k, {p});
            }
            // W = J V (r x k): W^T[j][i] = sum_l V[l,j] J[i,l]
            {
                heff::BProd p{};
                p.a_off = sc.v_off; p.a_rs = sc.k; p.a_cs = 1;
                p.b_off = sc.j_off; p.b_rs = sc.r; p.b_cs = 1;
                p.K = sc.k; p.c1 = -1; p.c2 = -1;
                S->jv.add_block(sc.w_off, sc.r, sc.k, sc.r, {p});
            }
            S->max_k = std::max(S->max_k, sc.k);
        }
        S->s_total = so;
        // load table: [sector, x_off, m_rows, n_cols, row0, col0] per x block
        std::vector<int64_t> tab;
        for (size_t b = 0; b < x->offsets.size(); ++b) {
            const int i = x->keys[b * 4], s1 = x->keys[b * 4 + 1], s2 = x->keys[b * 4 + 2], j = x->keys[b * 4 + 3];
            std::vector<int32_t> q = al.q(i);
            for (int c = 0; c < x->nq; ++c) q[c] += p1.charges[s1 * x->nq + c];
            const int id = qid[q];
            tab.insert(tab.end(), {(int64_t)id, x->offsets[b], (int64_t)al.dims[i], (int64_t)be.dims[j],
                                   (int64_t)rpos[id][{i, s1}], (int64_t)cpos[id][{s2, j}]});
        }
        S->xoff.assign(1, tab);   // stash the load table (one entry)
        S->ws_doubles = o + so + 64;
        S->off_words = ((size_t)S->ws_doubles * sizeof(double) + tab.size() * sizeof(int64_t) + 255) / 256 * 256;
        S->off_f32 = (S->off_words + (size_t)(16 + 3 + 2 * (nsec + 1)) * sizeof(int) + 255) / 256 * 256;
        S->ws_bytes = S->off_f32 + (size_t)o32 * sizeof(float) + 1024;
    } catch (const std::bad_alloc&) {
        delete S;
        return fail(HEFF_ERR_OOM, "out of host memory in heff_svd_create");
    }
    *out = S;
    return HEFF_OK;
}

extern "C" int heff_svd_workspace_size(const heff_svd* S, size_t* bytes) {
    heff::clear_error();
    if (!S || !bytes) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_workspace_size: null argument");
    *bytes = S->ws_bytes;
    return HEFF_OK;
}

#define SVD_CK(call)                                                                                     \
    do {                                                                                                 \
        cudaError_t e_ = (call);                                                                         \
        if (e_ != cudaSuccess) return fail(HEFF_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_));    \
    } while (0)

extern "C" int heff_svd_compute(heff_svd* S, const double* x, void* workspace, size_t workspace_bytes,
                                void* stream, int32_t* sweeps_out) try {
    heff::clear_error();
    if (!S || !x) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_compute: null argument");
    if (!workspace || workspace_bytes < S->ws_bytes || reinterpret_cast<uintptr_t>(workspace) % 256)
        return fail(HEFF_ERR_WORKSPACE, "SVD workspace of %zu bytes, needs %zu", workspace_bytes, S->ws_bytes);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double* ws = static_cast<double*>(workspace);
    double* sv = ws + (S->ws_doubles - S->s_total - 64);
    int* seen = reinterpret_cast<int*>(static_cast<char*>(workspace) + S->off_words);   // FP32 [0, 3), FP64 [3, 6); sweeps run [6, 8)
    const std::vector<int64_t>& tab = S->xoff[0];
    int64_t* d_tab = reinterpret_cast<int64_t*>(ws + S->ws_doubles);
    const int nsec = (int)S->sec.size();
    if (!S->d_sec) SVD_CK(cudaMalloc((void**)&S->d_sec, std::max<size_t>(1, S->sec.size()) * sizeof(SvdSector)));
    SVD_CK(cudaMemcpyAsync(S->d_sec, S->sec.data(), S->sec.size() * sizeof(SvdSector), cudaMemcpyHostToDevice, st));
    SVD_CK(cudaMemcpyAsync(d_tab, tab.data(), tab.size() * sizeof(int64_t), cudaMemcpyHostToDevice, st));
    const int ntab = (int)(tab.size() / 6);
    float* f32 = reinterpret_cast<float*>(static_cast<char*>(workspace) + S->off_f32);
    if (ntab) svd_load_kernel<<<dim3(std::min(ntab, 4096), COPY_SPLIT), 256, 0, st>>>(S->d_sec, d_tab, ntab, x, ws);
    svd_to_f32_kernel<<<dim3(128, nsec), 256, 0, st>>>(S->d_sec, ws, f32);
    heff::count_launches(2);
    if (!S->lists_uploaded) {
        int rc = HEFF_OK;
        for (heff::BList* b : {&S->gram, &S->vg, &S->jv})
            if (!rc) rc = heff::blist_upload(*b);
        if (rc) return rc;
        S->lists_uploaded = true;
    }
    // Jacobi sweeps until the largest off-diagonal measure is below a limit: one cooperative launch per phase
    const int kk_all = S->max_k + (S->max_k & 1);
    if (S->pair_off.empty()) {
        S->pair_off.push_back(0);
        for (const SvdSector& sc : S->sec) S->pair_off.push_back(S->pair_off.back() + (sc.k + (sc.k & 1)) / 2);
    }
    int* d_pair_off = seen + 16;
    unsigned int* d_bar = reinterpret_cast<unsigned int*>(d_pair_off + S->pair_off.size());
    int* d_err = reinterpret_cast<int*>(d_bar + 2);
    SVD_CK(cudaMemcpyAsync(d_pair_off, S->pair_off.data(), S->pair_off.size() * sizeof(int), cudaMemcpyHostToDevice,
                           st));
    SVD_CK(cudaMemsetAsync(d_bar, 0, 3 * sizeof(unsigned int), st));
    SVD_CK(cudaMemsetAsync(seen, 0, 8 * sizeof(int), st));
    int dev = 0, nsm = 0;
    SVD_CK(cudaGetDevice(&dev));
    SVD_CK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const SvdSector* secs = S->d_sec;
    int nsec_i = nsec;
    auto sweeps = [&](double* base, Sweeps sw) -> int {
        int per_sm = 0, kk_i = kk_all, ncols_i = (int)S->s_total;
        SVD_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, svd_sweep_kernel, SVD_SWEEP_NT, 0));
        // a pair to a block while SMs are free
        const int grid = std::max(1, std::min(nsm * std::max(per_sm, 1), S->pair_off.back()));
        double* nrm = sv;                                // the singular-value slots, free until the end
        void* args[] = {(void*)&secs, (void*)&nsec_i, (void*)&d_pair_off, (void*)&kk_i, (void*)&base,
                        (void*)&nrm, (void*)&ncols_i, (void*)&sw, (void*)&d_bar, (void*)&d_err};
        SVD_CK(cudaLaunchCooperativeKernel((const void*)svd_sweep_kernel, dim3(grid), dim3(SVD_SWEEP_NT), args, 0, st));
        heff::count_launches(1);
        return HEFF_OK;
    };
    // FP32 block sweeps: the same convergence test on the block pairs' Gram matrices
    auto block_sweeps = [&](float* base, Sweeps sw) -> int {
        std::vector<int> boff(1, 0);
        int nbb_all = 2, max_r = 0, per_sm = 0;
        for (const SvdSector& sc : S->sec) {
            const int nb = (sc.k + SVD_BW - 1) / SVD_BW, nbb = nb + (nb & 1);
            boff.push_back(boff.back() + nbb / 2);
            nbb_all = std::max(nbb_all, nbb);
            max_r = std::max(max_r, (int)sc.r);
        }
        int* d_boff = d_err + 2;
        SVD_CK(cudaMemcpyAsync(d_boff, boff.data(), boff.size() * sizeof(int), cudaMemcpyHostToDevice, st));
        // shared memory for the columns of a pair, where they fit (rows rounded up to the update's tiles)
        auto tiles = [](int rows) { return (rows + SVD_TR - 1) / SVD_TR * SVD_TR; };
        int rows_j = tiles(max_r);
        size_t smem = (size_t)(rows_j + tiles(S->max_k)) * SVD_TLD * sizeof(float);
        const bool res = smem <= SVD_RES_BYTES;
        if (!res) smem = (size_t)SVD_TR * SVD_TLD * sizeof(float);
        const auto kernel = res ? svd_block_sweep_kernel<true> : svd_block_sweep_kernel<false>;
        SVD_CK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    res ? (int)SVD_RES_BYTES : (int)smem));
        SVD_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, SVD_BT, smem));
        const int grid = std::max(1, std::min(nsm * std::max(per_sm, 1), boff.back()));
        void* args[] = {(void*)&secs, (void*)&nsec_i, (void*)&d_boff, (void*)&nbb_all, (void*)&base,
                        (void*)&sw, (void*)&d_bar, (void*)&d_err, (void*)&rows_j};
        SVD_CK(cudaLaunchCooperativeKernel((const void*)kernel, dim3(grid), dim3(SVD_BT), args, smem, st));
        heff::count_launches(1);
        return HEFF_OK;
    };
    int rc;
    // FP32 preconditioning sweeps.  A sweep's measure is taken before its rotations and Jacobi sweeps converge
    // quadratically: one that saw at most 1e-4 leaves FP32 rounding, and another would only confirm it.
    if ((rc = block_sweeps(f32, Sweeps{30, 1e-4f, seen, seen + 6}))) return rc;
    // V = orthonormalised double(V32), J = J V
    svd_v_to_f64_kernel<<<dim3(128, nsec), 256, 0, st>>>(S->d_sec, f32, ws);
    heff::count_launches(1);
    for (int it = 0; it < 2; ++it) {
        if ((rc = heff::launch_bgemm(S->gram, ws, ws, ws, nullptr, nullptr, 1.0, stream, d_err))) return rc;
        svd_residual_kernel<<<dim3(4, nsec), 256, 0, st>>>(S->d_sec, ws);
        heff::count_launches(1);
        if ((rc = heff::launch_bgemm(S->vg, ws, ws, ws, nullptr, nullptr, -0.5, stream, d_err))) return rc;
        svd_ns_kernel<<<dim3(128, nsec), 256, 0, st>>>(S->d_sec, ws);
        heff::count_launches(1);
    }
    if ((rc = heff::launch_bgemm(S->jv, ws, ws, ws, nullptr, nullptr, 1.0, stream, d_err))) return rc;
    svd_copy_w_kernel<<<dim3(128, nsec), 256, 0, st>>>(S->d_sec, ws);
    heff::count_launches(1);
    // FP64 sweeps to convergence: off-diagonal measure 1e-14, i.e. stop after the sweep that
    // saw at most 1e-7
    if (kk_all >= 2 && (rc = sweeps(ws, Sweeps{40, 1e-7f, seen + 3, seen + 7}))) return rc;
    svd_norms_kernel<<<dim3((S->max_k + 3) / 4 + 1, nsec), 128, 0, st>>>(S->d_sec, ws, sv);
    heff::count_launches(1);
    S->s.assign(S->s_total, 0.0);
    SVD_CK(cudaMemcpyAsync(S->s.data(), sv, S->s_total * sizeof(double), cudaMemcpyDeviceToHost, st));
    int state[8] = {0}, e = 0;
    SVD_CK(cudaMemcpyAsync(state, seen, sizeof state, cudaMemcpyDeviceToHost, st));
    SVD_CK(cudaMemcpyAsync(&e, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    SVD_CK(cudaStreamSynchronize(st));
    SVD_CK(cudaGetLastError());
    if (e) return fail(HEFF_ERR_TIMEOUT, "SVD sweep: grid barrier timed out");
    S->fp32_sweeps = state[6];
    S->fp64_sweeps = state[7];
    if (sweeps_out) *sweeps_out = S->fp64_sweeps;
    S->computed = true;
    S->kept.clear();
    return HEFF_OK;
} catch (const std::bad_alloc&) {
    return fail(HEFF_ERR_OOM, "out of host memory in heff_svd_compute");
}

extern "C" int heff_svd_info(const heff_svd* S, int32_t* fp32_sweeps, int32_t* fp64_sweeps) {
    heff::clear_error();
    if (!S) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_info: null argument");
    if (fp32_sweeps) *fp32_sweeps = S->fp32_sweeps;
    if (fp64_sweeps) *fp64_sweeps = S->fp64_sweeps;
    return HEFF_OK;
}

extern "C" int heff_svd_truncate(heff_svd* S, int32_t m_max, double cutoff, int32_t* nsec_out,
                                 int32_t* charges_out, int32_t* dims_out, double* discarded, double* norm) {
    heff::clear_error();
    if (!S || !nsec_out) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_truncate: null argument");
    if (!S->computed) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_truncate before heff_svd_compute");
    if (m_max < 1) return fail(HEFF_ERR_INVALID_ARG, "m_max must be >= 1");
    double tot = 0;
    for (double v : S->s) tot += v * v;
    const double nrm = std::sqrt(tot);
    S->norm = nrm;
    // candidates (normalised s, sector, rank inside the sector by decreasing s)
    struct Cand { double s; int sec; int rank; int col; };
    std::vector<Cand> cand;
    const int nsec = (int)S->sec.size();
    for (int q = 0; q < nsec; ++q) {
        const SvdSector& sc = S->sec[q];
        std::vector<int> idx(sc.k);
        std::iota(idx.begin(), idx.end(), 0);
        std::stable_sort(idx.begin(), idx.end(),
                         [&](int a, int b) { return S->s[sc.s_off + a] > S->s[sc.s_off + b]; });
        for (int r = 0; r < sc.k; ++r)
            cand.push_back({nrm > 0 ? S->s[sc.s_off + idx[r]] / nrm : 0.0, q, r, idx[r]});
    }
    double smax = 0;
    for (auto& c : cand) smax = std::max(smax, c.s);
    auto qabs = [&](int q) { long a = 0; for (int v : S->Q[q]) a += std::abs(v); return a; };
    // order: decreasing s (ties within 1e-12 s_max), then |Q|, Q, rank inside the sector
    std::stable_sort(cand.begin(), cand.end(), [&](const Cand& a, const Cand& b) {
        const double ka = std::nearbyint(a.s / std::max(smax, 1e-300) / 1e-12);
        const double kb = std::nearbyint(b.s / std::max(smax, 1e-300) / 1e-12);
        if (ka != kb) return ka > kb;
        if (qabs(a.sec) != qabs(b.sec)) return qabs(a.sec) < qabs(b.sec);
        if (S->Q[a.sec] != S->Q[b.sec]) return S->Q[a.sec] < S->Q[b.sec];
        return a.rank < b.rank;
    });
    S->kept.assign(nsec, {});
    std::vector<std::vector<std::pair<int, int>>> kr(nsec);   // (rank, col)
    double kept2 = 0, all2 = 0;
    int nk = 0;
    for (auto& c : cand) {
        all2 += c.s * c.s;
        if (c.s >= cutoff && nk < m_max) {
            kr[c.sec].push_back({c.rank, c.col});
            kept2 += c.s * c.s;
            ++nk;
        }
    }
    // new bond: sectors with at least one kept value, in increasing charge order
    std::vector<int> order(nsec);
    std::iota(order.begin(), order.end(), 0);
    std::sort(order.begin(), order.end(), [&](int a, int b) { return S->Q[a] < S->Q[b]; });
    int ns = 0;
    for (int q : order) {
        if (kr[q].empty()) continue;
        std::sort(kr[q].begin(), kr[q].end());
        for (auto& rc : kr[q]) S->kept[q].push_back(rc.second);
        if (charges_out) std::memcpy(charges_out + ns * S->nq, S->Q[q].data(), sizeof(int32_t) * S->nq);
        if (dims_out) dims_out[ns] = (int32_t)kr[q].size();
        ++ns;
    }
    *nsec_out = ns;
    S->discarded = all2 - kept2;
    if (discarded) *discarded = S->discarded;
    if (norm) *norm = nrm;
    return HEFF_OK;
}

extern "C" int heff_svd_singular_values(const heff_svd* S, double* out) {
    heff::clear_error();
    if (!S || !out) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_singular_values: null argument");
    std::vector<int> order(S->sec.size());
    std::iota(order.begin(), order.end(), 0);
    std::sort(order.begin(), order.end(), [&](int a, int b) { return S->Q[a] < S->Q[b]; });
    int64_t n = 0;
    for (int q : order)
        if (q < (int)S->kept.size())
            for (int c : S->kept[q]) out[n++] = S->s[S->sec[q].s_off + c];
    return HEFF_OK;
}

extern "C" int heff_svd_write(heff_svd* S, const heff_layout* A_layout, const heff_layout* B_layout, double* A,
                              double* B, int32_t absorb_right, void* workspace, size_t workspace_bytes,
                              void* stream) {
    heff::clear_error();
    if (!S || !A_layout || !B_layout || !A || !B) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_write: null argument");
    if (S->kept.empty()) return fail(HEFF_ERR_INVALID_ARG, "heff_svd_write before heff_svd_truncate");
    if (!workspace || workspace_bytes < S->ws_bytes) return fail(HEFF_ERR_WORKSPACE, "SVD workspace too small");
    if (A_layout->idx.size() != 3 || B_layout->idx.size() != 3)
        return fail(HEFF_ERR_CHARGE_MISMATCH, "left/right tensors must have order 3");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double* ws = static_cast<double*>(workspace);
    double* sv = ws + (S->ws_doubles - S->s_total - 64);
    // new bond sector number for each kept sector (charge order)
    std::map<std::vector<int32_t>, int> bond;
    const heff::IndexDesc& nb = A_layout->idx[2];
    for (int c = 0; c < nb.nsec; ++c) bond[nb.q(c)] = c;
    std::vector<WriteEntry> ents;
    std::vector<int32_t> keptflat;
    std::vector<int32_t> koff(S->sec.size(), 0);
    for (size_t q = 0; q < S->sec.size(); ++q) {
        koff[q] = (int32_t)keptflat.size();
        keptflat.insert(keptflat.end(), S->kept[q].begin(), S->kept[q].end());
    }
    for (size_t q = 0; q < S->sec.size(); ++q) {
        if (S->kept[q].empty()) continue;
        auto bit = bond.find(S->Q[q]);
        if (bit == bond.end() || nb.dims[bit->second] != (int)S->kept[q].size())
            return fail(HEFF_ERR_CHARGE_MISMATCH, "left tensor bond does not match the truncation");
        const int c = bit->second, nkeep = (int)S->kept[q].size();
        for (auto& t : S->rows[q]) {            // A block (i, s1, c)
            const int64_t off = A_layout->offset_of({std::get<0>(t), std::get<1>(t), c});
            if (off < 0) return fail(HEFF_ERR_CHARGE_MISMATCH, "left tensor block missing");
            ents.push_back({off, S->alpha_dims[std::get<0>(t)], nkeep, (int32_t)q, std::get<2>(t), koff[q], 1});
        }
        for (auto& t : S->cols[q]) {            // B block (c, s2, j)
            const int64_t off = B_layout->offset_of({c, std::get<0>(t), std::get<1>(t)});
            if (off < 0) return fail(HEFF_ERR_CHARGE_MISMATCH, "right tensor block missing");
            ents.push_back({off, nkeep, S->beta_dims[std::get<1>(t)], (int32_t)q, std::get<2>(t), koff[q], 0});
        }
    }
    // the write tables (sized by the truncation) go to temporary device buffers
    WriteEntry* d_ent = nullptr;
    int32_t* d_kept = nullptr;
    SVD_CK(cudaMalloc((void**)&d_ent, std::max<size_t>(1, ents.size()) * sizeof(WriteEntry)));
    SVD_CK(cudaMalloc((void**)&d_kept, std::max<size_t>(1, keptflat.size()) * sizeof(int32_t)));
    SVD_CK(cudaMemcpyAsync(d_ent, ents.data(), ents.size() * sizeof(WriteEntry), cudaMemcpyHostToDevice, st));
    SVD_CK(cudaMemcpyAsync(d_kept, keptflat.data(), keptflat.size() * sizeof(int32_t), cudaMemcpyHostToDevice, st));
    if (!ents.empty())
        svd_write_kernel<<<dim3((unsigned)ents.size(), COPY_SPLIT), 256, 0, st>>>(S->d_sec, d_ent, d_kept, ws, sv, A, B, absorb_right);
    heff::count_launches(1);
    SVD_CK(cudaStreamSynchronize(st));
    cudaFree(d_ent);
    cudaFree(d_kept);
    SVD_CK(cudaGetLastError());
    return HEFF_OK;
}

extern "C" void heff_svd_destroy(heff_svd* S) {
    if (!S) return;
    cudaFree(S->d_sec);
    heff::blist_free(S->gram);
    heff::blist_free(S->vg);
    heff::blist_free(S->jv);
    delete S;
}
