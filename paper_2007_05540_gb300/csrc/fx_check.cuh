// Which outputs of a fixed-point product the digits resolve, and the others in FP64 arithmetic.
//
// The digits of a row hold 62 bits below the row's scale A = 2^(E - 1022), so the error of an output depends on the
// scales of its row and its column, while that of a running FP64 sum depends on the terms, n 2^-53 S with
// S = sum |a||b| over its n terms.  In units of A B 2^-62 an output's error is at most
//   |a|_1 / A + |b|_1 / B    what the truncation of the elements takes, and
//   7 n                      the digit products i + j >= 8; of the digits of real numbers (their products have either
//                            sign and a standard deviation of 0.9 a term) 6 sqrt(n) is not passed,
// so that the digits' error stays below that of the FP64 sum where
//   S >= A B max(2^-9 (|a|_1 / A + |b|_1 / B) / n, 2^-6 / sqrt(n)).
// Where large elements of the row meet small ones of the column only (operands graded against each other, a row
// with one element, as the identity channel of an environment has), S may be less: such an output is computed in FP64.
//
// A kernel before each product kernel decides, a warp for a patch of 32 rows (one per lane) and 32 columns, computes such
// outputs and leaves a bit for each, by which the product kernel keeps them.  It adds |a||b| itself, the
// magnitudes as BF16 rounded down, on mma.sync, 16 contraction elements at a time, until every output has passed: one
// to three steps for dense operands.  Bound by the latency of a step's loads and, for sparse rows, by the FP64 units.
// What it costs: apply m = 1024, k = 14, 398 -> 466 us (15000 patches checked and 3000 sparse ones before GEMM 1, 31 us;
// 4300 before GEMM 2, 41 us), environment update m = 1024 253 -> 315 us, Lanczos m = 48 62 -> 66 us a step.
// Tried and left: the same in the warps that drain the digit sums (it is on the path of every tile there: GEMM 1
// of the apply at m = 1024, k = 14, 163 -> 254 us); |a||b| by shuffles and multiply-adds (1000 instructions a step instead of
// 180); bounds from minima and sums of 32 elements (a thirtieth of S on average).
#pragma once

#include "fixed.cuh"

namespace heff {
namespace fx {

// |v| / 2^(E - 1022) from the upper word of v, rounded down (0 for subnormals); base = (E - 126) 2^20
__device__ __forceinline__ int magnitude_base(int E) { return min(max(E - 126, 0), 2047) << 20; }
__device__ __forceinline__ uint32_t magnitude(double v, int base) {
    return (uint32_t)max((int)((uint32_t)__double2hiint(v) & 0x7fffffffu) - base, 0) << 3;
}

// One piece of a patch's contraction: element k of a row at a[k as], of column c at b[c bcs + k bs].
struct Piece {
    const double *a, *b;
    int64_t bcs;
    int as, bs, K;
    double coef;
};

// A patch, as its kernel describes it (Src):
//   pieces()           pieces of the contraction
//   piece(i, r)        piece i of row r
//   bias(i)            power of two of the piece's coefficient, or NO_TERM
//   words(i, j, a, b)  which of the elements 32 j .. of piece i are not zero: of row `lane`, of column `lane`
//   store(c, v)        an output of row `lane`
//   DENSE              elements of a row and of a column lie one after another, on 16 bytes, pieces a multiple of 16
// nrow, ncol: rows and columns of the patch.
constexpr int NO_TERM = -(1 << 20);

// The outputs (bits: columns) of this lane's row whose S stays below least times the scales Ea (of row `lane`)
// and Eb (of column `lane`).  rows, cols: those that have nonzero elements.
template <class Src>
__device__ __forceinline__ uint32_t weak_outputs(const Src& src, int nrow, int ncol, uint32_t rows, uint32_t cols, int Ea,
                                                 int Eb, float least) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    // acc[r][c][j]: row 16 r + 8 (j / 2) + g, column 8 c + 2 t + j % 2; A rows 8 x + g, B columns 8 x + g
    float acc[2][4][4];
    int ea[4], eb[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        ea[x] = __shfl_sync(0xffffffffu, Ea, 8 * x + g);
        eb[x] = magnitude_base(__shfl_sync(0xffffffffu, Eb, 8 * x + g));
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int row = 16 * r + 8 * (j >> 1) + g, col = 8 * c + 2 * t + (j & 1);
                acc[r][c][j] = ((rows >> row) & (cols >> col) & 1u) ? 0.f : 1.f;
            }
    auto pack = [](double2 v, int base) { return __byte_perm(magnitude(v.x, base), magnitude(v.y, base), 0x7632); };
    // (all loads of a step are issued before the first is used, without branches between them)
    auto load = [](const double* p, int step, int left) -> double2 {
        if constexpr (Src::DENSE) return __ldg(reinterpret_cast<const double2*>(p));
        return make_double2(left > 0 ? __ldg(p) : 0.0, left > 1 ? __ldg(p + step) : 0.0);
    };
    const int np = src.pieces();
    bool done = false;
    // (from the middle on: the pieces go by charge, and the outer sectors are the smallest)
    for (int n = 0, i = np / 2; n < np && !done; ++n, i = i + 1 < np ? i + 1 : 0) {
        const int bias = src.bias(i);
        if (bias == NO_TERM) continue;                            // warp-uniform
        const Piece q = src.piece(i, g);
        const double* a[4];
        const double* b[4];
        int ba[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            a[x] = src.piece(i, min(8 * x + g, nrow - 1)).a + (int64_t)(2 * t) * q.as;
            b[x] = q.b + (int64_t)min(8 * x + g, ncol - 1) * q.bcs + (int64_t)(2 * t) * q.bs;
            ba[x] = magnitude_base(ea[x] - bias);
        }
        for (int k0 = 0; k0 < q.K && !done; k0 += 16) {
            double2 va[4][2], vb[4][2];
            uint32_t fa[4][2], fb[4][2];
            const int left = q.K - k0 - 2 * t;
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    va[x][y] = load(a[x] + (int64_t)(k0 + 8 * y) * q.as, q.as, left - 8 * y);
                    vb[x][y] = load(b[x] + (int64_t)(k0 + 8 * y) * q.bs, q.bs, left - 8 * y);
                }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y < 2; ++y) {
                    fa[x][y] = pack(va[x][y], ba[x]);
                    fb[x][y] = pack(vb[x][y], eb[x]);
                }
            float low = 1.f;
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float (&d)[4] = acc[r][c];
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                        "{%0, %1, %2, %3};"
                        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                        : "r"(fa[2 * r][0]), "r"(fa[2 * r + 1][0]), "r"(fa[2 * r][1]), "r"(fa[2 * r + 1][1]),
                          "r"(fb[c][0]), "r"(fb[c][1]));
#pragma unroll
                    for (int j = 0; j < 4; ++j) low = fminf(low, d[j]);
                }
            done = __all_sync(0xffffffffu, low >= least);
        }
    }
    if (done) return 0;
    uint32_t weak = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            uint32_t mine = 0;                                    // this lane's row: group lane / 8, g = lane % 8
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t w = __ballot_sync(0xffffffffu, !(acc[x >> 1][c][2 * (x & 1) + j] >= least));
                mine = lane >> 3 == x ? w : mine;
            }
            mine = (mine >> (4 * (lane & 7))) & 0xfu;
            weak |= ((mine & 1u) | (mine & 2u) << 1 | (mine & 4u) << 2 | (mine & 8u) << 3) << (8 * c + j);
        }
    return weak;
}

// The bound's factor for rows and columns of at least n nonzero elements whose sums are at most sa and sb
// times their scales.
__device__ __forceinline__ float least_sum(float n, float sa, float sb) {
    return fmaxf((fminf(sa, n) + fminf(sb, n)) / (512.f * n), rsqrtf(n) * (1.f / 64));
}

// Up to two elements of a row or a column: piece and place.
struct Few {
    int i[2], k[2];
    __device__ __forceinline__ void find(int piece, int block, uint32_t bits, int& n) {
        while (bits && n < 2) {
            const int k_ = 32 * block + __ffs(bits) - 1;
            if (n == 0) { i[0] = piece; k[0] = k_; } else { i[1] = piece; k[1] = k_; }
            ++n;
            bits &= bits - 1;
        }
    }
};

// A patch whose rows (ROWS) or columns have two nonzero elements at most, all its outputs: two gathers and
// multiply-adds an output, eight outputs in flight.
template <bool ROWS, int CB, class Src>
__device__ __forceinline__ void sparse_outputs(const Src& src, bool rowed, int ncol) {
    const int lane = threadIdx.x & 31;
    Few e{{0, 0}, {0, 0}};
    int n = 0;
    const int np = src.pieces();
    for (int i = 0; i < np; ++i) {
        const int nb = (src.piece(i, 0).K + 31) / 32;
        for (int j0 = 0; j0 < nb; j0 += 4) {
            uint32_t z[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                uint32_t za = 0, zb = 0;
                if (j0 + j < nb) src.words(i, j0 + j, za, zb);
                z[j] = ROWS ? za : zb;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) e.find(i, j0 + j, z[j], n);
        }
    }
    const int most = __reduce_max_sync(0xffffffffu, n);
    double mine[2];                                       // this lane's elements
    const double* to[2];                                  // ROWS: what they multiply, column 0
    int64_t step[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const Piece q = src.piece(e.i[t], lane);
        mine[t] = 0.0;
        to[t] = q.b + (int64_t)e.k[t] * q.bs;
        step[t] = q.bcs;
        if (t < n) mine[t] = ROWS ? q.coef * __ldg(q.a + (int64_t)e.k[t] * q.as) : __ldg(to[t] + lane * q.bcs);
    }
    for (int c0 = 0; c0 < ncol; c0 += CB) {
        double v[CB];
#pragma unroll
        for (int c = 0; c < CB; ++c) v[c] = 0.0;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            if (t >= most) break;
            double f[CB];
#pragma unroll
            for (int c = 0; c < CB; ++c) {
                const int col = min(c0 + c, ncol - 1);
                if (ROWS) {
                    f[c] = __ldg(to[t] + col * step[t]);
                } else {
                    const Piece q = src.piece(__shfl_sync(0xffffffffu, e.i[t], col), lane);
                    const int k = __shfl_sync(0xffffffffu, e.k[t], col);
                    f[c] = rowed ? q.coef * __ldg(q.a + (int64_t)k * q.as) : 0.0;
                }
            }
#pragma unroll
            for (int c = 0; c < CB; ++c)
                v[c] = fma(ROWS ? mine[t] : __shfl_sync(0xffffffffu, mine[t], min(c0 + c, ncol - 1)), f[c], v[c]);
        }
        if (rowed)
#pragma unroll
            for (int c = 0; c < CB; ++c)
                if (c0 + c < ncol) src.store(c0 + c, v[c]);
    }
}

// The outputs `need` (bits: columns) of this lane's row in FP64.  all: as running sums (a row or a column holds
// infinities, NaNs or magnitudes near the ends of the range: what an intermediate sum does matters).
template <class Src>
__device__ __forceinline__ void fp64_outputs(const Src& src, bool rowed, int ncol, uint32_t need, bool all) {
    const int lane = threadIdx.x & 31, np = src.pieces();
    for (int c0 = 0; c0 < ncol; c0 += 8) {
        const uint32_t here = (need >> c0) & 0xffu;
        const int count = __reduce_add_sync(0xffffffffu, __popc(here));
        if (count == 0) continue;
        if (!all && count <= 64) {
            // a few: four at a time, the lanes along the contraction (four of K = 200 take 1700 cycles, eight
            // columns of all rows 26000)
            uint32_t rows = __ballot_sync(0xffffffffu, here != 0), cols = 0;
            int r = 0;
            for (int done = 0; done < count; done += 4) {
                int row[4], col[4];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    if (cols == 0 && rows) {
                        r = __ffs(rows) - 1;
                        rows &= rows - 1;
                        cols = __shfl_sync(0xffffffffu, here, r);
                    }
                    row[o] = r;                           // (past the last one: that one again)
                    col[o] = cols ? c0 + __ffs(cols) - 1 : col[o > 0 ? o - 1 : 0];
                    cols &= cols - 1;
                }
                double v[4] = {0.0, 0.0, 0.0, 0.0};
                for (int i = 0; i < np; ++i) {
                    const double *a[4], *b[4];
                    const Piece q = src.piece(i, 0);
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        a[o] = src.piece(i, row[o]).a;
                        b[o] = q.b + col[o] * q.bcs;
                    }
#pragma unroll 2
                    for (int k = lane; k < q.K; k += 32)
#pragma unroll
                        for (int o = 0; o < 4; ++o)
                            v[o] = fma(q.coef * __ldg(a[o] + (int64_t)k * q.as), __ldg(b[o] + (int64_t)k * q.bs), v[o]);
                }
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    for (int x = 16; x > 0; x >>= 1) v[o] += __shfl_xor_sync(0xffffffffu, v[o], x);
                    if (lane == row[o] && done + o < count) src.store(col[o], v[o]);
                }
            }
            continue;
        }
        // many: the lanes along the rows
        double v[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) v[c] = 0.0;
        for (int i = 0; i < np; ++i) {
            const Piece q = src.piece(i, lane);
            const double* b[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) b[c] = q.b + (int64_t)min(c0 + c, ncol - 1) * q.bcs;
            for (int k0 = 0; k0 < q.K; k0 += 2) {
                double a[2], f[2][8];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const bool in = k0 + e < q.K;
                    a[e] = in && rowed ? q.coef * __ldg(q.a + (int64_t)(k0 + e) * q.as) : 0.0;
#pragma unroll
                    for (int c = 0; c < 8; ++c) f[e][c] = in ? __ldg(b[c] + (int64_t)(k0 + e) * q.bs) : 0.0;
                }
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int c = 0; c < 8; ++c) v[c] = fma(a[e], f[e][c], v[c]);
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if ((here >> c) & 1u) src.store(c0 + c, v[c]);
    }
}

}  // namespace fx
}  // namespace heff
