// FP64 block products on the sm_103a tensor cores: fixed-point digits on the FP16 pipe.
//
// GB300 does about two FP64 multiply-adds per SM and clock (1.2 TFLOP/s in all), while its FP16
// tensor pipe does about 4000.  So a product of FP64 operands is computed here from integer
// digits, the error-free splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012):
// every row of A and every column of B gets one scale (a power of two from its largest
// element), each element becomes a 62-bit fixed-point number of eight signed 8-bit digits
// (fixed.cuh), and
//   C = sum_g 2^(-8 g) sum_{i + j = g} A_i B_j^T,      g = 0 .. 7,
// where the digit planes A_i, B_j are FP16 operands of tcgen05 MMAs.  The 36 digit products of a
// K step land in 8 accumulators (one per g) in tensor memory.  All sums that matter at FP64
// precision are exact: a digit product is at most 2^14, and a chunk of 256 contraction steps
// keeps the accumulators g <= 4 below 2^24, where FP32 adds integers exactly; the later ones
// weigh 2^-40 and less (5 and 6 leave FP32's integers only where the digits of a whole chunk are alike and near
// their largest value).  After each chunk the accumulators are added into 96-bit integers, and
// the sum is rounded to FP64 once at the end.  What is dropped is the part of an element below
// 2^-62 of its row's scale, and the digit products g >= 8: in all under 9 2^-62 K of the two scales' product, a
// bound by the largest elements of the row and the column.  Outputs whose terms are so small against the scales that
// this is more than the error of a running FP64 sum are found and computed in FP64 (fx_check.cuh).
//
// Rows that the scale cannot hold (infinities, NaNs, magnitudes beyond 2^+-400) make their tile
// run in FP64 arithmetic on the CUDA cores inside the same kernel.
//
// The work is lists of block products with arbitrary strides and scalar coefficients: gradients, two-site
// tensor, the SVD's products.  (The matvec's and the environment update's operands are converted once:
// fx_planes.cu.)
//
// One persistent CTA per SM, 128 x 64 output tiles, 20 warps:
//   warps 0-7    producers: load 128 + 64 rows x 16 K of FP64, convert to digits, write the FP16
//                planes into the 64-byte-swizzled K-major layout (a ring of 4 steps, 48 KB each)
//   warps 8-15   drain: 8 accumulators -> 96-bit integers in registers -> FP64 -> global
//   warp 16      allocates the 512 tensor-memory columns; one thread issues the MMAs: digit
//                plane A_i times the planes B_0 .. B_{7-i}, which lie one after another in shared
//                memory and so are one wide B operand, whose products go to the accumulators
//                i .. 7, which lie one after another in tensor memory
// Registers are moved from the other warps to the drain warps (96 integers a thread).
//
// Bound by the producers' conversions (1.9 us per step of 16 contraction elements, where the tensor pipe needs
// 0.6).  Against the FP64 units (64 x 64 tiles on the CUDA cores): gradients m = 320, 9.2 -> 1.44 ms a call, 0.14 of
// it for weak_list_kernel.
// Every mbarrier wait is bounded; on expiry the CTA raises the error flag, stops issuing work,
// waits (bounded) for its MMAs in flight, frees its tensor memory and returns.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "fixed.cuh"
#include "fx_check.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace heff {
namespace {

using namespace ptx;

constexpr int FM = FX_TILE_M, FN = FX_TILE_N;     // output tile
constexpr int FKS = 16;                           // contraction elements per step
constexpr int FD = 8;                             // digits
constexpr int FST = 4;                            // steps in the ring (two per 64-byte K block)
constexpr int FCH = 16;                           // steps per exact accumulation chunk (256 elements)
constexpr int PW = 8, EW = 8;                     // producer and drain warps
constexpr int FTHREADS = 32 * (PW + EW + 4);      // + the MMA warp's warpgroup
constexpr int A_PLANE = FM * 64;                  // one digit plane of A, 32 K elements
constexpr int A_BLK = FD * A_PLANE;               // 64 KB
constexpr int B_BLK = FD * FN * 64;               // 32 KB
constexpr int BLK = A_BLK + B_BLK;
constexpr int OFF_TR = (FST / 2) * BLK;           // drain transposes: 32 rows x 8 columns per warp
constexpr int TR_WARP = 32 * 9 * 8;
constexpr int OFF_DF = OFF_TR + EW * TR_WARP;     // FP64 tiles: 8 K x (64 + 1) for A and for B
constexpr int OFF_E = OFF_DF + 2 * 8 * 65 * 8;    // row and column scales, two tiles
constexpr int OFF_BAR = OFF_E + 2 * (FM + FN + PW) * 4;
constexpr int FSMEM = OFF_BAR + 256 + 1024;
static_assert(FSMEM <= 227 * 1024, "shared memory of one CTA");
// register split (per thread): producers, drain, MMA warpgroup; the kernel is compiled for
// R_ALL, and each SM partition holds two producer, two drain and one other warp
constexpr int R_ALL = 96, R_PROD = 80, R_DRAIN = 136, R_MMA = 48;
static_assert(2 * R_PROD + 2 * R_DRAIN + R_MMA <= 5 * R_ALL, "registers of a partition");

struct FxArgs {
    const BTile* tiles;
    const BProd* prods;
    const uint16_t* e;                   // exponent codes per operand row (BProd.ea, eb)
    const float* sums;                   // sum of its magnitudes over the code's power of two
    const uint32_t* words;               // and words of its nonzero elements (BProd.za, zb)
    uint32_t* fp64;                      // outputs computed in FP64 (BTile.fp64_at)
    const double *coef1, *coef2, *inv_scale;
    double scale;
    int accumulate;
    int ntiles;
    const double *A, *B;
    double* C;
    int* err;
};

// round i of this CTA: a snake over the sorted tiles
__device__ __forceinline__ long item_of(long i) {
    const long G = gridDim.x, c = blockIdx.x;
    return i * G + ((i & 1) ? G - 1 - c : c);
}

__device__ __forceinline__ double prod_coef(const FxArgs& g, const BProd& p) {
    return (p.c1 < 0 ? 1.0 : g.coef1[p.c1]) * (p.c2 < 0 ? 1.0 : g.coef2[p.c2]);
}

// Scale of row r of A (side 0) or column r of B (side 1) over the tile's products; ok: cleared
// when the row needs FP64.
__device__ __forceinline__ int row_scale(const FxArgs& g, const BTile& t, int side, int r, bool& ok) {
    int E = 0;
    for (int s = 0; s < t.prod_count; ++s) {
        const BProd& p = g.prods[t.prod_begin + s];
        int v = g.e[(side ? p.eb : p.ea) + r];
        if (side == 0 && (p.c1 >= 0 || p.c2 >= 0)) {
            const double c = prod_coef(g, p);
            const int ec = fx::exp_code((uint32_t)__double2hiint(c), (uint32_t)__double2loint(c));
            if (ec == 0x7ff) ok = false;
            // |c v| < 2^(ec - 1022) 2^(v - 1022)
            v = (v == 0 || ec == 0) && v != 0x7ff ? 0 : (v == 0x7ff ? v : max(v + ec - 1022, 1));
        }
        E = max(E, v);
    }
    if (!fx::exp_plain(E)) ok = false;
    return E ? E : fx::E_ZERO;
}

// A patch of a tile, as fx_check.cuh reads it: one piece per product.
struct ListSrc {
    static constexpr bool DENSE = false;
    const FxArgs& g;
    const BTile& t;
    int r0, c0;                          // the patch's first row and column in the tile
    bool rowed, coled;                   // whether there is a row, a column `lane`
    double scale;
    __device__ __forceinline__ int lane() const { return threadIdx.x & 31; }
    __device__ __forceinline__ const BProd& prod(int i) const { return g.prods[t.prod_begin + i]; }
    __device__ __forceinline__ int pieces() const { return t.prod_count; }
    __device__ __forceinline__ fx::Piece piece(int i, int r) const {
        const BProd& q = prod(i);
        return {g.A + q.a_off + (int64_t)(r0 + r) * q.a_rs, g.B + q.b_off + (int64_t)c0 * q.b_cs, q.b_cs, q.a_cs, q.b_rs,
                q.K, prod_coef(g, q)};
    }
    __device__ __forceinline__ int bias(int i) const {
        const BProd& q = prod(i);
        if (q.c1 < 0 && q.c2 < 0) return 0;
        const double c = prod_coef(g, q);
        const int ec = fx::exp_code((uint32_t)__double2hiint(c), (uint32_t)__double2loint(c));
        return ec > 1 ? ec - 1023 : fx::NO_TERM;
    }
    __device__ __forceinline__ void words(int i, int j, uint32_t& x, uint32_t& y) const {
        const BProd& q = prod(i);
        x = rowed ? g.words[q.za + (int64_t)j * q.na + r0 + lane()] : 0u;
        y = coled ? g.words[q.zb + (int64_t)j * q.nb + c0 + lane()] : 0u;
    }
    __device__ __forceinline__ void store(int c, double v) const {
        double* o = g.C + t.c_off + (int64_t)(r0 + lane()) * t.ldc + c0 + c;
        *o = g.accumulate ? *o + scale * v : scale * v;
    }
};

// The outputs that the digits do not resolve (fx_check.cuh): a block per tile, a warp per patch.
constexpr int WEAK_WARPS = 4;
__global__ void __launch_bounds__(32 * WEAK_WARPS) weak_list_kernel(const __grid_constant__ FxArgs g) {
    const BTile t = g.tiles[blockIdx.x];
    const int lane = threadIdx.x & 31, wpr = (t.n + 31) / 32, patches = (t.m + 31) / 32 * wpr;
    const double scale = g.inv_scale ? g.scale / g.inv_scale[0] : g.scale;
    auto power = [](int e) { return e >= -126 ? __int_as_float((127 + e) << 23) : 0.f; };
    for (int p = threadIdx.x >> 5; p < patches; p += WEAK_WARPS) {
        const int row0 = p / wpr * 32, col0 = p % wpr * 32, r = row0 + lane, c = col0 + lane;
        const int rows = min(t.m - row0, 32), cols = min(t.n - col0, 32);
        const ListSrc src{g, t, row0, col0, lane < rows, lane < cols, scale};
        const uint32_t valid = 0xffffffffu >> (32 - cols);
        bool plain = true;                               // (other tiles run in FP64 as a whole)
        const int er = src.rowed ? row_scale(g, t, 0, r, plain) : fx::E_ZERO;
        const int ec = src.coled ? row_scale(g, t, 1, c, plain) : fx::E_ZERO;
        uint32_t need = 0;
        if (__all_sync(0xffffffffu, plain) && t.steps > 0) {
            // nonzero elements and sums of the rows and columns, where counting them is cheap; else the contraction length
            const int most = max(t.steps * FKS - (FKS - 1) * t.prod_count, 1);
            int fewest = most;
            float sr = (float)most, sc = sr;
            uint32_t mr = most, mc = most;
            if (t.steps <= 64 && t.prod_count <= 4) {
                int nr = 0, nc = 0;
                sr = sc = 0.f;
                for (int i = 0; i < t.prod_count; ++i) {
                    const BProd& q = src.prod(i);
                    for (int j = 0; j < (q.K + 31) / 32; ++j) {
                        uint32_t x, y;
                        src.words(i, j, x, y);
                        nr += __popc(x);
                        nc += __popc(y);
                    }
                    const int bias = src.bias(i);
                    if (src.rowed && bias != fx::NO_TERM) sr += 2.f * g.sums[q.ea + r] * power(g.e[q.ea + r] + bias - er);
                    if (src.coled) sc += g.sums[q.eb + c] * power(g.e[q.eb + c] - ec);
                }
                mr = __reduce_max_sync(0xffffffffu, nr);
                mc = __reduce_max_sync(0xffffffffu, nc);
                fewest = (int)(__reduce_min_sync(0xffffffffu, min((uint32_t)nr - 1u, (uint32_t)nc - 1u)) + 1u);   // (zeros last)
                sr = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sr)));
                sc = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(sc)));
            }
            if (mr <= 2 || mc <= 2) {
                need = src.rowed ? valid : 0u;
                if (mr <= 2) fx::sparse_outputs<true, 16>(src, src.rowed, cols);
                else fx::sparse_outputs<false, 16>(src, src.rowed, cols);
            } else {
                need = fx::weak_outputs(src, rows, cols, __ballot_sync(0xffffffffu, src.rowed),
                                        __ballot_sync(0xffffffffu, src.coled), er, ec, fx::least_sum((float)fewest, sr, sc));
                need = src.rowed ? need & valid : 0u;
                if (__any_sync(0xffffffffu, need != 0)) fx::fp64_outputs(src, src.rowed, cols, need, false);
            }
        }
        if (src.rowed) g.fp64[t.fp64_at + r * wpr + col0 / 32] = need;
    }
}

// byte offset of the 8-element chunk h of row r in a plane, on the even steps of the ring (the
// odd ones lie 32 bytes further in the swizzled row: the offset ^ 32)
__device__ __forceinline__ uint32_t chunk_off(int r, int h) {
    return (uint32_t)r * 64 + ((uint32_t)(h ^ ((r >> 1) & 3)) << 4);
}

// A producer thread's walk over one operand of a tile: its row, and the eight K values of each
// step that it loads and converts.  SIDE 0: A, SIDE 1: B.
template <int SIDE>
struct Walk {
    const double* p;        // this thread's first element of the step
    int ks;                 // stride along K
    int left;               // elements of the product from there on (beyond them: zeros)
    int i, end;             // product, and the elements of it that the step's first half starts at
    int h;                  // which 8 of the step's 16 elements
    int E;                  // scale of the row
    uint32_t off;           // where the digits go; ~0 for an absent row
    double coef;

    __device__ __forceinline__ void place(int r, int rows, const int* es) {
        off = r < rows ? chunk_off(r, h) : ~0u;
        E = es[SIDE * FM + r];
    }
    // the first step of product n
    __device__ __forceinline__ void set(const FxArgs& g, const BTile& t, const int* es, int n) {
        i = n;
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        // K contiguous: 16 rows x 2 halves a warp, in an order that spreads its stores over the
        // banks; rows contiguous: 32 rows, one half
        const int rl = ((lane >> 1) & 1) | ((lane >> 2) & 1) << 2 | ((lane >> 3) & 1) << 1 | ((lane >> 4) & 1) << 3;
        const BProd& q = g.prods[t.prod_begin + n];
        end = q.K;
        ks = SIDE ? q.b_rs : q.a_cs;
        const int w = SIDE ? warp & 3 : warp;
        int r;
        if (ks == 1) {
            r = w * 16 + rl;
            h = lane & 1;
        } else {
            r = (SIDE ? w & 1 : w & 3) * 32 + lane;
            h = SIDE ? w >> 1 : w >> 2;
        }
        p = (SIDE ? g.B + q.b_off : g.A + q.a_off) + (int64_t)r * (SIDE ? q.b_cs : q.a_rs) + (int64_t)8 * h * ks;
        if (SIDE == 0) coef = prod_coef(g, q);
        place(r, SIDE ? t.n : t.m, es);
        left = off != ~0u ? end - 8 * h : 0;
    }
    // the next step
    __device__ __forceinline__ void next(const FxArgs& g, const BTile& t, const int* es) {
        end -= FKS;
        if (end > 0) {
            p += (int64_t)FKS * ks;
            left -= FKS;
        } else if (i + 1 < t.prod_count) {
            set(g, t, es, i + 1);
        } else {
            left = 0;
        }
    }
    __device__ __forceinline__ void load(double (&v)[8]) const {
        if (left >= 8) {
            if (ks == 1 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
                const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const double2 d = __ldg(q + e);
                    v[2 * e] = d.x;
                    v[2 * e + 1] = d.y;
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = __ldg(p + (int64_t)e * ks);
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = e < left ? __ldg(p + (int64_t)e * ks) : 0.0;
        }
    }
};

// Digits of eight K values into the eight planes (plane bytes apart), 16 bytes each at addr.
__device__ __forceinline__ void digits8(const double (&v)[8], int E, uint32_t addr, uint32_t plane) {
    uint64_t q[8];
#pragma unroll
    for (int e = 0; e < 8; ++e)
        q[e] = fx::to_fixed((uint32_t)__double2hiint(v[e]), (uint32_t)__double2loint(v[e]), E);
    // bytes of two elements side by side, each in the low byte of an FP16 1024 + b, of which
    // 1152 is taken off: the digit.  Planes in pairs, to keep few registers alive.
    const __half2 bias = __half2half2(__ushort_as_half((unsigned short)0x6480));
#pragma unroll
    for (int pair = 3; pair >= 0; --pair) {
        uint32_t d[2][4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const uint32_t x = (uint32_t)(q[2 * e] >> (32 * (pair >> 1)));
            const uint32_t y = (uint32_t)(q[2 * e + 1] >> (32 * (pair >> 1)));
            const uint32_t t = __byte_perm(x, y, (pair & 1) ? 0x7362 : 0x5140);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const uint32_t f = __byte_perm(t, 0x64646464u, c ? 0x4342 : 0x4140);
                const __half2 hv = __hsub2(*reinterpret_cast<const __half2*>(&f), bias);
                d[c][e] = *reinterpret_cast<const uint32_t*>(&hv);
            }
        }
        st_shared_v4(addr + (6 - 2 * pair) * plane, d[1][0], d[1][1], d[1][2], d[1][3]);
        st_shared_v4(addr + (7 - 2 * pair) * plane, d[0][0], d[0][1], d[0][2], d[0][3]);
    }
}

__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t& a, uint32_t& b) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(taddr));
}
// the loads have landed (the registers pass through, so that nothing reads them earlier)
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&d)[FD][2]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(d[0][0]), "+r"(d[0][1]), "+r"(d[1][0]), "+r"(d[1][1]), "+r"(d[2][0]), "+r"(d[2][1]),
                   "+r"(d[3][0]), "+r"(d[3][1]), "+r"(d[4][0]), "+r"(d[4][1]), "+r"(d[5][0]), "+r"(d[5][1]),
                   "+r"(d[6][0]), "+r"(d[6][1]), "+r"(d[7][0]), "+r"(d[7][1])
                 :
                 : "memory");
}

// FP16 operands, FP32 accumulate, K-major, M x N
__device__ __forceinline__ uint32_t idesc_f16(uint32_t M, uint32_t N) {
    return (1u << 4) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// The digit products of one step (16 contraction elements) or, with NK = 2, of the two steps of a
// 64-byte block, for B planes of N16 rows: A plane d times the B planes 0 .. 7 - d.  The two steps
// follow each other on the same operand shape, and everything but the base addresses is a
// constant: issued from a plain loop over the planes a step takes 1600 cycles at N16 = 64 (the
// tensor pipe needs 1152), in this order 1250.
template <int N16, int NK>
__device__ __forceinline__ void issue_planes(uint32_t tmem, uint64_t a, uint64_t b, uint32_t fresh) {
#pragma unroll
    for (int d = 0; d < FD; ++d)
#pragma unroll
        for (int c = 0; c < (FD - d) * N16; c += 256)
#pragma unroll
            for (int k = 0; k < NK; ++k)
                umma_bf16(tmem + d * N16 + c, a + d * (A_PLANE >> 4) + 2 * k, b + (c * 64 >> 4) + 2 * k,
                          idesc_f16(FM, (FD - d) * N16 - c < 256 ? (FD - d) * N16 - c : 256),
                          d == 0 && k == 0 ? (fresh ? 0u : 1u) : 1u);
}
template <int NK>
__device__ __forceinline__ void issue_step(int n16, uint32_t tmem, uint64_t a, uint64_t b, uint32_t fresh) {
    if (n16 == 64) issue_planes<64, NK>(tmem, a, b, fresh);
    else if (n16 == 48) issue_planes<48, NK>(tmem, a, b, fresh);
    else if (n16 == 32) issue_planes<32, NK>(tmem, a, b, fresh);
    else issue_planes<16, NK>(tmem, a, b, fresh);
}

// Producer warps meet (bounded, so that a CTA that gives up does not hang here).
struct PSync {
    uint64_t* bar;
    uint32_t n;
    volatile int* abort_flag;
    int* err;
    __device__ __forceinline__ bool operator()() {
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(bar);
        return mbar_wait(bar, n++ & 1, abort_flag, err);
    }
};

// A tile in FP64 arithmetic on the producer warps (256 threads, 4 x 4 outputs each, two halves
// of 64 rows).
__device__ __forceinline__ bool fp64_tile(const FxArgs& g, const BTile& t, double* sh, PSync& psync, double scale) {
    double (*As)[65] = reinterpret_cast<double (*)[65]>(sh);
    double (*Bs)[65] = As + 8;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    double* C = g.C + t.c_off;
    for (int half = 0; half < t.m; half += 64) {
        const int m = t.m - half < 64 ? t.m - half : 64;
        double acc[4][4] = {};
        for (int s = 0; s < t.prod_count; ++s) {
            const BProd& p = g.prods[t.prod_begin + s];
            const double* a = g.A + p.a_off;
            const double* b = g.B + p.b_off;
            const double coef = prod_coef(g, p);
            for (int k0 = 0; k0 < p.K; k0 += 8) {
                for (int l = 0; l < 2; ++l) {
                    const int idx = tid + 256 * l;
                    int r, k;
                    if (p.a_cs == 1) { r = idx >> 3; k = idx & 7; } else { r = idx & 63; k = idx >> 6; }
                    As[k][r] = r < m && k0 + k < p.K
                                   ? coef * a[(int64_t)(half + r) * p.a_rs + (int64_t)(k0 + k) * p.a_cs] : 0.0;
                    if (p.b_rs == 1) { r = idx >> 3; k = idx & 7; } else { r = idx & 63; k = idx >> 6; }
                    Bs[k][r] = r < t.n && k0 + k < p.K
                                   ? b[(int64_t)r * p.b_cs + (int64_t)(k0 + k) * p.b_rs] : 0.0;
                }
                if (!psync()) return false;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    double av[4], bv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) { av[i] = As[k][ty * 4 + i]; bv[i] = Bs[k][tx * 4 + i]; }
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
                }
                if (!psync()) return false;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int r = ty * 4 + i, c = tx * 4 + j;
                if (r < m && c < t.n) {
                    double* cp = C + (int64_t)(half + r) * t.ldc + c;
                    *cp = g.accumulate ? *cp + scale * acc[i][j] : scale * acc[i][j];
                }
            }
    }
    return true;
}

__global__ void __launch_bounds__(FTHREADS, 1) fx_gemm_kernel(const __grid_constant__ FxArgs g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
    uint64_t* empty = full + FST;
    uint64_t* tready = empty + FST;      // [2] scales of a tile are in shared memory
    uint64_t* edone = tready + 2;        // [2] the drain and the MMA issuer are done with them
    uint64_t* tfull = edone + 2;         // a chunk's sums are in tensor memory
    uint64_t* tempty = tfull + 1;        // they have been read
    uint64_t* pbar = tempty + 1;
    uint64_t* drain = pbar + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    int* escale = reinterpret_cast<int*>(smem + OFF_E);          // [2][FM + FN]
    int* ebad = escale + 2 * (FM + FN);                          // [2][PW]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < FST; ++s) { mbar_init(&full[s], PW); mbar_init(&empty[s], 1); }
        for (int b = 0; b < 2; ++b) { mbar_init(&tready[b], 1); mbar_init(&edone[b], EW + 1); }
        mbar_init(tfull, 1);
        mbar_init(tempty, EW);
        mbar_init(pbar, PW);
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == PW + EW) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t base = su32(smem);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long total = g.ntiles;
    const long rounds = (total + gridDim.x - 1) / gridDim.x;

    if (warp < PW) {
        // ------------------------------------------------ producers
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_PROD));
        PSync psync{pbar, 0, abort_flag, g.err};
        const double scale = g.inv_scale ? g.scale / g.inv_scale[0] : g.scale;
        uint32_t step = 0, tcount = 0;
        bool ok = true;
        for (long i = 0; i < rounds && ok; ++i) {
            const long item = item_of(i);
            if (item >= total) continue;
            const BTile t = g.tiles[item];
            if (t.m == 0) continue;
            const int b = tcount & 1;
            if (!(ok = mbar_wait(&edone[b], ((tcount >> 1) & 1) ^ 1, abort_flag, g.err))) break;
            ++tcount;
            // scales: one thread per row of A, then per column of B
            int* es = escale + b * (FM + FN);
            {
                const int side = threadIdx.x >= FM, r = side ? threadIdx.x - FM : threadIdx.x;
                bool plain = true;
                if (threadIdx.x < FM + FN)
                    es[threadIdx.x] = r < (side ? t.n : t.m) ? row_scale(g, t, side, r, plain) : fx::E_ZERO;
                const bool bad = __any_sync(0xffffffffu, !plain);
                if (lane == 0) ebad[b * PW + warp] = bad;
            }
            if (!(ok = psync())) break;
            if (threadIdx.x == 0) mbar_arrive(&tready[b]);
            bool bad = false;
#pragma unroll
            for (int w = 0; w < PW; ++w) bad |= ebad[b * PW + w] != 0;
            if (bad) {
                ok = fp64_tile(g, t, reinterpret_cast<double*>(smem + OFF_DF), psync, scale);
                continue;
            }
            if (t.steps == 0) continue;
            const uint32_t bplane = (uint32_t)((t.n + 15) & ~15) * 64;
            // warp w converts 16 (or half of 32) rows of A on every step; B has half as many rows:
            // warps 0-3 convert it on even steps, warps 4-7 on odd steps.  The loads of the next
            // item are issued before an item is converted.
            Walk<0> wa;
            Walk<1> wb;
            double va[8], vb[8];
            wa.set(g, t, es, 0);
            wa.load(va);
            wb.set(g, t, es, 0);
            if (((step & 1) != 0) != (warp >= 4)) wb.next(g, t, es);
            wb.load(vb);
            for (int s = 0; s < t.steps; ++s, ++step) {
                const uint32_t st = step % FST;
                double cur[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) cur[e] = va[e];
                const int E = wa.E;
                const uint32_t off = wa.off, odd = 32 * (st & 1);
                const double coef = wa.coef;
                if (coef != 1.0) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) cur[e] *= coef;
                }
                wa.next(g, t, es);
                wa.load(va);
                const uint32_t blk = base + (st >> 1) * BLK;
                if (!(ok = mbar_wait(&empty[st], ((step / FST) & 1) ^ 1, abort_flag, g.err))) break;
                if (off != ~0u) digits8(cur, E, blk + (off ^ odd), A_PLANE);
                if (((step & 1) != 0) == (warp >= 4)) {
                    if (wb.off != ~0u) digits8(vb, wb.E, blk + A_BLK + (wb.off ^ odd), bplane);
                    wb.next(g, t, es);
                    wb.next(g, t, es);
                    wb.load(vb);
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full[st]);
            }
        }
    } else if (warp < PW + EW) {
        // ------------------------------------------------ drain
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R_DRAIN));
        const double scale = g.inv_scale ? g.scale / g.inv_scale[0] : g.scale;
        const int q = warp & 3, h = (warp - PW) >> 2;       // tensor-memory lanes, column half
        double* tr = reinterpret_cast<double*>(smem + OFF_TR + (warp - PW) * TR_WARP);
        uint32_t ccount = 0, tcount = 0;
        bool ok = true;
        for (long i = 0; i < rounds && ok; ++i) {
            const long item = item_of(i);
            if (item >= total) continue;
            const BTile t = g.tiles[item];
            if (t.m == 0) continue;
            const int b = tcount & 1;
            if (!(ok = mbar_wait(&tready[b], (tcount >> 1) & 1, abort_flag, g.err))) break;
            ++tcount;
            bool bad = false;
#pragma unroll
            for (int w = 0; w < PW; ++w) bad |= ebad[b * PW + w] != 0;
            if (!bad) {
                const int n16 = (t.n + 15) & ~15;
                const int* es = escale + b * (FM + FN);
                const int rows = t.m - q * 32 < 32 ? t.m - q * 32 : 32, ncol = t.n - 32 * h < 32 ? t.n - 32 * h : 32;
                // outputs that are there already (weak_list_kernel); `whole`: all of the patch
                const bool rowed = lane < rows && ncol > 0;
                const uint32_t valid = ncol > 0 ? 0xffffffffu >> (32 - ncol) : 0u;
                const uint32_t need = rowed ? g.fp64[t.fp64_at + (q * 32 + lane) * ((t.n + 31) / 32) + h] : 0u;
                const bool whole = __all_sync(0xffffffffu, !rowed || need == valid);
                uint32_t w0[32], w1[32], w2[32];
#pragma unroll
                for (int c = 0; c < 32; ++c) { w0[c] = 0; w1[c] = 0; w2[c] = 0; }
                for (int s = 0; s < t.steps; s += FCH) {
                    if (!(ok = mbar_wait(tfull, ccount & 1, abort_flag, g.err))) break;
                    ++ccount;
                    tc_fence_after();
                    const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + 32 * h;
#pragma unroll
                    for (int c = 0; c < 32; c += 2) {
                        if (32 * h + c < n16 && !whole) {
                            uint32_t d[FD][2];
#pragma unroll
                            for (int e = 0; e < FD; ++e) tmem_ld2(ta + e * n16 + c, d[e][0], d[e][1]);
                            tmem_ld_wait(d);
#pragma unroll
                            for (int u = 0; u < 2; ++u) {
                                int64_t hi = 0, lo = 0;
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    hi += (int64_t)__float2int_rn(__uint_as_float(d[e][u])) * (1 << (8 * (3 - e)));
                                    lo += (int64_t)__float2int_rn(__uint_as_float(d[4 + e][u])) * (1 << (8 * (3 - e)));
                                }
                                hi += lo >> 32;
                                // (w2, w1, w0) += hi 2^32 + low word of lo
                                asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
                                    : "+r"(w0[c + u]), "+r"(w1[c + u]), "+r"(w2[c + u])
                                    : "r"((uint32_t)lo), "r"((uint32_t)hi), "r"((uint32_t)(hi >> 32)));
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(tempty);
                }
                if (!ok) break;
                // round to FP64 and store, 8 columns at a time
                const int er = es[q * 32 + lane] - 2112;
                double* C = g.C + t.c_off + (int64_t)(q * 32) * t.ldc;
#pragma unroll
                for (int c0 = 0; c0 < 32; c0 += 8) {
                    const int col0 = 32 * h + c0;
                    if (col0 < t.n && rows > 0) {
#pragma unroll
                        for (int c = 0; c < 8; ++c) {
                            double v = 0.0;
                            if ((need >> (c0 + c)) & 1u) {
                                if (!g.accumulate) v = C[(int64_t)lane * t.ldc + col0 + c];
                            } else if (col0 + c < t.n) {
                                v = fx::from_fixed(w2[c0 + c], w1[c0 + c], w0[c0 + c], er + es[FM + col0 + c]);
                                if (scale != 1.0) v *= scale;
                            }
                            tr[lane * 9 + c] = v;
                        }
                        __syncwarp();
                        const int c = lane & 7;
                        for (int r = lane >> 3; r < rows; r += 4)
                            if (col0 + c < t.n) {
                                double* cp = C + (int64_t)r * t.ldc + col0 + c;
                                const double v = tr[r * 9 + c];
                                *cp = g.accumulate ? *cp + v : v;
                            }
                        __syncwarp();
                    }
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&edone[b]);
        }
    } else {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R_MMA));
        if (warp == PW + EW && lane == 0) {
            // -------------------------------------------- MMA issuer
            uint32_t step = 0, ccount = 0, tcount = 0;
            bool ok = true;
            for (long i = 0; i < rounds && ok; ++i) {
                const long item = item_of(i);
                if (item >= total) continue;
                const BTile t = g.tiles[item];
                if (t.m == 0) continue;
                const int b = tcount & 1;
                if (!(ok = mbar_wait(&tready[b], (tcount >> 1) & 1, abort_flag, g.err))) break;
                ++tcount;
                bool bad = false;
                for (int w = 0; w < PW; ++w) bad |= ebad[b * PW + w] != 0;
                mbar_arrive(&edone[b]);
                if (bad) continue;
                const int n16 = (t.n + 15) & ~15;
                for (int s = 0; s < t.steps;) {
                    const uint32_t st = step % FST;
                    const bool first = s % FCH == 0;
                    // both steps of a 64-byte block, unless the tile or its chunk ends in between
                    const bool two = !(st & 1) && s + 1 < t.steps && s % FCH != FCH - 1;
                    if (first) {
                        if (!(ok = mbar_wait(tempty, (ccount & 1) ^ 1, abort_flag, g.err))) break;
                        tc_fence_after();
                    }
                    if (!(ok = mbar_wait(&full[st], (step / FST) & 1, abort_flag, g.err))) break;
                    if (two && !(ok = mbar_wait(&full[st + 1], (step / FST) & 1, abort_flag, g.err))) break;
                    tc_fence_after();
                    const uint32_t blk = base + (st >> 1) * BLK + 32 * (st & 1);
                    const uint64_t da = sdesc64(blk), db = sdesc64(blk + A_BLK);
                    if (two) issue_step<2>(n16, tmem, da, db, first);
                    else issue_step<1>(n16, tmem, da, db, first);
                    umma_commit(&empty[st]);
                    if (two) umma_commit(&empty[st + 1]);
                    s += two ? 2 : 1;
                    step += two ? 2 : 1;
                    if (s % FCH == 0 || s == t.steps) {
                        umma_commit(tfull);
                        ++ccount;
                    }
                }
            }
            if (!ok) {
                umma_commit(drain);
                mbar_wait_drain(drain, 0);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == PW + EW) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// Exponent codes of operand rows: unit u covers up to 32 rows of one operand view, element
// (r, k) at off + r rs + k ks; out[r] = the largest code E of row r, sums[r] = the sum of its magnitudes over
// 2^(E - 1022).  And which of its elements are not zero, 32 to a word.
__global__ void __launch_bounds__(256) row_code_kernel(const FxRows* __restrict__ units, const double* __restrict__ A,
                                                       const double* __restrict__ B, uint16_t* __restrict__ out,
                                                       uint32_t* __restrict__ words, float* __restrict__ sums) {
    __shared__ int part[8][32];
    __shared__ float fpart[8][32];
    const FxRows u = units[blockIdx.x];
    const double* src = (u.which ? B : A) + u.off;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a running sum for the largest code so far
    auto add = [](int& e, float& f, int e2, float f2) {
        const int d = e2 - e, s = d > 0 ? d : -d;
        const float down = s < 126 ? __int_as_float((127 - s) << 23) : 0.f;
        f = d > 0 ? fmaf(f, down, f2) : fmaf(f2, down, f);
        e = max(e, e2);
    };
    // (the mantissa's upper bits over the code's power of two; subnormals count as the largest)
    auto part_of = [](double v, int c) {
        return c ? (c == 1 ? 1.f : __int_as_float(0x3f000000 | ((__double2hiint(v) & 0xfffff) << 3))) : 0.f;
    };
    auto code = [](double v) { return fx::exp_code((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v)); };
    if (u.ks == 1) {
        // lanes along K; each warp four rows, loads of the four in flight together
        int e[4] = {0, 0, 0, 0};
        float f[4] = {0.f, 0.f, 0.f, 0.f};
        for (int k = lane; k - lane < u.K; k += 32) {
            double v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int r = warp + 8 * j;
                v[j] = r < u.rows && k < u.K ? src[(int64_t)r * u.rs + k] : 0.0;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int r = warp + 8 * j, c = code(v[j]);
                add(e[j], f[j], c, part_of(v[j], c));
                const uint32_t bits = __ballot_sync(0xffffffffu, c != 0);
                if (lane == 0 && r < u.rows) words[u.word + (int64_t)(k / 32) * u.all + r] = bits;
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            for (int o = 16; o > 0; o >>= 1)
                add(e[j], f[j], __shfl_xor_sync(0xffffffffu, e[j], o), __shfl_xor_sync(0xffffffffu, f[j], o));
            if (lane == 0 && warp + 8 * j < u.rows) {
                out[u.out + warp + 8 * j] = (uint16_t)e[j];
                sums[u.out + warp + 8 * j] = f[j] * 1.001f;
            }
        }
    } else {
        // lanes along the rows, warps along K
        int e = 0;
        float f = 0.f;
        if (lane < u.rows) {
            for (int b = warp; 32 * b < u.K; b += 8) {
                uint32_t bits = 0;
#pragma unroll 8
                for (int k = 0; k < 32; ++k) {
                    const double v = 32 * b + k < u.K ? src[(int64_t)lane * u.rs + (int64_t)(32 * b + k) * u.ks] : 0.0;
                    const int c = code(v);
                    add(e, f, c, part_of(v, c));
                    bits |= (c ? 1u : 0u) << k;
                }
                words[u.word + (int64_t)b * u.all + lane] = bits;
            }
        }
        part[warp][lane] = e;
        fpart[warp][lane] = f;
        __syncthreads();
        if (warp == 0 && lane < u.rows) {
#pragma unroll
            for (int w = 1; w < 8; ++w) add(e, f, part[w][lane], fpart[w][lane]);
            out[u.out + lane] = (uint16_t)e;
            sums[u.out + lane] = f * 1.001f;
        }
    }
}

int launch_fx(const FxArgs& g, int num_sms, cudaStream_t st) {
    static PerDevice done;
    if (int rc = raise_smem_limit(done, (const void*)fx_gemm_kernel, FSMEM)) return rc;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)(g.ntiles < num_sms ? g.ntiles : num_sms));
    cfg.blockDim = dim3(FTHREADS);
    cfg.dynamicSmemBytes = FSMEM;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = HEFF_PDL ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, fx_gemm_kernel, g);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "fx_gemm launch: %s", cudaGetErrorString(e));
    count_launches(1);
    return HEFF_OK;
}

}  // namespace

int launch_bgemm(const BList& b, const double* A, const double* B, double* C, const double* coef1,
                 const double* coef2, double scale, void* stream, int* err, const double* inv_scale) {
    if (b.tiles.empty()) return HEFF_OK;
    if (b.tile_m != FM || b.tile_n != FN)
        return fail(HEFF_ERR_INVALID_ARG, "FP64 block products need %d x %d tiles", FM, FN);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!b.rows.empty()) {
        row_code_kernel<<<(unsigned)b.rows.size(), 256, 0, st>>>(b.d_rows, A, B, b.d_codes, b.d_words, b.d_sums);
        count_launches(1);
    }
    FxArgs g{};
    g.tiles = b.d_tiles;
    g.prods = b.d_prods;
    g.e = b.d_codes;
    g.words = b.d_words;
    g.sums = b.d_sums;
    g.fp64 = b.d_fp64;
    g.coef1 = coef1;
    g.coef2 = coef2;
    g.inv_scale = inv_scale;
    g.scale = scale;
    g.accumulate = b.accumulate ? 1 : 0;
    g.ntiles = (int)b.tiles.size();
    g.A = A;
    g.B = B;
    g.C = C;
    g.err = err;
    weak_list_kernel<<<(unsigned)b.tiles.size(), 32 * WEAK_WARPS, 0, st>>>(g);
    count_launches(1);
    return launch_fx(g, b.num_sms > 0 ? b.num_sms : 148, st);
}

}  // namespace heff
