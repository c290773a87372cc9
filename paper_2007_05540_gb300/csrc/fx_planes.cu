// FP64 matvec products from digit planes: the arithmetic of fx_gemm.cu (62-bit fixed-point rows, eight
// signed 8-bit digits, 36 FP16 digit products per contraction step, exact sums), with the operands
// converted once into planes of FP16 digits in the workspace and brought in by TMA.
//
// fx_gemm.cu converts an operand row in every tile that reads it; its producer warps take about
// 1.9 us per step of 16 contraction elements where the tensor pipe needs 0.6, and each tile starts with a
// search for its rows' scales.  Here
//   digit_kernel     finds the scale of each operand row and writes its digit planes (8 bytes read, 16
//                    written per element: bound by HBM or L2)
//   fx_plane_kernel  multiplies planes: a persistent CTA per SM, 128 x 64 tiles, one thread issuing TMA
//                    loads, one issuing MMAs, eight drain warps
//   weak_plane_kernel  finds the outputs that digits do not resolve and computes them in FP64 (fx_check.cuh)
// Prepared matvec, m = 1024, k = 14: 577 us with the conversion in every tile, 400 us here (GEMM 1 163, GEMM 2 124,
// planes of T 45, of x 7) and 466 with the check; environment update m = 1024 309, 253 and 315 us.  Bound by the
// drain, in which the tensor pipe waits (active 27 % of GEMM 1's cycles and 25 % of the environment update's), and by the
// loads' latency on contractions of two to ten K blocks.  128 x 32 tiles with two accumulator sets drain under the next
// tile's MMAs, but read A twice as often: GEMM 1 164, GEMM 2 217 us.
// The planes take 16 bytes per operand element: plans whose workspace would pass FX_PLANES_MAX and calls on a
// smaller workspace (heff_apply_noalloc) run on the FP64 units (apply.cu).
//
// Plane layout.  A virtual row is one row's K block of 32 elements, numbered kb R + row (R rows in the
// array): the rows of a K block lie one after another, so a TMA box is one contiguous piece.
//   A operands: [pair of planes, 4][virtual row][128 bytes: plane 2 p, then plane 2 p + 1]
//   B operands: [plane, 8][virtual row][64 bytes]; a box takes all 8 planes of up to 64 rows, which in
//               shared memory are one wide B operand (see fx_gemm.cu)
// The ring holds two K blocks: A in slots of one pair (16 KB), each released as soon as its MMAs are
// done, so that a slot's load has more than one K block's MMAs (2500 cycles) to arrive.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstring>

#include "fixed.cuh"
#include "fx_check.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace heff {
namespace {

using namespace ptx;

constexpr int FM = FX_TILE_M, FN = FX_TILE_N;
constexpr int FD = 8;                             // digits
constexpr int PAIRS = FD / 2;
constexpr int PCH = 8;                            // K blocks per exact accumulation chunk (256 elements)
constexpr int DW = 8;                             // drain warps
constexpr int CODE_COLS = FX_T_CODE_COLS;         // columns per exponent code of T
constexpr int PTHREADS = 32 * (2 + DW);
constexpr int A_SLOT = FM * 128;                  // one pair of planes of a K block
constexpr int B_STAGE = FD * FN * 64;
constexpr int P_STAGES = 2;
constexpr int OFF_B = P_STAGES * PAIRS * A_SLOT;
constexpr int OFF_TR = OFF_B + P_STAGES * B_STAGE;
constexpr int TR_WARP = 32 * 9 * 8;               // drain transposes: 32 rows x 8 columns
constexpr int OFF_BAR = OFF_TR + DW * TR_WARP;
constexpr int PSMEM = OFF_BAR + 256 + 1024;
static_assert(PSMEM <= 227 * 1024, "shared memory of one CTA");

// row scale of a row that needs FP64 arithmetic
constexpr int E_BAD = -1;

__device__ __forceinline__ int code_of(double v) {
    return fx::exp_code((uint32_t)__double2hiint(v), (uint32_t)__double2loint(v));
}

// ------------------------------------------------------------------ digit planes
struct DigitArgs {
    const FxUnit* units;
    const KSeg* segs;
    const double* src;       // rows of ld elements
    int64_t ld;
    const uint16_t* codes;   // [column / code_cols][row]
    int code_cols;
    char* planes;
    int32_t* scale;          // per row
    uint32_t* nonzero;       // per virtual row: which elements are not zero
    uint2* total;            // per row: its elements' sum over the scale (a float, rounded up), nonzero elements
    int64_t rows;            // rows of the array (all batch entries): stride of codes and virtual rows
    int64_t batch_rows;
    int a_side;              // plane layout: A (pairs) or B
};

// One block per unit of up to 8 rows that share their segments: a warp per row finds the scale from the
// rows' exponent codes, then a warp per K block converts 8 rows x 32 elements.
__global__ void __launch_bounds__(256) digit_kernel(DigitArgs g) {
    __shared__ int es[8];
    __shared__ unsigned int sum[8], count[8];            // (integers: the same whatever the order of the warps)
    const FxUnit u = g.units[blockIdx.x];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t row0 = u.row0 + (int64_t)blockIdx.y * g.batch_rows;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    {
        // lanes over the segments' K blocks
        int e = 0;
        if (warp < u.nrows)
            for (int s = 0; s < u.seg_count; ++s) {
                const KSeg sg = g.segs[u.seg_begin + s];
                for (int k = sg.k0 / g.code_cols + lane; k < (sg.k0 + sg.klen) / g.code_cols; k += 32)
                    e = max(e, (int)g.codes[(int64_t)k * g.rows + row0 + warp]);
            }
        for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        if (lane == 0) {
            const int E = fx::exp_plain(e) ? (e ? e : fx::E_ZERO) : E_BAD;
            es[warp] = E < 0 ? fx::E_ZERO : E;           // a bad row's digits are not used
            sum[warp] = count[warp] = 0;
            if (warp < u.nrows) g.scale[row0 + warp] = E;
        }
    }
    __syncthreads();
    const int r = lane >> 2, c = lane & 3;               // row, 8-element chunk of the K block
    const int64_t vrows = (g.ld / KPAD) * g.rows;
    const int E = es[r];
    int nkb = 0;
    for (int s = 0; s < u.seg_count; ++s) {
        const KSeg sg = g.segs[u.seg_begin + s];
        for (int k = sg.k0 / KPAD; k < (sg.k0 + sg.klen) / KPAD; ++k, ++nkb) {
            if ((nkb & 7) != warp || r >= u.nrows) continue;
            const double2* p = reinterpret_cast<const double2*>(g.src + (row0 + r) * g.ld + k * KPAD + 8 * c);
            double v[8];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const double2 d = p[e];
                v[2 * e] = d.x;
                v[2 * e + 1] = d.y;
            }
            uint64_t q[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                q[e] = fx::to_fixed((uint32_t)__double2hiint(v[e]), (uint32_t)__double2loint(v[e]), E);
            const int64_t vr = (int64_t)k * g.rows + row0 + r;
            // eight elements a lane, four lanes a row
            uint32_t nz = 0;
            float f = 0.f;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                f += __uint_as_float(fx::magnitude(v[e], fx::magnitude_base(E)));
                nz |= (code_of(v[e]) ? 1u : 0u) << (8 * c + e);
            }
            const unsigned lanes = 0xffffffffu >> (32 - 4 * u.nrows);
#pragma unroll
            for (int o = 1; o < 4; o <<= 1) {
                nz |= __shfl_xor_sync(lanes, nz, o);
                f += __shfl_xor_sync(lanes, f, o);
            }
            if (c == 0) {
                g.nonzero[vr] = nz;
                atomicAdd(&sum[r], (unsigned int)(f * 16384.f) + 2u);
                atomicAdd(&count[r], (unsigned int)__popc(nz));
            }
            const __half2 bias = __half2half2(__ushort_as_half((unsigned short)0x6480));
#pragma unroll
            for (int d = 0; d < FD; ++d) {
                // byte 7 - d of each value, in the low byte of an FP16 1024 + b; 1152 off: the digit
                uint4 o;
                uint32_t* w = reinterpret_cast<uint32_t*>(&o);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t x = (uint32_t)(q[2 * e] >> (d < 4 ? 32 : 0));
                    const uint32_t y = (uint32_t)(q[2 * e + 1] >> (d < 4 ? 32 : 0));
                    const int b = 3 - (d & 3);
                    const uint32_t t = __byte_perm(x, y, b | (4 + b) << 4);           // bytes b of x, y
                    const uint32_t h = __byte_perm(t, 0x64646464u, 0x4140);
                    const __half2 hv = __hsub2(*reinterpret_cast<const __half2*>(&h), bias);
                    w[e] = *reinterpret_cast<const uint32_t*>(&hv);
                }
                char* dst = g.a_side ? g.planes + (((d >> 1) * vrows + vr) * 128 + (d & 1) * 64 + c * 16)
                                     : g.planes + ((d * vrows + vr) * 64 + c * 16);
                *reinterpret_cast<uint4*>(dst) = o;
            }
        }
    }
    __syncthreads();
    if ((int)threadIdx.x < u.nrows)
        g.total[row0 + threadIdx.x] = make_uint2(__float_as_uint((float)sum[threadIdx.x] * (1.f / 16384)), count[threadIdx.x]);
}

// ------------------------------------------------------------------ plane products
struct PlaneArgs {
    CUtensorMap a[3];                    // A planes in boxes of 32, 64, 128 rows
    CUtensorMap b[4];                    // B planes in boxes of 16, 32, 48, 64 rows, all planes
    const GemmTask* tasks;
    const KSeg* segs;
    int ntasks, nbatch, b0, to_y;
    int64_t ld, a_rows, b_rows;          // operand pitch; rows of the arrays
    int64_t a_batch_rows, b_batch_rows;
    const int32_t *ea, *eb;              // row scales
    const uint32_t *za, *zb;             // nonzero elements of the virtual rows, and totals of the rows
    const uint2 *ta, *tb;
    uint32_t* fp64;                      // outputs computed in FP64: a bit each, [batch entry][fp64_at[task] + row * words + word]
    const int32_t* fp64_at;
    int64_t fp64_words;                  // of a batch entry
    const double *A, *B;                 // FP64 operands (outputs that need FP64 arithmetic)
    double* C;
    int64_t c_batch_elems, c_batch_rows;
    uint16_t* et;                        // exponent codes of T, per CODE_COLS columns
    int64_t et_rows;
    PtrBatch y;
    double* split;                       // scratch of split tiles
    const SplitTile* split_tiles;
    int64_t split_elems;
    int* err;
};

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(su32(bar)), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void tma_3d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int x, int y, int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(su32(bar)), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(bar)), "r"(bytes) : "memory");
}

// K-major operand in 128-byte swizzled rows, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t sdesc128(uint32_t saddr) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
__device__ __forceinline__ uint32_t idesc_f16(uint32_t M, uint32_t N) {
    return (1u << 4) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// The products of the A planes 2 P and 2 P + 1 (one slot) of a K block with the B planes 0 .. 7 - d, for
// B planes of N16 rows: accumulators d .. 7, both 16-element steps on one operand shape.
template <int N16, int P>
__device__ __forceinline__ void issue_pair(uint32_t tmem, uint64_t a, uint64_t b, bool fresh) {
#pragma unroll
    for (int d = 2 * P; d < 2 * P + 2; ++d)
#pragma unroll
        for (int c = 0; c < (FD - d) * N16; c += 256)
#pragma unroll
            for (int k = 0; k < 2; ++k)
                umma_bf16(tmem + d * N16 + c, a + 4 * (d & 1) + 2 * k, b + (c * 64 >> 4) + 2 * k,
                          idesc_f16(FM, (FD - d) * N16 - c < 256 ? (FD - d) * N16 - c : 256),
                          d == 0 && k == 0 ? (fresh ? 0u : 1u) : 1u);
}
template <int P>
__device__ __forceinline__ void issue(int n16, uint32_t tmem, uint64_t a, uint64_t b, bool fresh) {
    if (n16 == 64) issue_pair<64, P>(tmem, a, b, fresh);
    else if (n16 == 48) issue_pair<48, P>(tmem, a, b, fresh);
    else if (n16 == 32) issue_pair<32, P>(tmem, a, b, fresh);
    else issue_pair<16, P>(tmem, a, b, fresh);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr));
}
// the loads have landed (the registers pass through, so that nothing reads them earlier)
__device__ __forceinline__ void tmem_wait(uint32_t (&d)[FD][4]) {
#pragma unroll
    for (int e = 0; e < FD; ++e) {
        if (e == 0)
            asm volatile("tcgen05.wait::ld.sync.aligned;"
                         : "+r"(d[e][0]), "+r"(d[e][1]), "+r"(d[e][2]), "+r"(d[e][3]) : : "memory");
        else
            asm volatile("" : "+r"(d[e][0]), "+r"(d[e][1]), "+r"(d[e][2]), "+r"(d[e][3]) : : "memory");
    }
}

// A patch of a tile, as fx_check.cuh reads it: one piece per segment.
struct PlaneSrc {
    static constexpr bool DENSE = true;
    const KSeg* segs;
    int nseg;
    bool rowed, coled;                   // whether there is a row, a column `lane`
    const double *a, *b;                 // the patch's first row and column
    int64_t ld;
    const uint32_t *za, *zb;             // of row `lane`, of column `lane`
    int64_t a_rows, b_rows;
    double* out;                         // row `lane` of the output
    __device__ __forceinline__ int pieces() const { return nseg; }
    __device__ __forceinline__ fx::Piece piece(int i, int r) const {
        const KSeg s = segs[i];
        return {a + r * ld + s.k0, b + s.k0, ld, 1, 1, s.klen, 1.0};
    }
    __device__ __forceinline__ int bias(int) const { return 0; }
    __device__ __forceinline__ void words(int i, int j, uint32_t& x, uint32_t& y) const {
        const int64_t kb = segs[i].k0 / KPAD + j;
        x = rowed ? za[kb * a_rows] : 0u;
        y = coled ? zb[kb * b_rows] : 0u;
    }
    __device__ __forceinline__ void store(int c, double v) const { out[c] = v; }
};

// where a task's values go: T, y, or a split tile's part of its scratch (bat: batch entry of the launch)
__device__ __forceinline__ double* task_out(const PlaneArgs& g, const GemmTask& t, int bat, int64_t& ldc) {
    ldc = t.ldc;
    if (t.split) {
        ldc = t.n;
        return g.split + (int64_t)bat * g.split_elems + g.split_tiles[t.split >> 9].off +
               (int64_t)((t.split >> 5) & 15) * t.m * t.n;
    }
    return (g.to_y ? static_cast<double*>(const_cast<void*>(g.y.p[bat])) : g.C + (int64_t)(g.b0 + bat) * g.c_batch_elems) +
           t.c_off;
}

// The outputs of a patch (rows x cols from row0, col0 of the tile; C: its first row, column col0 of the output)
// that the digits do not resolve, computed in FP64: their bits in this lane's row.
__device__ __forceinline__ uint32_t check_patch(const PlaneArgs& g, const GemmTask& t, int b, int row0, int col0, int rows,
                                                int cols, double* C, int64_t ldc) {
    if (t.seg_count == 0) return 0;
    const int lane = threadIdx.x & 31;
    const int64_t a_row = t.a_row + b * g.a_batch_rows, b_row = t.b_row + b * g.b_batch_rows;
    rows = min(rows, 32);
    const bool rowed = lane < rows, coled = lane < cols;
    const int er = rowed ? g.ea[a_row + row0 + lane] : fx::E_ZERO;
    const int ec = coled ? g.eb[b_row + col0 + lane] : fx::E_ZERO;
    const uint2 rt = rowed ? g.ta[a_row + row0 + lane] : make_uint2(0, 0);
    const uint2 ct = coled ? g.tb[b_row + col0 + lane] : make_uint2(0, 0);
    auto patch = [&](int seg_begin, int seg_count) {
        return PlaneSrc{g.segs + seg_begin, seg_count, rowed, coled, g.A + (a_row + row0) * g.ld,
                        g.B + (b_row + col0) * g.ld, g.ld, g.za + a_row + row0 + lane, g.zb + b_row + col0 + lane,
                        g.a_rows, g.b_rows, C + (int64_t)lane * ldc};
    };
    const PlaneSrc src = patch(t.seg_begin, t.seg_count);
    const uint32_t valid = 0xffffffffu >> (32 - cols);
    const uint32_t bad_cols = __ballot_sync(0xffffffffu, ec < 0);
    const bool any_bad = __any_sync(0xffffffffu, er < 0) || bad_cols;
    const uint32_t mr = __reduce_max_sync(0xffffffffu, rt.y), mc = __reduce_max_sync(0xffffffffu, ct.y);
    if (!any_bad && (mr <= 2 || mc <= 2)) {
        if (mr <= 2) fx::sparse_outputs<true, 16>(src, rowed, cols);
        else fx::sparse_outputs<false, 16>(src, rowed, cols);
        return rowed ? valid : 0u;
    }
    const uint32_t fewest = __reduce_min_sync(0xffffffffu, min(rt.y - 1, ct.y - 1)) + 1;     // (zeros last)
    const float least = fx::least_sum((float)fewest, __uint_as_float(__reduce_max_sync(0xffffffffu, rt.x)),
                                      __uint_as_float(__reduce_max_sync(0xffffffffu, ct.x)));
    // (a part of a split tile decides on the whole contraction, whose rows' scales it has)
    const SplitTile* whole = t.split ? &g.split_tiles[t.split >> 9] : nullptr;
    uint32_t need = fx::weak_outputs(whole ? patch(whole->seg_begin, whole->seg_count) : src, rows, cols,
                                     __ballot_sync(0xffffffffu, rt.y != 0), __ballot_sync(0xffffffffu, ct.y != 0),
                                     max(er, 0), max(ec, 0), least);
    need = rowed ? (need | bad_cols | (er < 0 ? 0xffffffffu : 0u)) & valid : 0u;
    if (__any_sync(0xffffffffu, need != 0)) fx::fp64_outputs(src, rowed, cols, need, any_bad);
    return need;
}

// The same for all patches of a task and batch entry, a block each, a warp per patch.
constexpr int WEAK_WARPS = 4;
__global__ void __launch_bounds__(32 * WEAK_WARPS) weak_plane_kernel(const __grid_constant__ PlaneArgs g) {
    const GemmTask t = g.tasks[blockIdx.x];
    const int lane = threadIdx.x & 31, bat = blockIdx.y;
    const int wpr = (t.n + 31) / 32, patches = (t.m + 31) / 32 * wpr;
    int64_t ldc;
    double* const C = task_out(g, t, bat, ldc);
    uint32_t* const bits = g.fp64 + bat * g.fp64_words + g.fp64_at[blockIdx.x];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int p = threadIdx.x >> 5; p < patches; p += WEAK_WARPS) {
        const int row0 = p / wpr * 32, col0 = p % wpr * 32;
        const uint32_t need = check_patch(g, t, g.b0 + bat, row0, col0, t.m - row0, min(t.n - col0, 32),
                                          C + (int64_t)row0 * ldc + col0, ldc);
        if (lane < t.m - row0) bits[(row0 + lane) * wpr + col0 / 32] = need;
    }
}

// CHECK: with the check in the drain warps; else weak_plane_kernel has run.
template <bool CHECK>
__global__ void __launch_bounds__(PTHREADS, 1) fx_plane_kernel(const __grid_constant__ PlaneArgs g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* fullA = reinterpret_cast<uint64_t*>(smem + OFF_BAR);    // [stage][pair]
    uint64_t* emptyA = fullA + P_STAGES * PAIRS;
    uint64_t* fullB = emptyA + P_STAGES * PAIRS;                      // [stage]
    uint64_t* emptyB = fullB + P_STAGES;
    uint64_t* tfull = emptyB + P_STAGES;
    uint64_t* tempty = tfull + 1;
    uint64_t* drain = tempty + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int s = 0; s < P_STAGES * PAIRS; ++s) { mbar_init(&fullA[s], 1); mbar_init(&emptyA[s], 1); }
        for (int s = 0; s < P_STAGES; ++s) { mbar_init(&fullB[s], 1); mbar_init(&emptyB[s], 1); }
        mbar_init(tfull, 1);
        mbar_init(tempty, DW);
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tmem_slot, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t base = su32(smem);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long total = (long)g.ntasks * g.nbatch;
    auto task_at = [&](long item) { return g.tasks[item / g.nbatch]; };

    if (warp == 0 && lane == 0) {
        // ------------------------------------------------ TMA
        uint32_t step = 0;                 // K blocks
        uint32_t nb = 0, na = 0;           // loads of B and of A slots issued
        bool ok = true;
        GemmTask nt = blockIdx.x < total ? task_at(blockIdx.x) : GemmTask{};
        for (long item = blockIdx.x; item < total && ok; item += gridDim.x) {
            const GemmTask t = nt;
            if (item + gridDim.x < total) nt = task_at(item + gridDim.x);
            if (t.m == 0) continue;
            const int b = g.b0 + (int)(item % g.nbatch);
            const int ar = (int)(t.a_row + b * g.a_batch_rows), br = (int)(t.b_row + b * g.b_batch_rows);
            const int n16 = (t.n + 15) & ~15;
            const int ia = t.m <= 32 ? 0 : (t.m <= 64 ? 1 : 2);
            const CUtensorMap *ma = &g.a[ia], *mb = &g.b[n16 / 16 - 1];
            const uint32_t abox = (uint32_t)(32 << ia) * 128, bbytes = (uint32_t)(FD * n16 * 64);
            const int64_t avr = (g.ld / KPAD) * g.a_rows;
            KSeg sn = t.seg_count > 0 ? g.segs[t.seg_begin] : KSeg{};
            for (int s = 0; s < t.seg_count && ok; ++s) {
                const KSeg sg = sn;
                if (s + 1 < t.seg_count) sn = g.segs[t.seg_begin + s + 1];
                for (int kb = sg.k0 / KPAD; kb < (sg.k0 + sg.klen) / KPAD && ok; ++kb, ++step) {
                    const uint32_t st = step % P_STAGES, ph = (step / P_STAGES) & 1;
                    if (!(ok = mbar_wait(&emptyB[st], ph ^ 1, abort_flag, g.err))) break;
                    expect_tx(&fullB[st], bbytes);
                    tma_3d(base + OFF_B + st * B_STAGE, mb, &fullB[st], 0, (int)(kb * g.b_rows + br), 0);
                    ++nb;
                    for (int p = 0; p < PAIRS; ++p) {
                        const uint32_t sl = st * PAIRS + p;
                        if (!(ok = mbar_wait(&emptyA[sl], ph ^ 1, abort_flag, g.err))) break;
                        // tiles of up to 32 or 64 rows: the rows four times or twice (see the drain)
                        expect_tx(&fullA[sl], A_SLOT);
                        for (uint32_t o = 0; o < (uint32_t)A_SLOT; o += abox)
                            tma_2d(base + sl * A_SLOT + o, ma, &fullA[sl], 0, (int)(p * avr + kb * g.a_rows + ar));
                        ++na;
                    }
                }
            }
        }
        if (!ok) {
            // aborted: wait (bounded) for the loads in flight, the last fill of each slot, before the
            // shared memory goes away
            for (uint32_t i = 1; i <= P_STAGES && i <= nb; ++i) {
                const uint32_t f = nb - i;
                mbar_wait_drain(&fullB[f % P_STAGES], (f / P_STAGES) & 1);
            }
            for (uint32_t i = 1; i <= P_STAGES * PAIRS && i <= na; ++i) {
                const uint32_t f = na - i;
                mbar_wait_drain(&fullA[f % (P_STAGES * PAIRS)], (f / (P_STAGES * PAIRS)) & 1);
            }
        }
    } else if (warp == 1 && lane == 0) {
        // ------------------------------------------------ MMA
        uint32_t step = 0, ccount = 0;
        bool ok = true;
        GemmTask nt = blockIdx.x < total ? task_at(blockIdx.x) : GemmTask{};
        for (long item = blockIdx.x; item < total && ok; item += gridDim.x) {
            const GemmTask t = nt;
            if (item + gridDim.x < total) nt = task_at(item + gridDim.x);
            if (t.m == 0) continue;
            const int n16 = (t.n + 15) & ~15, nkb = t.ktotal / KPAD;
            for (int k = 0; k < nkb && ok; ++k, ++step) {
                const uint32_t st = step % P_STAGES, ph = (step / P_STAGES) & 1;
                const bool fresh = k % PCH == 0;
                if (fresh) {
                    if (!(ok = mbar_wait(tempty, (ccount & 1) ^ 1, abort_flag, g.err))) break;
                    tc_fence_after();
                }
                if (!(ok = mbar_wait(&fullB[st], ph, abort_flag, g.err))) break;
                const uint64_t db = sdesc64(base + OFF_B + st * B_STAGE);
                const uint64_t da = sdesc128(base + st * PAIRS * A_SLOT);
#pragma unroll
                for (int p = 0; p < PAIRS; ++p) {
                    const uint32_t sl = st * PAIRS + p;
                    if (!(ok = mbar_wait(&fullA[sl], ph, abort_flag, g.err))) break;
                    tc_fence_after();
                    const uint64_t a = da + p * (A_SLOT >> 4);
                    if (p == 0) issue<0>(n16, tmem, a, db, fresh);
                    else if (p == 1) issue<1>(n16, tmem, a, db, false);
                    else if (p == 2) issue<2>(n16, tmem, a, db, false);
                    else issue<3>(n16, tmem, a, db, false);
                    umma_commit(&emptyA[sl]);
                }
                if (!ok) break;
                umma_commit(&emptyB[st]);
                if (k % PCH == PCH - 1 || k + 1 == nkb) {
                    umma_commit(tfull);
                    ++ccount;
                }
            }
        }
        if (!ok) {
            umma_commit(drain);
            mbar_wait_drain(drain, 0);
        }
    } else if (warp >= 2) {
        // ------------------------------------------------ drain
        // A warp's instructions go by columns, and it reaches the 32 tensor-memory lanes of its quarter
        // only: a tile of at most 32 (64) rows would leave its drain to two (four) of the eight warps.
        // Its rows therefore fill all four quarters, four times (twice), at no cost to the MMAs, and
        // the quarters take different columns.
        const int q = warp & 3, h = (warp - 2) >> 2;         // tensor-memory lanes, half of the warps
        double* tr = reinterpret_cast<double*>(smem + OFF_TR + (warp - 2) * TR_WARP);
        uint32_t ccount = 0;
        bool ok = true;
        GemmTask nt = blockIdx.x < total ? task_at(blockIdx.x) : GemmTask{};
        for (long item = blockIdx.x; item < total && ok; item += gridDim.x) {
            const GemmTask t = nt;
            if (item + gridDim.x < total) nt = task_at(item + gridDim.x);
            if (t.m == 0) continue;
            const int bat = (int)(item % g.nbatch), b = g.b0 + bat;
            const int64_t a_row = t.a_row + b * g.a_batch_rows, b_row = t.b_row + b * g.b_batch_rows;
            const int n16 = (t.n + 15) & ~15, nkb = t.ktotal / KPAD;
            const int rep = t.m <= 32 ? 4 : (t.m <= 64 ? 2 : 1);
            const int row0 = 32 * (rep == 4 ? 0 : (rep == 2 ? q & 1 : q));            // this warp's rows
            const int wc = 32 / rep, colb = wc * (rep == 4 ? 2 * q + h : (rep == 2 ? 2 * (q >> 1) + h : h));   // and columns
            const int rows = t.m - row0 < 32 ? t.m - row0 : 32;                        // may be <= 0
            int64_t ldc;
            double* C = task_out(g, t, bat, ldc);
            C += (int64_t)row0 * ldc;
            const int ncols = t.n + t.n_zero;
            // scales of this lane's row and of this lane's column
            const int ncol = min(wc, t.n - colb);                                       // may be <= 0
            const bool rowed = lane < rows && ncol > 0, coled = lane < ncol && rows > 0;
            const int er = rowed ? g.ea[a_row + row0 + lane] : fx::E_ZERO;
            const int ec = coled ? g.eb[b_row + colb + lane] : fx::E_ZERO;
            // outputs that are there already (check_patch); `whole`: all of the patch, whose sums are left alone
            double* const out = C + (int64_t)lane * ldc + colb;
            const uint32_t valid = ncol > 0 ? 0xffffffffu >> (32 - ncol) : 0u;
            uint32_t need = 0;
            if (CHECK) {
                if (rows > 0 && ncol > 0) need = check_patch(g, t, b, row0, colb, rows, ncol, C + colb, ldc);
            } else if (rowed) {
                need = g.fp64[bat * g.fp64_words + g.fp64_at[item / g.nbatch] + (row0 + lane) * ((t.n + 31) / 32) + colb / 32] >>
                       (colb % 32) & valid;
            }
            const bool whole = __all_sync(0xffffffffu, !rowed || need == valid);
            uint32_t w0[32], w1[32], w2[32];
#pragma unroll
            for (int c = 0; c < 32; ++c) { w0[c] = 0; w1[c] = 0; w2[c] = 0; }
            for (int k = 0; k < nkb; k += PCH) {
                if (!(ok = mbar_wait(tfull, ccount & 1, abort_flag, g.err))) break;
                ++ccount;
                tc_fence_after();
                const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + colb;
#pragma unroll
                for (int c = 0; c < 32; c += 4) {
                    if (c < wc && colb + c < n16 && rows > 0 && !whole) {
                        uint32_t d[FD][4];
#pragma unroll
                        for (int e = 0; e < FD; ++e) tmem_ld4(ta + e * n16 + c, d[e]);
                        tmem_wait(d);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
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
            if (rows <= 0) continue;
            // exponent codes of T: this lane's row, per 8 columns
            uint16_t* et = !g.to_y ? g.et + (t.c_off % t.ldc) / CODE_COLS * g.et_rows + t.c_off / t.ldc + row0 + lane +
                                         (int64_t)b * g.c_batch_rows : nullptr;
            // 8 columns at a time: FP64 values into the transpose, then row pieces of 64 bytes
#pragma unroll
            for (int c0 = 0; c0 < 32; c0 += 8) {
                const int col0 = colb + c0;
                if (c0 < wc && col0 < ncols) {
                    int code = 0;
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const int e = __shfl_sync(0xffffffffu, ec, c0 + c);
                        double v = 0.0;
                        if ((need >> (c0 + c)) & 1u) v = out[c0 + c];
                        else if (col0 + c < t.n) v = fx::from_fixed(w2[c0 + c], w1[c0 + c], w0[c0 + c], er + e - 2112);
                        code = max(code, code_of(v));
                        tr[lane * 9 + c] = v;
                    }
                    if (et && lane < rows) et[col0 / CODE_COLS * g.et_rows] = (uint16_t)code;
                    __syncwarp();
                    const int c = lane & 7;
                    if (col0 + c < ncols)
                        for (int r = lane >> 3; r < rows; r += 4) C[(int64_t)r * ldc + col0 + c] = tr[r * 9 + c];
                    __syncwarp();
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ------------------------------------------------------------------ host side
int plane_map(CUtensorMap* m, void* base, bool a_side, int64_t vrows, int box_rows) {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        if (!fn) return fail(HEFF_ERR_CUDA, "cuTensorMapEncodeTiled is unavailable");
    }
    CUresult r;
    cuuint32_t estr[3] = {1, 1, 1};
    if (a_side) {
        cuuint64_t dims[2] = {64, (cuuint64_t)(PAIRS * vrows)}, strides[1] = {128};
        cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    } else {
        cuuint64_t dims[3] = {32, (cuuint64_t)vrows, FD}, strides[2] = {64, (cuuint64_t)vrows * 64};
        cuuint32_t box[3] = {32, (cuuint32_t)box_rows, FD};
        r = fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    }
    return r == CUDA_SUCCESS ? HEFF_OK : fail(HEFF_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
}

}  // namespace

int launch_digits(heff_plan* p, int array, void* ws, int nbatch, void* stream) {
    const FxOperand& o = p->fxo[array];
    if (o.units.empty()) return HEFF_OK;
    char* w = static_cast<char*>(ws);
    DigitArgs g{};
    g.units = o.d_units;
    g.segs = o.d_segs;
    g.src = reinterpret_cast<const double*>(w + o.off_src);
    g.ld = o.ld;
    g.codes = reinterpret_cast<const uint16_t*>(w + o.off_codes);
    g.code_cols = o.code_cols;
    g.planes = w + o.off_planes;
    g.scale = reinterpret_cast<int32_t*>(w + o.off_scale);
    g.rows = o.rows;
    g.batch_rows = o.batch_rows;
    g.a_side = o.a_side;
    g.nonzero = reinterpret_cast<uint32_t*>(w + o.off_nonzero);
    g.total = reinterpret_cast<uint2*>(w + o.off_total);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)o.units.size(), (unsigned)(o.batch_rows ? nbatch : 1));
    cfg.blockDim = dim3(256);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cfg.attrs = at;
    cfg.numAttrs = HEFF_PDL ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, digit_kernel, g);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "digit launch: %s", cudaGetErrorString(e));
    count_launches(1);
    return HEFF_OK;
}

int launch_fx_planes(heff_plan* p, int which, void* ws, void* const* y, int nbatch, void* stream) {
    const GemmList& gl = which == 1 ? p->g1 : (p->kchunk ? p->sp2 : p->g2);
    if (gl.tasks.empty()) return HEFF_OK;
    static PerDevice done[2];
    int rc = raise_smem_limit(done[0], (const void*)fx_plane_kernel<false>, PSMEM);
    if (!rc) rc = raise_smem_limit(done[1], (const void*)fx_plane_kernel<true>, PSMEM);
    if (rc) return rc;
    char* w = static_cast<char*>(ws);
    // operand arrays: LW, XT (the environment update's site tensor), T, RW
    const int ia = p->env ? 1 : (which == 1 ? 0 : 2), ib = p->env ? (which == 1 ? 0 : 2) : (which == 1 ? 1 : 3);
    const FxOperand &A = p->fxo[ia], &B = p->fxo[ib], &T = p->fxo[2];
    if (which == 2) {
        rc = launch_digits(p, 2, ws, nbatch, stream);
        if (rc) return rc;
    }
    PlaneArgs g{};
    // the workspace's tensor maps: encoded once, kept for the last two workspaces
    int slot = p->fx_ws[0] == ws ? 0 : (p->fx_ws[1] == ws ? 1 : -1);
    if (slot < 0) {
        slot = p->fx_next;
        p->fx_next ^= 1;
        p->fx_ws[slot] = nullptr;
        for (int o = 0; o < 4; ++o) {
            const FxOperand& f = p->fxo[o];
            CUtensorMap* m = reinterpret_cast<CUtensorMap*>(p->fx_maps[slot][o]);
            for (int k = 0; k < (f.a_side ? 3 : 4) && !f.units.empty(); ++k)
                if ((rc = plane_map(&m[k], w + f.off_planes, f.a_side, f.ld / KPAD * f.rows,
                                    f.a_side ? 32 << k : 16 * (k + 1))))
                    return rc;
        }
        p->fx_ws[slot] = ws;
    }
    std::memcpy(g.a, p->fx_maps[slot][ia], sizeof(g.a));
    std::memcpy(g.b, p->fx_maps[slot][ib], sizeof(g.b));
    g.tasks = gl.d_tasks;
    g.segs = gl.d_segs;
    g.ntasks = (int)gl.tasks.size();
    g.ld = A.ld;
    g.a_rows = A.rows;
    g.b_rows = B.rows;
    g.a_batch_rows = A.batch_rows;
    g.b_batch_rows = B.batch_rows;
    g.ea = reinterpret_cast<const int32_t*>(w + A.off_scale);
    g.eb = reinterpret_cast<const int32_t*>(w + B.off_scale);
    g.za = reinterpret_cast<const uint32_t*>(w + A.off_nonzero);
    g.zb = reinterpret_cast<const uint32_t*>(w + B.off_nonzero);
    g.ta = reinterpret_cast<const uint2*>(w + A.off_total);
    g.tb = reinterpret_cast<const uint2*>(w + B.off_total);
    g.A = reinterpret_cast<const double*>(w + A.off_src);
    g.B = reinterpret_cast<const double*>(w + B.off_src);
    g.fp64 = reinterpret_cast<uint32_t*>(w + p->off_fp64);
    g.fp64_at = gl.d_fp64_at;
    g.fp64_words = gl.fp64_words();
    g.err = reinterpret_cast<int*>(w + p->off_flags);
    if (which == 1) {
        g.C = reinterpret_cast<double*>(w + T.off_src);
        g.c_batch_elems = p->rows_t * p->ld_t;
        g.c_batch_rows = p->rows_t;
        g.et = reinterpret_cast<uint16_t*>(w + T.off_codes);
        g.et_rows = T.rows;
    } else {
        g.to_y = 1;
        if (p->kchunk) {
            g.split = reinterpret_cast<double*>(w + p->off_split);
            g.split_tiles = gl.d_split;
            g.split_elems = gl.split_elems;
        }
    }
    for (int b0 = 0; b0 < nbatch; b0 += MAXB) {
        g.b0 = b0;
        g.nbatch = nbatch - b0 < MAXB ? nbatch - b0 : MAXB;
        if (which == 2)
            for (int b = 0; b < g.nbatch; ++b) g.y.p[b] = y[b0 + b];
        const long total = (long)g.ntasks * g.nbatch;
        const int nsm = p->num_sms > 0 ? p->num_sms : 148;
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = dim3((unsigned)(total < nsm ? total : nsm));
        cfg.blockDim = dim3(PTHREADS);
        cfg.dynamicSmemBytes = PSMEM;
        cfg.stream = static_cast<cudaStream_t>(stream);
        cfg.attrs = at;
        cfg.numAttrs = HEFF_PDL ? 1 : 0;
        // one tile a CTA: the check while its first loads arrive; more: in a launch of its own (m = 48, 10 Lanczos
        // steps: 683 and 749 us; apply m = 1024: 539 and 457)
        const bool inline_check = total <= nsm;
        cudaError_t e = cudaSuccess;
        if (!inline_check) {
            cudaLaunchConfig_t weak = cfg;
            weak.gridDim = dim3((unsigned)g.ntasks, (unsigned)g.nbatch);
            weak.blockDim = dim3(32 * WEAK_WARPS);
            weak.dynamicSmemBytes = 0;
            e = cudaLaunchKernelEx(&weak, weak_plane_kernel, g);
            count_launches(1);
        }
        if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, inline_check ? fx_plane_kernel<true> : fx_plane_kernel<false>, g);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "fx_plane launch: %s", cudaGetErrorString(e));
        count_launches(1);
        if (which == 2 && p->kchunk && (rc = launch_sum_parts(p, gl, ws, y + b0, g.nbatch, stream))) return rc;
    }
    return HEFF_OK;
}

}  // namespace heff
