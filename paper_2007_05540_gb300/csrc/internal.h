// Internal declarations shared by the host planner (plan.cpp, capi.cpp) and the
// CUDA translation units.  Nothing here is part of the C ABI.
#pragma once

#include <array>
#include <cstddef>
#include <cstdint>
#include <map>
#include <string>
#include <vector>

#include "../../include/heff.h"
#include "per_device.h"

namespace heff {

// Padding unit of every contraction (K) segment in the workspace operand arrays: one K
// block of the tensor-core kernel (64-byte swizzled rows: 32 bf16 or 16 fp32 elements;
// the FP64 kernel steps K by 16).  K tiles never straddle segments.
#ifndef HEFF_KPAD
#define HEFF_KPAD 32
#endif
constexpr int KPAD = HEFF_KPAD;

inline int64_t pad_up(int64_t v, int64_t p) { return (v + p - 1) / p * p; }

// Programmatic dependent launch of the matvec's kernels (pack, GEMM 1, GEMM 2): each may be
// scheduled while its predecessor on the stream finishes, runs its prologue (barriers,
// tensor memory), and waits (griddepcontrol.wait) before it touches global memory that
// the predecessor or earlier work writes or reads.  0 launches them in plain stream order.
#ifndef HEFF_PDL
#define HEFF_PDL 1
#endif

int fail(int code, const char* fmt, ...);
void clear_error();
void count_launches(int64_t n);

struct IndexDesc {
    int nsec = 0, nq = 0, flow = 1;
    std::vector<int32_t> charges;   // nsec * nq
    std::vector<int32_t> dims;      // nsec
    std::vector<int32_t> q(int s) const {
        return std::vector<int32_t>(charges.begin() + s * nq, charges.begin() + (s + 1) * nq);
    }
    int find(const std::vector<int32_t>& qv) const;
    bool same_sectors(const IndexDesc& o) const { return charges == o.charges && dims == o.dims; }
};

// ---------------------------------------------------------------- device tables
// x block -> XT (x transposed per charge sector, contraction index contiguous)
struct PackTile {
    int64_t x_off;     // element offset of the x block (rows a, cols b, row-major)
    int64_t xt_row0;   // XT row of b = 0 of this block
    int32_t xt_col0;   // XT column of a = 0 of this block
    int32_t m_a, m_b;  // block dims
    int32_t a_pad;     // padded extent of a (multiple of KPAD): columns [m_a, a_pad) get 0
    int32_t a0, b0;    // origin of this 32 x 32 tile inside the block
};

// LW / RW preparation: dst[r][c] = sum_t W[w_idx_t] * src[src_off_t + r * cols + c]
struct MixTile {
    int64_t dst_row0;  // first destination row in LW or RW
    int32_t dst_col0;  // first destination column (segment start)
    int32_t rows, cols, cols_pad;
    int32_t r0, nrows; // row range handled by this tile
    int32_t term_begin, term_count;
    int32_t which;     // 0: L with W1 into LW, 1: R with W2 into RW
};
struct MixTerm {
    int64_t src_off;   // element offset of the environment block
    int32_t w_idx;     // element index into the MPO buffer; -1: coefficient 1 (a plain copy)
    int32_t pad_;
};

// One output tile C[m x n] = sum over segments of A[a_row.., k0:k0+klen] . B[b_row.., k0:k0+klen]^T
struct GemmTask {
    int64_t a_row, b_row;   // first row of the tile in the A and B operand arrays
    int64_t c_off;          // element offset of the tile origin in the output
    int32_t m, n;           // valid rows / columns of the tile
    int32_t ldc;            // output row pitch (elements)
    int32_t n_zero;         // columns [n, n + n_zero) of the tile are written as 0 (padding)
    int32_t seg_begin, seg_count;
    int32_t ktotal;         // sum of the segments' klen (padded contraction length)
    int32_t split;          // 0, or one of several parts of the tile's contraction (split_code)
};
// A tile whose contraction is split over several tasks: group (of the list), part, number of parts.
// Each part leaves its sum in the group's scratch, and sum_parts_kernel adds them in order.
struct SplitTile {
    int64_t c_off, off;     // tile origin in y; the group's scratch (parts x m x n elements)
    int32_t ldc, m, n, parts;
    int32_t seg_begin, seg_count;   // segments of the whole contraction
};
constexpr int SPLIT_MAX = 16;
inline int32_t split_code(int group, int part, int parts) { return group << 9 | part << 5 | parts; }
struct KSeg {
    int32_t k0, klen;       // column range shared by A and B (klen multiple of KPAD)
};

// ---------------------------------------------------------------- block-product engine
// One output tile C[m x n] = scale * sum over its products of
//   coef * A[a_off + r * a_rs + k * a_cs] * B[b_off + k * b_rs + c * b_cs],  k < K,
// coef = (c1 < 0 ? 1 : coef1[c1]) * (c2 < 0 ? 1 : coef2[c2]).
struct BProd {
    int64_t a_off, b_off;
    int32_t a_rs, a_cs, b_rs, b_cs;
    int32_t K;
    int32_t c1, c2;
    int32_t ea, eb;         // FP64 lists: exponent codes of the A rows and of the B columns
    int32_t za, zb, na, nb; // and words of nonzero elements, and rows of a view
};
struct BTile {
    int64_t c_off;
    int32_t ldc, m, n;
    int32_t prod_begin, prod_count;
    int32_t steps;          // FP64 lists: steps of 16 contraction elements, each product rounded up
    int32_t fp64_at;        // FP64 lists: first word of the bits for outputs computed in FP64
};
// up to 32 rows of one operand view whose exponent codes and nonzero elements an FP64 list needs
struct FxRows {
    int64_t off;
    int32_t rs, ks, rows, K;
    int32_t out;            // first code
    int32_t which;          // 0: A, 1: B
    int32_t word, all;      // first word of nonzero elements, and rows of the view
};
// output tile of the FP64 products (fx_gemm.cu, fx_planes.cu)
constexpr int FX_TILE_M = 128, FX_TILE_N = 64;
struct BList {
    std::vector<BTile> tiles;
    std::vector<BProd> prods;
    char* d_tables = nullptr;  // the device tables' one allocation
    BTile* d_tiles = nullptr;
    BProd* d_prods = nullptr;
    double flops = 0;
    bool accumulate = false;   // C += result instead of C = result
    // output tile shape the block list is cut into: FP64 products, or 128 x 128 (tensor cores, BF16x3)
    int tile_m = FX_TILE_M, tile_n = FX_TILE_N;
    // FP64 products: the operand rows and columns whose exponent codes they need, one slot per
    // row of each distinct view of an operand block; the codes are recomputed on every call
    std::vector<FxRows> rows;
    FxRows* d_rows = nullptr;
    uint16_t* d_codes = nullptr;
    float* d_sums = nullptr;        // of a row's magnitudes, over its scale, rounded up
    uint32_t* d_fp64 = nullptr;     // outputs computed in FP64: a word per row and 32 columns of a tile
    int32_t nfp64 = 0;
    int* d_err = nullptr;      // a flag for launches that have none elsewhere, zero after the upload
    uint32_t* d_words = nullptr;    // nonzero elements, [32 elements][row] of a view
    int32_t ncodes = 0, nwords = 0;
    struct View { int32_t code, word; };
    std::map<std::array<int64_t, 6>, View> views;
    int num_sms = 0;
    View view(int which, int64_t off, int32_t rs, int32_t ks, int32_t n, int32_t K);
    // the output blocks as added (products given for the block origin), kept for re-tiling
    struct Block { int64_t c_off; int32_t ldc, m, n, prod_begin, prod_count; };
    std::vector<Block> blocks;
    std::vector<BProd> block_prods;
    // append the tiles of an m x n output block whose products are given for the block origin
    void add_block(int64_t c_off, int32_t ldc, int32_t m, int32_t n, const std::vector<BProd>& ps);
    // cut every block again into tm x tn tiles (the device tables must be re-uploaded)
    void retile(int tm, int tn);
};
int blist_upload(BList& b);
void blist_free(BList& b);
// the list's products in FP64 accuracy (fixed-point digits on the tensor cores, fx_gemm.cu); err:
// device int raised when a bounded wait expires
int launch_bgemm(const BList& b, const double* A, const double* B, double* C, const double* coef1,
                 const double* coef2, double scale, void* stream, int* err, const double* inv_scale = nullptr);
// the same products on the tensor cores (BF16x3 split, FP32 accumulation; blockops_tc.cu)
// on FP32 copies of the operands (launch_convert_f64_f32), with an FP32 (c_f64 false) or
// FP64 output; needs 128 x 128 tiles (retile); err: device int raised when a bounded wait
// expires
int launch_bgemm_tc(const BList& b, const float* A, const float* B, void* C, bool c_f64, const double* coef1,
                    const double* coef2, double scale, void* stream, const double* inv_scale, int* err);
// dst[i] = src[i] rounded to FP32 (round to nearest even, on the integer pipes)
int launch_convert_f64_f32(const double* src, float* dst, int64_t n, void* stream);
// out[j] = scale * sum over the dots d in [off[j], off[j+1]) of <X[x_off..], Y[y_off..]>
// (dots sorted by output index; scratch holds one double per dot)
struct BDot {
    int64_t x_off, y_off;
    int64_t len;
};
// (accumulate: out[j] += instead of out[j] =)
int launch_block_dots(const BDot* d_dots, int ndots, const int32_t* d_off, const double* X, const double* Y,
                      double* out, int nout, double* scratch, double scale, void* stream, bool accumulate = false);
int launch_block_dots_f32(const BDot* d_dots, int ndots, const int32_t* d_off, const float* X, const float* Y,
                          double* out, int nout, double* scratch, double scale, void* stream, bool accumulate = false);

constexpr int MAXB = 64;   // batch entries per launch (kernel parameter arrays)
struct PtrBatch { const void* p[MAXB]; };

struct GemmList {
    std::vector<GemmTask> tasks;
    std::vector<KSeg> segs;
    GemmTask* d_tasks = nullptr;
    KSeg* d_segs = nullptr;
    int tm = 0, tn = 0;
    int cl = 1;             // CTAs per entry: 2 = tasks 2e, 2e + 1 share their B tile (cluster pair)
    double flops = 0;       // executed (valid m, n; padded K)
    double useful = 0;      // valid m, n and unpadded K
    // split tiles, one per group, and the elements of their scratch
    std::vector<SplitTile> split;
    SplitTile* d_split = nullptr;
    int64_t split_elems = 0;
    // FP64 lists: first word of each task's bits for outputs computed in FP64 (a word per row and 32 columns)
    std::vector<int32_t> fp64_at;
    int32_t* d_fp64_at = nullptr;
    void count_fp64() {
        fp64_at.assign(1, 0);
        for (const GemmTask& t : tasks) fp64_at.push_back(fp64_at.back() + t.m * ((t.n + 31) / 32));
    }
    int64_t fp64_words() const { return fp64_at.empty() ? 0 : fp64_at.back(); }
    // host only, one entry per task: output left sector a' and the task's flop counts
    std::vector<int32_t> owner;
    std::vector<double> task_flops, task_useful;
};

// The tasks of a GEMM list by merge class (batched launches, tc_gemm.cu): class c holds the tasks
// [first[c], first[c + 1]), longest first
struct MergeList {
    std::vector<GemmTask> tasks;
    GemmTask* d_tasks = nullptr;
    int first[7] = {0, 0, 0, 0, 0, 0, 0};
};

// An FP64 plan's operand array as digit planes (fx_planes.cu).  Units: up to 8 rows that share their
// column segments (the ones that are written and read).
struct FxUnit {
    int64_t row0;
    int32_t nrows, seg_begin, seg_count;
};
struct FxOperand {
    std::vector<FxUnit> units;
    std::vector<KSeg> segs;
    FxUnit* d_units = nullptr;
    KSeg* d_segs = nullptr;
    int64_t ld = 0, rows = 0, batch_rows = 0;     // rows: of all batch entries; 0 batch_rows: shared by them
    bool a_side = false;
    int code_cols = KPAD;           // columns per exponent code
    size_t off_src = 0, off_codes = 0, off_planes = 0, off_scale = 0, off_nonzero = 0, off_total = 0;    // in the workspace
    // rows [row0, row0 + n) over the given segments
    void add(int64_t row0, int n, const std::vector<KSeg>& s) {
        const int32_t sb = (int32_t)segs.size();
        segs.insert(segs.end(), s.begin(), s.end());
        for (int r = 0; r < n; r += 8) units.push_back({row0 + r, n - r < 8 ? n - r : 8, sb, (int32_t)s.size()});
    }
};
// the largest workspace with digit planes (16 bytes per operand element beside 8)
constexpr size_t FX_PLANES_MAX = (size_t)64 << 30;
// columns per exponent code of T where fx_planes.cu writes it (eight columns go through its drain at a time)
constexpr int FX_T_CODE_COLS = 8;

}  // namespace heff

struct heff_layout {
    std::vector<heff::IndexDesc> idx;
    std::vector<int32_t> target;
    int nq = 0;
    std::vector<int32_t> keys;      // nblocks * nidx
    std::vector<int64_t> offsets;   // nblocks
    int64_t nelem = 0;
    std::map<std::vector<int32_t>, int64_t> block_of;
    int64_t offset_of(const std::vector<int32_t>& key) const {
        auto it = block_of.find(key);
        return it == block_of.end() ? -1 : offsets[it->second];
    }
};

struct heff_plan {
    heff_plan_opts opts{};
    int planes = 1;           // values per operand element in the workspace (hi and lo: 2)
    int esize = 8;            // bytes per value
    int64_t nelem_x = 0, nelem_L = 0, nelem_R = 0, nelem_W1 = 0, nelem_W2 = 0;
    // operand arrays (rows x pitch columns; a row holds planes x pitch values, the split
    // precisions' hi and lo interleaved by K block)
    int64_t rows_x = 0, ld_x = 0, rows_lw = 0, rows_t = 0, ld_t = 0, rows_rw = 0;
    // workspace byte offsets
    size_t off_xt = 0, off_lw = 0, off_t = 0, off_rw = 0, off_flags = 0, ws_bytes = 0;
    double flops_canonical = 0;
    std::vector<int32_t> shard_sectors;   // left sectors a' of y this plan computes
    // device tables: one allocation, the pointers below into it
    void* d_tables = nullptr;
    std::vector<heff::PackTile> pack;
    std::vector<heff::MixTile> mix;
    std::vector<heff::MixTerm> terms;
    heff::PackTile* d_pack = nullptr;
    heff::MixTile* d_mix = nullptr;
    heff::MixTerm* d_terms = nullptr;
    // MPO entries the schedule dropped (exactly zero in the host copies), for heff_plan_check_mpo
    std::vector<int32_t> w1_zero, w2_zero;
    int32_t* d_w1_zero = nullptr;
    int32_t* d_w2_zero = nullptr;
    unsigned long long* d_wcount = nullptr;
    heff::GemmList g1, g2;            // active task lists
    heff::GemmList g1_alt, g2_alt;    // the other tile width (tensor-core paths), see heff_plan_autotune
    heff::GemmList g1_pair, g2_pair;  // N = 256 tiles in CTA pairs sharing B (tensor-core paths)
    // the environment update's plan (env.cu): GEMM 1 contracts XT with LW into T, GEMM 2 XT with T;
    // there is no RW, and which = 1 mix tiles fill XT
    bool env = false;
    // FP64 plans: exponent codes of the operand arrays, [column / KPAD][row], after the arrays and the
    // flags (ws_min: the workspace up to here, enough without digit planes)
    size_t off_ex = 0, off_elw = 0, off_et = 0, off_erw = 0, ws_min = 0;
    // split tiles of GEMM 2: chunk of the contraction (in KPAD units; 0: no limit) and their scratch in
    // the workspace (after ws_min too).
    // sp2, sp2_alt: the N = 256 (FP64: FX_TILE_N) and N = 128 lists of GEMM 2 with their long tiles split (g2
    // and g2_alt describe them whole)
    heff::GemmList sp2, sp2_alt;
    int kchunk = 0;
    size_t off_split = 0;
    // FP64 plans: LW, XT, T, RW as digit planes, last in the workspace (planes_ok: whether it has them), and
    // their tensor maps for the last two workspaces
    heff::FxOperand fxo[4];
    bool planes_ok = false;
    size_t off_fp64 = 0;
    void* fx_ws[2] = {nullptr, nullptr};
    int fx_next = 0;
    alignas(64) unsigned char fx_maps[2][4][4 * 128];
    int64_t stats[24] = {0};
    // tensor-map cache for the tensor-core path: two entries keyed by workspace pointer
    // (two streams alternating workspaces reuse their maps), replaced round-robin
    void* tmap_ws[2] = {nullptr, nullptr};
    int tmap_next = 0;
    alignas(64) unsigned char tmaps[2][24][128];
    heff::MergeList mg1, mg2;  // max_batch > 1, split precisions: the N = 256 tasks by merge class
    int device = 0;
    int num_sms = 0;
    bool uploaded = false;    // false: created without a CUDA device (inspection only)
    // phase timers: events recorded around prepare, pack, GEMM 1, GEMM 2 when enabled
    bool timing = false;
    void* ev[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    bool ev_prepare = false;  // whether the last call ran the prepare phase
};

namespace heff {
// A kernel's dynamic shared memory limit on the current device (done: the kernel's marks); apply.cu
int raise_smem_limit(PerDevice& done, const void* kernel, int bytes);
// The error flag of a workspace: an int that a kernel whose bounded wait expires sets to 1, before seven more that
// show that the flag was ever initialised (a workspace is the caller's memory); apply.cu.
constexpr size_t FLAG_BYTES = 32;
int reset_flag(void* flag, void* stream);
// HEFF_ERR_TIMEOUT where the flag is raised (cleared then), else HEFF_OK; synchronises
int read_flag(void* flag, const char* what, void* stream);
// launchers (apply.cu)
// planes: an FP64 plan's call has the digit planes and the operands' exponent codes in its workspace; without
// them its products run on the FP64 units
bool has_planes(const heff_plan* p, size_t ws_bytes);
int launch_pack_batch(heff_plan* p, const void* const* x, int nbatch, void* ws, bool planes, void* stream);
int launch_mix(heff_plan* p, const void* L, const void* W1, const void* W2, const void* R,
               void* ws, bool planes, void* stream);
int launch_gemm(heff_plan* p, int which, void* ws, void* const* y, int nbatch, bool planes, void* stream);
int launch_digits(heff_plan* p, int array, void* ws, int nbatch, void* stream);
int launch_fx_planes(heff_plan* p, int which, void* ws, void* const* y, int nbatch, void* stream);
// workspace of the digit planes from `end` on, and of fp64_words words of bits for FP64 outputs (offsets set);
// returns the new end, or `without` when the planes would pass FX_PLANES_MAX
size_t plane_layout(heff_plan* p, size_t end, int64_t fp64_words, size_t without);
// y's split tiles from their parts (batch entries [0, nbatch), scratch copies of split_elems)
int launch_sum_parts(heff_plan* p, const GemmList& g, void* ws, void* const* y, int nbatch, void* stream);
// one apply in the first `bytes` of ws, which may hold less than ws_bytes but at least ws_min
int apply_in(heff_plan* p, const void* L, const void* W1, const void* W2, const void* R, const void* x, void* y,
             void* ws, size_t bytes, void* stream);
void lpt_schedule(GemmList& G, int units, bool tc, bool first);
// KPAD units per part of GEMM 2's contractions that balances the list over the units (0: as is)
int split_chunk(const GemmList& G, int units, bool tc, int least, double uneven, int shortest);
void split_tasks(GemmList& G, int chunk);
// clusters of two tensor-core CTAs resident at once (tc_gemm.cu; num_sms / 2 without a device)
int tc_pair_clusters(int num_sms, int precision);
// one block waiting at the SVD sweeps' grid barrier set up for two (svd.cu; wait self-test)
void svd_barrier_selftest(unsigned int* bar, int* flag, void* stream);
int plan_upload(heff_plan* p);
void plan_free_device(heff_plan* p);
void record_phase(heff_plan* p, int k, void* stream);
}  // namespace heff
