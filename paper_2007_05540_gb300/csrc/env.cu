// Environment extension on the GPU (Section II-C: the left environment A and right
// environment B grow by one site as the sweep moves).
//
// Both sides have one form.  With i the sectors of env_old's bond, j those of env_new's, u and n
// their channels, S_j[b, (s, i) a] the site tensor as a matrix (out-bond state b, columns the
// site's state and in-bond state), and c(u, t, s, n) the entries of W:
//   Lnew[j', n, j] = S_j' . T^T,     T[(n, j', j) b, (t, i') a'] = S_j . LW^T               (GEMMs 2, 1)
//   LW[(n, t, i', j) a', (s, i) a] = sum_u c(u, t, s, n) env_old[i', u, i]                  (mix)
// so the update is one operator preparation and two grouped GEMMs over workspace operands with
// the contraction index contiguous: the kernels of the H_eff matvec (apply.cu, tc_gemm.cu,
// fx_planes.cu) run it from tables of the same form (heff_plan with env set).  W enters with the
// environment, before the GEMMs: a product per entry of W, as in the list form below, contracts the
// same site block with up to k blocks that differ by a coefficient.
//
// An update whose dense operands would take more than ENV_DENSE_MAX bytes of workspace runs as lists of
// block products instead (blockops.cu; spin, k = 14, m = 4096: 290 MB, where the dense form takes 1.5 GB, and
// 4.4 GB with the digit planes of FP64):
//   X[(a', w), (s, b)]  = L[a', w, a] . A[a, s, b],   Lnew[c, v, d] = sum W A[a', t, c]^T . X     (left)
//   Y[(b', v), (a, s)]  = R[b', v, b] . B[a, s, b]^T, Rnew[c, w, d] = sum W B[c, t, b'] . Y       (right)
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <memory>
#include <new>
#include <set>
#include <tuple>

#include "internal.h"

using heff::fail;
using heff::BList;
using heff::BProd;
using heff::GemmTask;
using heff::KPAD;
using heff::pad_up;

struct heff_env_plan {
    int side = 0;
    int precision = HEFF_PREC_FP64;   // of the block products
    double flops = 0;                 // of the list form (the block pairs of Algorithm 2)
    // Workspace: what HEFF_PREC_FP64 runs in at full speed, and the least, in which both precisions run (FP64
    // without digit planes, on the FP64 units: the planes are two thirds of it, and BF16x3 has no use for them).
    size_t ws_bytes = 0, ws_least = 0;
    int64_t n_env = 0, n_site = 0;
    bool device = false;              // created with a CUDA device
    // dense form: block-level tasks, and the tiles and device tables of the current precision
    bool dense = true;
    std::vector<GemmTask> blocks1, blocks2;
    std::vector<heff::KSeg> segs1, segs2;
    std::vector<std::tuple<int, int64_t, int, std::vector<heff::KSeg>>> units;   // array, row, rows, segments
    std::vector<heff::PackTile> pack;
    std::vector<heff::MixTile> mix;
    std::vector<heff::MixTerm> terms;
    int64_t rows_sp = 0, ld = 0, rows_lw = 0, rows_t = 0;
    std::unique_ptr<heff_plan> plan;
    // list form.  Workspace: [error flag, 256 B][intermediate X or Y][tensor-core precision only: FP32
    // copies of env_old and of the site tensor].  The FP64 products keep the intermediate in FP64;
    // the tensor-core products read FP32 copies and keep it in FP32.
    BList step1, step2;
    size_t off_x = 256, off_env32 = 0, off_site32 = 0;
};

namespace {

constexpr size_t ENV_DENSE_MAX = (size_t)64 << 30;

using Charge = std::vector<int32_t>;

bool same(const heff::IndexDesc& a, const heff::IndexDesc& b) { return a.same_sectors(b); }

Charge add(const Charge& a, const Charge& b, int sb = 1) {
    Charge r(a);
    for (size_t c = 0; c < r.size(); ++c) r[c] += sb * b[c];
    return r;
}

// Operand layout, block-level GEMM tasks and copy / mix tiles of the dense form, and the flop count of
// the list form.  c(u, t, s, n): index of the kept entry of W, or -1; nu: channels of env_old.
template <typename C>
void build_dense(heff_env_plan* P, const heff_layout* env_old, const heff_layout* site, const heff_layout* env_new,
                 const heff::IndexDesc& sa, const heff::IndexDesc& sp, const heff::IndexDesc& sb, int d, int nu, C c) {
    const bool left = P->side == 0;
    const heff::IndexDesc &in = left ? sa : sb, &out = left ? sb : sa;
    const int ni = in.nsec, nj = out.nsec, nn = env_new->idx[1].nsec;
    // the site blocks that the products use: (i, s) -> j and (j, t) -> i by charge
    auto off_of = [&](int i, int s, int j) { return left ? site->offset_of({i, s, j}) : site->offset_of({j, s, i}); };
    std::vector<int> out_of((size_t)ni * d, -1), in_of((size_t)nj * d, -1);
    for (int s = 0; s < d; ++s) {
        for (int i = 0; i < ni; ++i) {
            const int j = out.find(add(in.q(i), sp.q(s), left ? 1 : -1));
            if (j >= 0 && off_of(i, s, j) >= 0) out_of[(size_t)i * d + s] = j;
        }
        for (int j = 0; j < nj; ++j) {
            const int i = in.find(add(out.q(j), sp.q(s), left ? -1 : 1));
            if (i >= 0 && off_of(i, s, j) >= 0) in_of[(size_t)j * d + s] = i;
        }
    }
    // columns of S_j: one padded segment per site block
    std::map<std::tuple<int, int, int>, int32_t> col;          // (j, s, i)
    std::vector<int32_t> width(nj, 0);
    std::vector<int64_t> sp_row(nj, 0);
    int64_t rows = 0;
    for (int j = 0; j < nj; ++j) { sp_row[j] = rows; rows += out.dims[j]; }
    for (size_t b = 0; b < site->offsets.size(); ++b) {
        const int i = site->keys[b * 3 + (left ? 0 : 2)], s = site->keys[b * 3 + 1], j = site->keys[b * 3 + (left ? 2 : 0)];
        const int mi = in.dims[i], mj = out.dims[j], pad = (int)pad_up(mi, KPAD);
        const int32_t c0 = width[j];
        col[{j, s, i}] = c0;
        width[j] += pad;
        if (left) {                                             // stored a x b: transposed copy
            for (int a0 = 0; a0 < pad; a0 += 32)
                for (int b0 = 0; b0 < mj; b0 += 32)
                    P->pack.push_back({site->offsets[b], sp_row[j], c0, mi, mj, pad, a0, b0});
        } else {                                                // stored b x a: plain copy
            const int32_t tb = (int32_t)P->terms.size();
            P->terms.push_back({site->offsets[b], -1, 0});
            for (int r0 = 0; r0 < mj; r0 += 32)
                P->mix.push_back({sp_row[j], c0, mj, mi, pad, r0, std::min(32, mj - r0), tb, 1, 1});
        }
    }
    for (int j = 0; j < nj; ++j)
        if (width[j]) P->units.push_back({1, sp_row[j], (int)out.dims[j], {{0, width[j]}}});
    P->rows_sp = std::max<int64_t>(rows, 1);
    P->ld = KPAD;
    for (int j = 0; j < nj; ++j) P->ld = std::max<int64_t>(P->ld, width[j]);
    // LW row groups (n, t, i', j): segments (s, i) with their terms (u), from env_old's blocks; and the
    // intermediate blocks (i', u, s, j) of the list form, for its flop count
    struct Seg { int s, i; std::vector<heff::MixTerm> terms; };
    struct Group { int64_t row = -1; std::map<std::pair<int, int>, Seg> segs; };
    std::map<std::tuple<int, int, int, int>, Group> groups;
    std::set<std::tuple<int, int, int, int>> inter;
    for (size_t b = 0; b < env_old->offsets.size(); ++b) {
        const int ip = env_old->keys[b * 3], u = env_old->keys[b * 3 + 1], i = env_old->keys[b * 3 + 2];
        for (int s = 0; s < d; ++s) {
            const int j = out_of[(size_t)i * d + s];
            if (j < 0) continue;
            bool used = false;
            for (int t = 0; t < d; ++t)
                for (int n = 0; n < nn; ++n) {
                    const int32_t w = c(u, t, s, n);
                    if (w < 0) continue;
                    used = true;
                    Seg& sg = groups[{n, t, ip, j}].segs[{s, i}];
                    sg.s = s;
                    sg.i = i;
                    sg.terms.push_back({env_old->offsets[b], w, 0});
                }
            if (!used) continue;
            inter.insert({ip, u, s, j});
            P->flops += 2.0 * in.dims[ip] * out.dims[j] * in.dims[i];
        }
    }
    // env_new's blocks: T rows, GEMM 1 (one task per site state t of the bra), GEMM 2
    int64_t t_rows = 0, lw_rows = 0;
    for (size_t b = 0; b < env_new->offsets.size(); ++b) {
        const int jp = env_new->keys[b * 3], n = env_new->keys[b * 3 + 1], j = env_new->keys[b * 3 + 2];
        const int mjp = out.dims[jp], mj = out.dims[j];
        GemmTask g2{};
        g2.a_row = sp_row[jp];
        g2.b_row = t_rows;
        g2.m = mjp;
        g2.n = mj;
        g2.c_off = env_new->offsets[b];
        g2.ldc = mj;
        g2.seg_begin = (int32_t)P->segs2.size();
        for (int t = 0; t < d; ++t) {
            const int ip = in_of[(size_t)jp * d + t];
            if (ip < 0) continue;
            for (int u = 0; u < nu; ++u)
                for (int s = 0; s < d; ++s)
                    if (c(u, t, s, n) >= 0 && inter.count({ip, u, s, j})) P->flops += 2.0 * mjp * mj * in.dims[ip];
            auto it = groups.find({n, t, ip, j});
            if (it == groups.end()) continue;
            Group& g = it->second;
            const int mip = in.dims[ip], pad = (int)pad_up(mip, KPAD);
            const bool fresh = g.row < 0;
            if (fresh) {
                g.row = lw_rows;
                lw_rows += mip;
                for (auto& kv : g.segs) {
                    const Seg& sg = kv.second;
                    const int mi = in.dims[sg.i];
                    const int32_t tb = (int32_t)P->terms.size();
                    P->terms.insert(P->terms.end(), sg.terms.begin(), sg.terms.end());
                    for (int r0 = 0; r0 < mip; r0 += 32)
                        P->mix.push_back({g.row, col[{j, sg.s, sg.i}], mip, mi, (int32_t)pad_up(mi, KPAD), r0,
                                          std::min(32, mip - r0), tb, (int32_t)sg.terms.size(), 0});
                }
            }
            GemmTask g1{};
            g1.a_row = sp_row[j];
            g1.b_row = g.row;
            g1.m = mj;
            g1.n = mip;
            const int32_t c0 = col[{jp, t, ip}];
            g1.c_off = t_rows * P->ld + c0;
            g1.ldc = (int32_t)P->ld;
            g1.n_zero = pad - mip;
            g1.seg_begin = (int32_t)P->segs1.size();
            for (auto& kv : g.segs) {
                const int32_t len = (int32_t)pad_up(in.dims[kv.second.i], KPAD);
                P->segs1.push_back({col[{j, kv.second.s, kv.second.i}], len});
                g1.ktotal += len;
            }
            g1.seg_count = (int32_t)P->segs1.size() - g1.seg_begin;
            if (fresh)
                P->units.push_back({0, g.row, mip, std::vector<heff::KSeg>(P->segs1.begin() + g1.seg_begin,
                                                                           P->segs1.end())});
            P->blocks1.push_back(g1);
            P->segs2.push_back({c0, pad});
            g2.ktotal += pad;
        }
        g2.seg_count = (int32_t)P->segs2.size() - g2.seg_begin;
        P->units.push_back({2, t_rows, mj, std::vector<heff::KSeg>(P->segs2.begin() + g2.seg_begin, P->segs2.end())});
        P->blocks2.push_back(g2);
        t_rows += mj;
    }
    P->rows_lw = std::max<int64_t>(lw_rows, 1);
    P->rows_t = std::max<int64_t>(t_rows, 1);
}

// Workspace of the dense form in a precision (FP64: with its digit planes, unless they are left out); with p, its
// offsets too.
size_t dense_bytes(const heff_env_plan* P, int precision, heff_plan* p, bool digits = true) {
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    const bool tc = precision != HEFF_PREC_FP64;
    const size_t e = (size_t)(tc ? 4 : 8) * P->ld, kb = (size_t)(P->ld / KPAD) * sizeof(uint16_t);
    // the error flag comes first in every precision and form
    size_t off = 256, o_sp, o_lw, o_t;
    o_sp = off; off = al(off + e * P->rows_sp);
    o_lw = off; off = al(off + e * P->rows_lw);
    o_t = off;  off = al(off + e * P->rows_t);
    const size_t least = off;
    if (p) {
        p->off_xt = o_sp; p->off_lw = o_lw; p->off_t = o_t; p->off_rw = o_t; p->off_flags = 0;
        p->ws_min = off;
    }
    if (!tc && digits) {
        size_t o_ex, o_elw, o_et;
        o_ex = off;  off = al(off + kb * P->rows_sp);
        o_elw = off; off = al(off + kb * P->rows_lw);
        o_et = off;  off = al(off + kb * P->rows_t);
        heff_plan size_only;
        heff_plan* f = p ? p : &size_only;
        f->off_ex = o_ex; f->off_elw = o_elw; f->off_et = o_et; f->off_erw = o_et;
        const struct { int64_t rows; bool a; size_t src, codes; } ops[3] = {
            {P->rows_lw, false, o_lw, o_elw}, {P->rows_sp, true, o_sp, o_ex}, {P->rows_t, false, o_t, o_et}};
        for (int o = 0; o < 3; ++o) {
            f->fxo[o].ld = P->ld;
            f->fxo[o].rows = ops[o].rows;
            f->fxo[o].a_side = ops[o].a;
            f->fxo[o].off_src = ops[o].src;
            f->fxo[o].off_codes = ops[o].codes;
        }
        // (bits for FP64 outputs: a word per row and 32 columns, GEMM 1's, then GEMM 2's)
        int64_t words[2] = {0, 0};
        for (int g = 0; g < 2; ++g)
            for (const GemmTask& k : g == 0 ? P->blocks1 : P->blocks2)
                words[g] += (int64_t)k.m * ((k.n + 31) / 32);
        off = heff::plane_layout(f, off, std::max(words[0], words[1]), least);
    }
    if (p) p->ws_bytes = off;
    return off;
}

void free_plan(heff_env_plan* P) {
    if (P->plan) heff::plan_free_device(P->plan.get());
    P->plan.reset();
}

// The device tables of a precision, in the place of the plan's.  (At creation and when the precision is set: an
// update neither allocates nor synchronises, and can be captured.)
int build_plan(heff_env_plan* P, int precision) {
    int rc;
    try {
        std::unique_ptr<heff_plan> p(new heff_plan());
        const bool tc = precision != HEFF_PREC_FP64;
        p->env = true;
        p->opts.precision = precision;
        p->opts.io_dtype = HEFF_DTYPE_F64;
        p->opts.max_batch = 1;
        p->planes = tc ? 2 : 1;
        p->esize = tc ? 2 : 8;
        p->nelem_x = P->n_site;
        p->rows_x = P->rows_sp; p->ld_x = P->ld; p->rows_lw = P->rows_lw;
        p->rows_t = P->rows_t; p->ld_t = P->ld; p->rows_rw = 0;
        dense_bytes(P, precision, p.get());
        if (!tc)
            for (const auto& u : P->units) p->fxo[std::get<0>(u)].add(std::get<1>(u), std::get<2>(u), std::get<3>(u));
        p->pack = P->pack;
        p->mix = P->mix;
        p->terms = P->terms;
        int nsm = 148, dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            nsm = v;
        cudaGetLastError();
        const int tm = tc ? 128 : heff::FX_TILE_M, tn = tc ? 256 : heff::FX_TILE_N;
        auto cut = [&](const std::vector<GemmTask>& blocks, const std::vector<heff::KSeg>& segs, heff::GemmList& G,
                       bool first) {
            G.tm = tm;
            G.tn = tn;
            G.segs = segs;
            for (const GemmTask& k : blocks)
                for (int m0 = 0; m0 < k.m; m0 += tm)
                    for (int n0 = 0; n0 < k.n; n0 += tn) {
                        GemmTask t = k;
                        t.a_row += m0;
                        t.b_row += n0;
                        t.m = std::min(tm, k.m - m0);
                        t.n = std::min(tn, k.n - n0);
                        t.c_off += (int64_t)m0 * k.ldc + n0;
                        t.n_zero = n0 + tn >= k.n ? k.n_zero : 0;
                        G.tasks.push_back(t);
                    }
            G.owner.assign(G.tasks.size(), 0);
            G.task_flops.assign(G.tasks.size(), 0.0);
            G.task_useful.assign(G.tasks.size(), 0.0);
            heff::lpt_schedule(G, nsm, tc, first);
            if (!tc) G.count_fp64();
        };
        cut(P->blocks1, P->segs1, p->g1, true);
        cut(P->blocks2, P->segs2, p->g2, false);
        if ((rc = heff::plan_upload(p.get())) != HEFF_OK) {
            heff::plan_free_device(p.get());
            return rc;
        }
        free_plan(P);
        P->plan = std::move(p);
        P->precision = precision;
    } catch (const std::bad_alloc&) {
        return fail(HEFF_ERR_OOM, "out of host memory while planning the environment update");
    }
    return HEFF_OK;
}

}  // namespace

extern "C" int heff_env_plan_create(const heff_layout* env_old, const heff_layout* site, const heff_layout* W,
                                    const heff_layout* env_new, const double* W_host, int32_t side,
                                    heff_env_plan** out) try {
    heff::clear_error();
    if (!env_old || !site || !W || !env_new || !W_host || !out || (side != 0 && side != 1))
        return fail(HEFF_ERR_INVALID_ARG, "heff_env_plan_create: bad arguments");
    *out = nullptr;
    if (env_old->idx.size() != 3 || env_new->idx.size() != 3 || site->idx.size() != 3 || W->idx.size() != 4)
        return fail(HEFF_ERR_CHARGE_MISMATCH, "orders must be env 3, site 3, W 4");
    const heff::IndexDesc &sa = site->idx[0], &sp = site->idx[1], &sb = site->idx[2];
    if (sa.flow != 1 || sp.flow != 1 || sb.flow != -1)
        return fail(HEFF_ERR_CHARGE_MISMATCH, "site tensor flows must be (+1, +1, -1)");
    const heff::IndexDesc& bond_in = side == 0 ? sa : sb;    // bond of env_old
    const heff::IndexDesc& bond_out = side == 0 ? sb : sa;   // bond of env_new
    const heff::IndexDesc &wi = side == 0 ? W->idx[0] : W->idx[3];    // channels of env_old
    const heff::IndexDesc &wo = side == 0 ? W->idx[3] : W->idx[0];    // channels of env_new
    if (!same(env_old->idx[0], bond_in) || !same(env_old->idx[2], bond_in) || !same(env_old->idx[1], wi))
        return fail(HEFF_ERR_CHARGE_MISMATCH, "env_old must be (bond, channel, bond) on the site's %s bond",
                    side == 0 ? "left" : "right");
    if (!same(env_new->idx[0], bond_out) || !same(env_new->idx[2], bond_out) || !same(env_new->idx[1], wo))
        return fail(HEFF_ERR_CHARGE_MISMATCH, "env_new must be (bond, channel, bond) on the site's %s bond",
                    side == 0 ? "right" : "left");
    if (!same(W->idx[1], sp) || !same(W->idx[2], sp))
        return fail(HEFF_ERR_CHARGE_MISMATCH, "W physical indices must match the site tensor");
    heff_env_plan* P = new (std::nothrow) heff_env_plan();
    if (!P) return fail(HEFF_ERR_OOM, "out of host memory");
    P->side = side;
    try {
        const int d = sp.nsec, kw = W->idx[0].nsec, kv = W->idx[3].nsec;
        // W entries kept (nonzero in the host copy) as a dense (w, t, s, v) table, -1: dropped
        std::vector<int32_t> wtab((size_t)kw * d * d * kv, -1);
        for (size_t bk = 0; bk < W->offsets.size(); ++bk) {
            const int32_t* k = &W->keys[bk * 4];
            const int64_t o = W->offsets[bk];
            if (W_host[o] != 0.0) wtab[(((size_t)k[0] * d + k[1]) * d + k[2]) * kv + k[3]] = (int32_t)o;
        }
        auto widx = [&](int w, int t, int s, int v) -> int32_t {
            return wtab[(((size_t)w * d + t) * d + s) * kv + v];
        };
        // site blocks by key
        auto site_off = [&](int a, int s, int b) { return site->offset_of({a, s, b}); };
        P->n_env = env_old->nelem;
        P->n_site = site->nelem;
        build_dense(P, env_old, site, env_new, sa, sp, sb, d, side == 0 ? kw : kv,
                    [&](int u, int t, int s, int n) { return side == 0 ? widx(u, t, s, n) : widx(n, t, s, u); });
        P->ws_bytes = dense_bytes(P, HEFF_PREC_FP64, nullptr);
        P->ws_least = dense_bytes(P, HEFF_PREC_FP64, nullptr, false);
        P->dense = P->ws_bytes <= ENV_DENSE_MAX;
        if (!P->dense) {
        std::map<std::tuple<int, int, int, int>, int64_t> inter;   // intermediate blocks -> offset
        int64_t ioff = 0;
        if (side == 0) {
            // X(ia, w, s, jd) = L(ia, w, ib) A(ib, s, jd): needed when some W[w, t, s, v] != 0
            for (size_t bk = 0; bk < env_old->offsets.size(); ++bk) {
                const int ia = env_old->keys[bk * 3], w = env_old->keys[bk * 3 + 1], ib = env_old->keys[bk * 3 + 2];
                for (int s = 0; s < d; ++s) {
                    bool used = false;
                    for (int t = 0; t < d && !used; ++t)
                        for (int v = 0; v < kv && !used; ++v) used = widx(w, t, s, v) >= 0;
                    if (!used) continue;
                    int jd = sb.find(add(sa.q(ib), sp.q(s)));
                    if (jd < 0) continue;
                    int64_t so = site_off(ib, s, jd);
                    if (so < 0) continue;
                    const int mia = sa.dims[ia], mib = sa.dims[ib], mjd = sb.dims[jd];
                    inter[{ia, w, s, jd}] = ioff;
                    BProd p{};
                    p.a_off = env_old->offsets[bk]; p.a_rs = mib; p.a_cs = 1;
                    p.b_off = so; p.b_rs = mjd; p.b_cs = 1;
                    p.K = mib; p.c1 = -1; p.c2 = -1;
                    P->step1.add_block(ioff, mjd, mia, mjd, {p});
                    ioff += (int64_t)mia * mjd;
                }
            }
            // Lnew(jc, v, jd) = sum W[w,t,s,v] A(ia, t, jc)^T X(ia, w, s, jd)
            for (size_t bk = 0; bk < env_new->offsets.size(); ++bk) {
                const int jc = env_new->keys[bk * 3], v = env_new->keys[bk * 3 + 1], jd = env_new->keys[bk * 3 + 2];
                const int mjc = sb.dims[jc], mjd = sb.dims[jd];
                std::vector<BProd> ps;
                for (int t = 0; t < d; ++t) {
                    int ia = sa.find(add(sb.q(jc), sp.q(t), -1));
                    if (ia < 0) continue;
                    int64_t so = site_off(ia, t, jc);
                    if (so < 0) continue;
                    for (int w = 0; w < kw; ++w)
                        for (int s = 0; s < d; ++s) {
                            int32_t c = widx(w, t, s, v);
                            if (c < 0) continue;
                            auto it = inter.find({ia, w, s, jd});
                            if (it == inter.end()) continue;
                            BProd p{};
                            p.a_off = so; p.a_rs = 1; p.a_cs = mjc;          // A^T: (c, a) at a*mjc + c
                            p.b_off = it->second; p.b_rs = mjd; p.b_cs = 1;
                            p.K = sa.dims[ia]; p.c1 = c; p.c2 = -1;
                            ps.push_back(p);
                        }
                }
                P->step2.add_block(env_new->offsets[bk], mjd, mjc, mjd, ps);
            }
        } else {
            // Y(ja, v, id, s) = R(ja, v, jb) B(id, s, jb)^T
            for (size_t bk = 0; bk < env_old->offsets.size(); ++bk) {
                const int ja = env_old->keys[bk * 3], v = env_old->keys[bk * 3 + 1], jb = env_old->keys[bk * 3 + 2];
                for (int s = 0; s < d; ++s) {
                    bool used = false;
                    for (int t = 0; t < d && !used; ++t)
                        for (int w = 0; w < kw && !used; ++w) used = widx(w, t, s, v) >= 0;
                    if (!used) continue;
                    int id = sa.find(add(sb.q(jb), sp.q(s), -1));
                    if (id < 0) continue;
                    int64_t so = site_off(id, s, jb);
                    if (so < 0) continue;
                    const int mja = sb.dims[ja], mjb = sb.dims[jb], mid = sa.dims[id];
                    inter[{ja, v, id, s}] = ioff;
                    BProd p{};
                    p.a_off = env_old->offsets[bk]; p.a_rs = mjb; p.a_cs = 1;
                    p.b_off = so; p.b_rs = 1; p.b_cs = mjb;          // B^T: (b, d) at d*mjb + b
                    p.K = mjb; p.c1 = -1; p.c2 = -1;
                    P->step1.add_block(ioff, mid, mja, mid, {p});
                    ioff += (int64_t)mja * mid;
                }
            }
            // Rnew(ic, w, id) = sum W[w,t,s,v] B(ic, t, ja) Y(ja, v, id, s)
            for (size_t bk = 0; bk < env_new->offsets.size(); ++bk) {
                const int ic = env_new->keys[bk * 3], w = env_new->keys[bk * 3 + 1], id = env_new->keys[bk * 3 + 2];
                const int mic = sa.dims[ic], mid = sa.dims[id];
                std::vector<BProd> ps;
                for (int t = 0; t < d; ++t) {
                    int ja = sb.find(add(sa.q(ic), sp.q(t)));
                    if (ja < 0) continue;
                    int64_t so = site_off(ic, t, ja);
                    if (so < 0) continue;
                    const int mja = sb.dims[ja];
                    for (int v = 0; v < kv; ++v)
                        for (int s = 0; s < d; ++s) {
                            int32_t c = widx(w, t, s, v);
                            if (c < 0) continue;
                            auto it = inter.find({ja, v, id, s});
                            if (it == inter.end()) continue;
                            BProd p{};
                            p.a_off = so; p.a_rs = mja; p.a_cs = 1;
                            p.b_off = it->second; p.b_rs = mid; p.b_cs = 1;
                            p.K = mja; p.c1 = c; p.c2 = -1;
                            ps.push_back(p);
                        }
                }
                P->step2.add_block(env_new->offsets[bk], mid, mic, mid, ps);
            }
        }
        auto al = [](size_t v) { return (v + 255) / 256 * 256; };
        const size_t fp64_bytes = P->off_x + al((size_t)ioff * sizeof(double));
        P->off_env32 = P->off_x + al((size_t)ioff * sizeof(float));
        P->off_site32 = P->off_env32 + al((size_t)P->n_env * sizeof(float));
        const size_t tc_bytes = P->off_site32 + al((size_t)P->n_site * sizeof(float));
        P->ws_bytes = P->ws_least = std::max(fp64_bytes, tc_bytes);
        }
    } catch (const std::bad_alloc&) {
        delete P;
        return fail(HEFF_ERR_OOM, "out of host memory while planning the environment update");
    }
    int ndev = 0;
    P->device = cudaGetDeviceCount(&ndev) == cudaSuccess && ndev > 0;
    cudaGetLastError();
    if (P->device && P->dense) {
        if (const int rc = build_plan(P, P->precision)) {
            delete P;
            return rc;
        }
    } else if (P->device) {
        int rc;
        if ((rc = heff::blist_upload(P->step1)) || (rc = heff::blist_upload(P->step2))) {
            heff::blist_free(P->step1);
            heff::blist_free(P->step2);
            delete P;
            return rc;
        }
    }
    *out = P;
    return HEFF_OK;
} catch (const std::bad_alloc&) {
    return fail(HEFF_ERR_OOM, "out of host memory while checking the layouts of the environment update");
}

extern "C" int heff_env_workspace_size(const heff_env_plan* plan, size_t* bytes) {
    heff::clear_error();
    if (!plan || !bytes) return fail(HEFF_ERR_INVALID_ARG, "heff_env_workspace_size: null argument");
    *bytes = plan->precision == HEFF_PREC_FP64 ? plan->ws_bytes : plan->ws_least;
    return HEFF_OK;
}

extern "C" int heff_env_flops(const heff_env_plan* plan, double* flops) {
    heff::clear_error();
    if (!plan || !flops) return fail(HEFF_ERR_INVALID_ARG, "heff_env_flops: null argument");
    *flops = plan->flops;
    return HEFF_OK;
}

extern "C" int heff_env_update(heff_env_plan* plan, const double* env_old, const double* site, const double* W,
                               double* env_new, void* workspace, size_t workspace_bytes, void* stream) {
    heff::clear_error();
    if (!plan || !env_old || !site || !W || !env_new)
        return fail(HEFF_ERR_INVALID_ARG, "heff_env_update: null argument");
    if (!plan->device) return fail(HEFF_ERR_UNSUPPORTED, "env plan was created without a CUDA device");
    if (!workspace || workspace_bytes < plan->ws_least || reinterpret_cast<uintptr_t>(workspace) % 256)
        return fail(HEFF_ERR_WORKSPACE, "environment workspace of %zu bytes, needs %zu (256-byte aligned)",
                    workspace_bytes, plan->ws_least);
    char* ws = static_cast<char*>(workspace);
    int rc = heff::reset_flag(ws, stream);
    if (rc) return rc;
    if (plan->dense) {
        heff_plan* p = plan->plan.get();
        const void* xs[1] = {site};
        void* ys[1] = {env_new};
        // the mix tiles read env_old as L with W as W1, and (side 1) the site tensor as R
        const bool planes = heff::has_planes(p, workspace_bytes);
        if ((rc = heff::launch_mix(p, env_old, W, W, site, ws, planes, stream))) return rc;
        if ((rc = heff::launch_pack_batch(p, xs, 1, ws, planes, stream))) return rc;
        if (planes)
            for (int array : {1, 0})
                if ((rc = heff::launch_digits(p, array, ws, 1, stream))) return rc;
        if ((rc = heff::launch_gemm(p, 1, ws, ys, 1, planes, stream))) return rc;
        return heff::launch_gemm(p, 2, ws, ys, 1, planes, stream);
    }
    int* err = reinterpret_cast<int*>(ws);
    if (plan->precision == HEFF_PREC_FP64) {
        double* X = reinterpret_cast<double*>(ws + plan->off_x);
        if ((rc = heff::launch_bgemm(plan->step1, env_old, site, X, nullptr, nullptr, 1.0, stream, err))) return rc;
        return heff::launch_bgemm(plan->step2, site, X, env_new, W, nullptr, 1.0, stream, err);
    }
    float* X = reinterpret_cast<float*>(ws + plan->off_x);
    float* E32 = reinterpret_cast<float*>(ws + plan->off_env32);
    float* S32 = reinterpret_cast<float*>(ws + plan->off_site32);
    if ((rc = heff::launch_convert_f64_f32(env_old, E32, plan->n_env, stream))) return rc;
    if ((rc = heff::launch_convert_f64_f32(site, S32, plan->n_site, stream))) return rc;
    if ((rc = heff::launch_bgemm_tc(plan->step1, E32, S32, X, false, nullptr, nullptr, 1.0, stream, nullptr, err)))
        return rc;
    return heff::launch_bgemm_tc(plan->step2, S32, X, env_new, true, W, nullptr, 1.0, stream, nullptr, err);
}

extern "C" int heff_env_plan_set_precision(heff_env_plan* plan, int32_t precision) try {
    heff::clear_error();
    if (!plan) return fail(HEFF_ERR_INVALID_ARG, "heff_env_plan_set_precision: null plan");
    if (precision != HEFF_PREC_FP64 && precision != HEFF_PREC_BF16X3)
        return fail(HEFF_ERR_UNSUPPORTED, "environment updates run in HEFF_PREC_FP64 or HEFF_PREC_BF16X3");
    if (precision == plan->precision) return HEFF_OK;
    if (plan->dense) {
        if (plan->device) return build_plan(plan, precision);
        plan->precision = precision;
        return HEFF_OK;
    }
    const bool fx = precision == HEFF_PREC_FP64;
    heff::blist_free(plan->step1);
    heff::blist_free(plan->step2);
    plan->step1.retile(fx ? heff::FX_TILE_M : 128, fx ? heff::FX_TILE_N : 128);
    plan->step2.retile(fx ? heff::FX_TILE_M : 128, fx ? heff::FX_TILE_N : 128);
    plan->precision = precision;
    if (plan->device) {
        int rc;
        if ((rc = heff::blist_upload(plan->step1)) || (rc = heff::blist_upload(plan->step2))) {
            plan->device = false;
            return rc;
        }
    }
    return HEFF_OK;
} catch (const std::bad_alloc&) {      // (the lists are not whole)
    plan->device = false;
    return fail(HEFF_ERR_OOM, "out of host memory while planning the environment update");
}

extern "C" int heff_env_status(const heff_env_plan* plan, void* workspace, size_t workspace_bytes, void* stream) {
    heff::clear_error();
    if (!plan || !workspace) return fail(HEFF_ERR_INVALID_ARG, "heff_env_status: null argument");
    if (workspace_bytes < heff::FLAG_BYTES) return fail(HEFF_ERR_WORKSPACE, "heff_env_status: workspace too small");
    return heff::read_flag(workspace, "the environment update", stream);
}

extern "C" void heff_env_plan_destroy(heff_env_plan* plan) {
    if (!plan) return;
    free_plan(plan);
    heff::blist_free(plan->step1);
    heff::blist_free(plan->step2);
    delete plan;
}

// ---------------------------------------------------------------- two-site tensor
// x[a, s1, s2, b] = sum_c A[a, s1, c] B[c, s2, b] (Fig. 1d: the two MPS sites joined over
// their shared bond, the starting vector of a bond's eigensolve).  One block product per
// charge-matched (A block, B block) pair, summed per x block; x blocks without a matching
// pair are written as zeros.
struct heff_two_site {
    BList prods;
    bool uploaded = false;
    int64_t nx = 0;
};

namespace {

// A bounded wait of the products expired: x is not the product; it becomes NaN and the flag zero again.
// (One block; a flag that the host can read would cost 330 us of pinning per plan, and a plan lives for one
// bond.)
__global__ void __launch_bounds__(1024) two_site_check_kernel(int* __restrict__ err, double* __restrict__ x, int64_t n) {
    const int e = *err;
    __syncthreads();
    if (e == 0) return;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) x[i] = nan("");
    if (threadIdx.x == 0) *err = 0;
}

}  // namespace

extern "C" int heff_two_site_create(const heff_layout* A, const heff_layout* B, const heff_layout* x,
                                    heff_two_site** out) try {
    heff::clear_error();
    if (!A || !B || !x || !out) return fail(HEFF_ERR_INVALID_ARG, "heff_two_site_create: null argument");
    *out = nullptr;
    if (A->idx.size() != 3 || B->idx.size() != 3 || x->idx.size() != 4)
        return fail(HEFF_ERR_CHARGE_MISMATCH, "orders must be A 3, B 3, x 4");
    const heff::IndexDesc &aa = A->idx[0], &ap = A->idx[1], &ac = A->idx[2];
    const heff::IndexDesc &bc = B->idx[0], &bp = B->idx[1], &bb = B->idx[2];
    if (aa.flow != 1 || ap.flow != 1 || ac.flow != -1 || bc.flow != 1 || bp.flow != 1 || bb.flow != -1)
        return fail(HEFF_ERR_CHARGE_MISMATCH, "A and B flows must be (+1, +1, -1)");
    if (!same(ac, bc) || !same(aa, x->idx[0]) || !same(ap, x->idx[1]) || !same(bp, x->idx[2]) ||
        !same(bb, x->idx[3]))
        return fail(HEFF_ERR_CHARGE_MISMATCH, "A (a, s1, c), B (c, s2, b) and x (a, s1, s2, b) indices disagree");
    heff_two_site* P = new (std::nothrow) heff_two_site();
    if (!P) return fail(HEFF_ERR_OOM, "out of host memory");
    P->nx = x->nelem;
    try {
        std::map<std::pair<int, int>, std::vector<std::pair<int, int64_t>>> a_by;   // (a, s1) -> (c, offset)
        for (size_t k = 0; k < A->offsets.size(); ++k)
            a_by[{A->keys[k * 3], A->keys[k * 3 + 1]}].push_back({A->keys[k * 3 + 2], A->offsets[k]});
        for (size_t k = 0; k < x->offsets.size(); ++k) {
            const int a = x->keys[k * 4], s1 = x->keys[k * 4 + 1], s2 = x->keys[k * 4 + 2], b = x->keys[k * 4 + 3];
            const int ma = aa.dims[a], mb = bb.dims[b];
            std::vector<BProd> ps;
            auto it = a_by.find({a, s1});
            if (it != a_by.end())
                for (auto& co : it->second) {
                    const int64_t boff = B->offset_of({co.first, s2, b});
                    if (boff < 0) continue;
                    const int mc = ac.dims[co.first];
                    BProd p{};
                    p.a_off = co.second; p.a_rs = mc; p.a_cs = 1;
                    p.b_off = boff; p.b_rs = mb; p.b_cs = 1;
                    p.K = mc; p.c1 = -1; p.c2 = -1;
                    ps.push_back(p);
                }
            P->prods.add_block(x->offsets[k], mb, ma, mb, ps);
        }
    } catch (const std::bad_alloc&) {
        delete P;
        return fail(HEFF_ERR_OOM, "out of host memory while planning the two-site tensor");
    }
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) == cudaSuccess && ndev > 0) {
        int rc = heff::blist_upload(P->prods);
        if (rc) {
            heff::blist_free(P->prods);
            delete P;
            return rc;
        }
        P->uploaded = true;
    } else {
        cudaGetLastError();
    }
    *out = P;
    return HEFF_OK;
} catch (const std::bad_alloc&) {
    return fail(HEFF_ERR_OOM, "out of host memory while checking the layouts of the two-site tensor");
}

extern "C" int heff_two_site_apply(heff_two_site* P, const double* A, const double* B, double* x, void* stream) {
    heff::clear_error();
    if (!P || !A || !B || !x) return fail(HEFF_ERR_INVALID_ARG, "heff_two_site_apply: null argument");
    if (!P->uploaded) return fail(HEFF_ERR_UNSUPPORTED, "two-site plan was created without a CUDA device");
    const int rc = heff::launch_bgemm(P->prods, A, B, x, nullptr, nullptr, 1.0, stream, P->prods.d_err);
    if (rc || !P->prods.d_err) return rc;
    two_site_check_kernel<<<1, 1024, 0, static_cast<cudaStream_t>(stream)>>>(P->prods.d_err, x, P->nx);
    heff::count_launches(1);
    if (cudaGetLastError() != cudaSuccess) return fail(HEFF_ERR_CUDA, "heff_two_site_apply: launch failed");
    return HEFF_OK;
}

extern "C" void heff_two_site_destroy(heff_two_site* P) {
    if (!P) return;
    heff::blist_free(P->prods);
    delete P;
}
