// Block-product engine: lists of strided dense block products summed into output tiles (run by
// fx_gemm.cu in FP64 accuracy, or by blockops_tc.cu in BF16x3), and block dot products.  Used by the environment update,
// the two-site tensor, the SVD and the Rayleigh-quotient gradients (the block-pair contractions of Algorithm 2 with charge-matched blocks, each
// product a small dense GEMM, Section IV "list" algorithm).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>

#include "convert.cuh"
#include "internal.h"

namespace heff {

void BList::add_block(int64_t c_off, int32_t ldc, int32_t m, int32_t n, const std::vector<BProd>& ps) {
    blocks.push_back(Block{c_off, ldc, m, n, (int32_t)block_prods.size(), (int32_t)ps.size()});
    block_prods.insert(block_prods.end(), ps.begin(), ps.end());
    const bool fx = tile_n == FX_TILE_N;
    std::vector<std::pair<View, View>> v(ps.size());
    int32_t steps = 0;
    for (size_t i = 0; fx && i < ps.size(); ++i) {
        const BProd& p = ps[i];
        v[i] = {view(0, p.a_off, p.a_rs, p.a_cs, m, p.K), view(1, p.b_off, p.b_cs, p.b_rs, n, p.K)};
        steps += (p.K + 15) / 16;
    }
    for (int r0 = 0; r0 < m; r0 += tile_m)
        for (int c0 = 0; c0 < n; c0 += tile_n) {
            BTile t{};
            t.c_off = c_off + (int64_t)r0 * ldc + c0;
            t.ldc = ldc;
            t.m = m - r0 < tile_m ? m - r0 : tile_m;
            t.n = n - c0 < tile_n ? n - c0 : tile_n;
            t.prod_begin = (int32_t)prods.size();
            t.prod_count = (int32_t)ps.size();
            t.steps = steps;
            t.fp64_at = nfp64;
            if (fx) nfp64 += t.m * ((t.n + 31) / 32);
            for (size_t i = 0; i < ps.size(); ++i) {
                const BProd& p = ps[i];
                BProd q = p;
                q.ea = v[i].first.code + r0;
                q.eb = v[i].second.code + c0;
                q.za = v[i].first.word + r0;
                q.zb = v[i].second.word + c0;
                q.na = m;
                q.nb = n;
                q.a_off += (int64_t)r0 * p.a_rs;
                q.b_off += (int64_t)c0 * p.b_cs;
                prods.push_back(q);
                flops += 2.0 * t.m * t.n * p.K;
            }
            tiles.push_back(t);
        }
}

BList::View BList::view(int which, int64_t off, int32_t rs, int32_t ks, int32_t n, int32_t K) {
    auto ins = views.insert({{which, off, rs, ks, n, K}, {ncodes, nwords}});
    if (ins.second) {
        for (int32_t r = 0; r < n; r += 32)
            rows.push_back({off + (int64_t)r * rs, rs, ks, n - r < 32 ? n - r : 32, K, ncodes + r, which, nwords + r, n});
        ncodes += n;
        nwords += (K + 31) / 32 * n;
    }
    return ins.first->second;
}

void BList::retile(int tm, int tn) {
    std::vector<Block> bl;
    std::vector<BProd> bp;
    bl.swap(blocks);
    bp.swap(block_prods);
    tiles.clear();
    prods.clear();
    rows.clear();
    views.clear();
    ncodes = nwords = nfp64 = 0;
    flops = 0;
    tile_m = tm;
    tile_n = tn;
    for (const Block& k : bl)
        add_block(k.c_off, k.ldc, k.m, k.n,
                  std::vector<BProd>(bp.begin() + k.prod_begin, bp.begin() + k.prod_begin + k.prod_count));
}

int blist_upload(BList& b) try {
    b.d_tables = nullptr;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&b.num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return fail(HEFF_ERR_CUDA, "device query failed");
    // the longest tiles first
    if (b.tile_n == FX_TILE_N)
        std::stable_sort(b.tiles.begin(), b.tiles.end(), [](const BTile& x, const BTile& y) {
            return (int64_t)x.steps * (x.n + 32) > (int64_t)y.steps * (y.n + 32);
        });
    // one allocation for the tables, an error flag (zero), the codes, words, sums and bits
    auto al = [](size_t v) { return (v + 255) / 256 * 256; };
    const size_t nt = b.tiles.size() * sizeof(BTile), np = b.prods.size() * sizeof(BProd), nr = b.rows.size() * sizeof(FxRows);
    const size_t op = al(nt), orow = op + al(np), oe = orow + al(nr), oc = oe + 256;
    const size_t ow = oc + al(b.ncodes * sizeof(uint16_t)), os = ow + al(b.nwords * sizeof(uint32_t));
    const size_t of = os + al(b.ncodes * sizeof(float));
    if (nt + np + nr == 0) return HEFF_OK;
    std::vector<char> host(oc, 0);
    if (nt) std::memcpy(host.data(), b.tiles.data(), nt);
    if (np) std::memcpy(host.data() + op, b.prods.data(), np);
    if (nr) std::memcpy(host.data() + orow, b.rows.data(), nr);
    char* d = nullptr;
    if (cudaMalloc((void**)&d, of + b.nfp64 * sizeof(uint32_t)) != cudaSuccess ||
        cudaMemcpy(d, host.data(), oc, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(d);
        return fail(HEFF_ERR_CUDA, "block list upload failed");
    }
    b.d_tables = d;
    b.d_tiles = reinterpret_cast<BTile*>(d);
    b.d_prods = reinterpret_cast<BProd*>(d + op);
    b.d_rows = reinterpret_cast<FxRows*>(d + orow);
    b.d_err = reinterpret_cast<int*>(d + oe);
    b.d_codes = reinterpret_cast<uint16_t*>(d + oc);
    b.d_words = reinterpret_cast<uint32_t*>(d + ow);
    b.d_sums = reinterpret_cast<float*>(d + os);
    b.d_fp64 = reinterpret_cast<uint32_t*>(d + of);
    return HEFF_OK;
} catch (const std::bad_alloc&) {      // (the callers are C entries)
    return fail(HEFF_ERR_OOM, "out of host memory for the block products' tables");
}

void blist_free(BList& b) {
    cudaFree(b.d_tables);
    b.d_tables = nullptr;
    b.d_tiles = nullptr;
    b.d_prods = nullptr;
    b.d_rows = nullptr;
    b.d_err = nullptr;
    b.d_codes = nullptr;
    b.d_words = nullptr;
    b.d_sums = nullptr;
    b.d_fp64 = nullptr;
}

namespace {

// one CTA per dot: partial[d] = <X[x_off..], Y[y_off..]>, accumulated in the element type
// (FP32 vectors come from the tensor-core products, whose values carry ~1e-5 anyway).  Bound by the
// latency of its loads: four of each vector are issued before the first product.
template <typename T>
__global__ void __launch_bounds__(256) block_dot_kernel(const BDot* __restrict__ dots, const T* __restrict__ X,
                                                        const T* __restrict__ Y, double* __restrict__ partial) {
    __shared__ T sh[8];
    const BDot d = dots[blockIdx.x];
    const T* x = X + d.x_off;
    const T* y = Y + d.y_off;
    T a4[4] = {0, 0, 0, 0};
    int64_t i = threadIdx.x;
    for (; i + 3 * 256 < d.len; i += 4 * 256) {
        T u[4], v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            u[j] = x[i + j * 256];
            v[j] = y[i + j * 256];
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) a4[j] = fma(u[j], v[j], a4[j]);
    }
    for (; i < d.len; i += 256) a4[0] = fma(x[i], y[i], a4[0]);
    T a = (a4[0] + a4[1]) + (a4[2] + a4[3]);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        T s = 0;
        for (int w = 0; w < 8; ++w) s += sh[w];
        if constexpr (std::is_same<T, double>::value) partial[blockIdx.x] = s;
        else partial[blockIdx.x] = f32_to_f64(s);
    }
}

// out[j] = scale * sum of partial[d] for d in [off[j], off[j+1]) (dots sorted by output), L lanes per output: each
// sums every L-th partial, then the lanes in a fixed tree (deterministic).
template <int L>
__global__ void __launch_bounds__(256) gather_dots_kernel(const int32_t* __restrict__ off,
                                                          const double* __restrict__ partial,
                                                          double* __restrict__ out, int nout, double scale,
                                                          int accumulate) {
    const int lane = threadIdx.x % L, j = blockIdx.x * (256 / L) + threadIdx.x / L;
    double s = 0.0;
    if (j < nout)
        for (int d = off[j] + lane; d < off[j + 1]; d += L) s += partial[d];
    for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (j < nout && lane == 0) out[j] = accumulate ? out[j] + scale * s : scale * s;
}

}  // namespace

template <typename T>
static int block_dots_t(const BDot* d_dots, int ndots, const int32_t* d_off, const T* X, const T* Y, double* out,
                        int nout, double* scratch, double scale, void* stream, bool accumulate) {
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (ndots > 0) {
        block_dot_kernel<T><<<ndots, 256, 0, st>>>(d_dots, X, Y, scratch);
        count_launches(1);
    }
    // lanes per output by the partials of an average one (us for 1, 4, 32 lanes: 82944 outputs of 2: 4.1, 6.2, 35;
    // 12544 of 64: 12, 6.2, 10; one of 2000: 92, 27, 6.2)
    auto gather = [&](auto kernel, int lanes) {
        kernel<<<(nout + 256 / lanes - 1) / (256 / lanes), 256, 0, st>>>(d_off, scratch, out, nout, scale, accumulate ? 1 : 0);
    };
    if (ndots <= 8 * (int64_t)nout) gather(gather_dots_kernel<1>, 1);
    else if (ndots <= 128 * (int64_t)nout) gather(gather_dots_kernel<4>, 4);
    else gather(gather_dots_kernel<32>, 32);
    count_launches(1);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(HEFF_ERR_CUDA, "block dots launch: %s", cudaGetErrorString(e));
    return HEFF_OK;
}

int launch_block_dots(const BDot* d_dots, int ndots, const int32_t* d_off, const double* X, const double* Y,
                      double* out, int nout, double* scratch, double scale, void* stream, bool accumulate) {
    return block_dots_t(d_dots, ndots, d_off, X, Y, out, nout, scratch, scale, stream, accumulate);
}

int launch_block_dots_f32(const BDot* d_dots, int ndots, const int32_t* d_off, const float* X, const float* Y,
                          double* out, int nout, double* scratch, double scale, void* stream, bool accumulate) {
    return block_dots_t(d_dots, ndots, d_off, X, Y, out, nout, scratch, scale, stream, accumulate);
}

}  // namespace heff
