// FP64 values as 64-bit fixed-point numbers of eight signed 8-bit digits, and back: the
// arithmetic of the FP64 products on the FP16 tensor pipe (fx_gemm.cu, fx_planes.cu).
//
// A row of an operand shares one exponent code E (|v| < 2^(E - 1022) for every v of the row),
// and v is held as q = trunc(v 2^(1084 - E)), |q| < 2^62, written in balanced base 256:
// q = sum_s d_s 2^(56 - 8 s), d_0 in [-64, 64], the others in [-128, 127].  A digit is an
// integer that FP16 holds exactly, a product of two digits is at most 2^14, and sums of them
// stay exact in FP32 up to 2^24.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace heff {
namespace fx {

#define FX_HD __host__ __device__ __forceinline__

// Exponent code of a value given by its two words: 0 for a zero, else the biased exponent (at
// least 1: a subnormal counts as 1); 0x7ff for infinities and NaNs.
FX_HD int exp_code(uint32_t hi, uint32_t lo) {
    const int e = (int)((hi >> 20) & 0x7ffu);
    return e ? e : (((hi & 0x7fffffffu) | lo) ? 1 : 0);
}

// Codes that the fixed-point path takes: zero rows, and rows whose largest magnitude lies in
// [2^-400, 2^400).  In that range the scaled result of a product is a normal number and what a
// row's scale drops (below 2^-62 of its largest element) includes every subnormal.  Any other
// row (infinities and NaNs among them) is computed in FP64.
constexpr int E_MIN = 623, E_MAX = 1422;
FX_HD bool exp_plain(int e) { return e == 0 || (e >= E_MIN && e <= E_MAX); }
// scale of a zero row: everything shifts out
constexpr int E_ZERO = 1023;

// The digits of one value for the row scale E, each offset by 128: byte 7 (the top of the
// returned word) is digit 0.
FX_HD uint64_t to_fixed(uint32_t hi, uint32_t lo, int E) {
    const int e = (int)((hi >> 20) & 0x7ffu);
    const int s = E - e < 63 ? E - e : 63;
    const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 9;
    const uint64_t q = m >> s;                                  // e = 0 shifts out: E >= E_MIN
    const uint64_t g = (uint64_t)((int64_t)(int32_t)hi >> 31);  // all ones for a negative value
    return (q ^ g) - g + 0x8080808080808080ull;
}

// The double nearest to X 2^p, X the signed 96-bit number (w2, w1, w0).  p keeps the result
// normal.
FX_HD double from_fixed(uint32_t w2, uint32_t w1, uint32_t w0, int p) {
    const uint32_t neg = (uint32_t)((int32_t)w2 >> 31);
    // two's complement magnitude
    uint64_t low = ((uint64_t)(w1 ^ neg) << 32) | (w0 ^ neg);
    w2 ^= neg;
    const uint64_t lown = low + (neg & 1u);
    w2 += lown < low ? 1u : 0u;
    w1 = (uint32_t)(lown >> 32);
    w0 = (uint32_t)lown;
    // the top word nonzero
    if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; p -= 32; }
    if (w2 == 0) { w2 = w1; w1 = 0; p -= 32; }
    if (w2 == 0) return 0.0;
#ifdef __CUDA_ARCH__
    const int c = __clz((int)w2);
    const uint32_t h = __funnelshift_l(w1, w2, c), m = __funnelshift_l(w0, w1, c);
    const uint64_t t = ((uint64_t)h << 32) | m;
#else
    const int c = __builtin_clz(w2);
    uint64_t t = ((uint64_t)w2 << 32) | w1;
    t = c ? (t << c) | (w0 >> (32 - c)) : t;
#endif
    // X 2^p ~ t 2^(32 - c + p): 53 bits, rounded on the next one
    const uint64_t mant = (t >> 11) + ((t >> 10) & 1u);
    const uint64_t bits = ((uint64_t)(43 - c + p + 1074) << 52) + mant + ((uint64_t)(neg & 1u) << 63);
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)bits);
#else
    double d;
    __builtin_memcpy(&d, &bits, 8);
    return d;
#endif
}

}  // namespace fx
}  // namespace heff
