// FP64 values as 62-bit whole numbers in eight signed digits of base 256, and sums
// of digit products back to FP64: the arithmetic of the FP64 products on the tensor
// cores (split_gemm.cuh: tcgen05 tiles; sweep64.cuh: warp-level MMAs of the solve).
//
// x with |x| < 2^E is the whole number X = round(x 2^(62 - E)), |X| <= 2^62,
//   X = sum_{i = 1..8} d_i 256^(8 - i),  d_i in [-128, 127],  |d_1| <= 65.
// A sum of products is
//   sum_k x_k y_k = 2^(E_x + E_y) sum_{g = 1..8} 2^(-4 - 8 g) G_g,
//   G_g = sum_k sum_{i + j = g + 1} d_i(x_k) d_j(y_k),
// with the groups g > 8 left out (below 2^-64 of 2^(E_x + E_y) per term). Over at most
// 128 terms |G_g| <= 114944 * 128 < 2^24: FP32 accumulation of the FP16 digit
// products is exact.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace sc {
namespace fx {

constexpr int S = 8;  // digits
constexpr int32_t kBadExp = 1 << 20; // exponent of a row or column that holds an infinity or a NaN

// X = round(x 2^(62 - E)) + 0x8080808080808080 for a finite |x| < 2^E: its bytes,
// the highest first, are the digits d_1 .. d_8 plus 128.
__device__ __forceinline__ uint64_t split_bytes(double x, int E) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const int ex = (int)(b >> 52) & 0x7ff;
    uint64_t m = b & 0xFFFFFFFFFFFFFull;
    if (ex) m |= 1ull << 52;
    // x = m 2^(max(ex, 1) - 1075)
    const int sh = max(ex, 1) - 1075 + 62 - E;  // <= 10
    uint64_t X;
    if (sh >= 0) X = m << sh;
    else if (sh > -55) X = ((m >> (-sh - 1)) + 1) >> 1;  // to nearest
    else X = 0;
    if (b >> 63) X = 0 - X;
    return X + 0x8080808080808080ull;
}

// 96-bit accumulator (t: upper 64 bits, r: lower 32) of an entry, in units of 2^-68
struct Acc96 {
    int64_t t;
    uint32_t r;
};
__device__ __forceinline__ int as_int(uint32_t v) { return __float2int_rn(__uint_as_float(v)); }
// groups 1..4 of an entry: |g_1| <= 2^20, |g_2| <= 2^22, |g_3|, |g_4| <= 2^23, so
// both pairs fit in 32 bits
__device__ __forceinline__ void acc_add_high(Acc96 &a, uint32_t g1, uint32_t g2, uint32_t g3, uint32_t g4) {
    const int p12 = as_int(g1) * 256 + as_int(g2), p34 = as_int(g3) * 256 + as_int(g4);
    a.t += (int64_t)p12 * 65536 + p34;
}
// groups 5..8
__device__ __forceinline__ void acc_add_low(Acc96 &a, uint32_t g5, uint32_t g6, uint32_t g7, uint32_t g8) {
    const int64_t L =
        (int64_t)as_int(g5) * (1 << 24) + ((int64_t)as_int(g6) * (1 << 16) + ((int64_t)as_int(g7) * 256 + as_int(g8)));
    const uint32_t lo = (uint32_t)L, r = a.r + lo;
    a.t += (L >> 32) + (r < lo ? 1 : 0);
    a.r = r;
}
// the accumulator times 2^(e - 68), rounded to FP64, in integer operations (the
// conversion of a 64-bit whole number and a scaling would go through the FP64 pipe)
__device__ __forceinline__ double acc_value(const Acc96 &a, int e) {
    // magnitude (m, r), then normalised: the highest bit of m at bit 62
    const bool neg = a.t < 0;
    uint64_t m = neg ? ~(uint64_t)a.t : (uint64_t)a.t;
    uint32_t r = neg ? 0u - a.r : a.r;
    if (neg && r == 0) m++;
    int sc = e - 68 + 32;
    if ((m >> 31) == 0) {  // 96 bits down to the lower 64
        m = (m << 32) | r;
        r = 0;
        sc -= 32;
    }
    const int z = __clzll((long long)m) - 1;  // m < 2^63; at most 31 here unless r is 0
    if (z == 63) return 0.0;
    m = (m << z) | (z < 32 ? (uint64_t)(r >> 1) >> (31 - z) : 0ull);
    if (z < 32 && (r << z)) m |= 1;  // whatever is below the last bit
    // round to nearest even at bit 10: 53 bits from bit 62
    m += 0x1ff + ((m >> 10) & 1);
    m >>= 10;  // 2^52 <= m <= 2^53
    sc += 62 - z;  // exponent of the highest bit
    if (sc >= -1021 && sc <= 1022)
        return __longlong_as_double((long long)((((uint64_t)(neg ? 2048 : 0) + (uint64_t)(sc + 1022)) << 52) + m));
    const double d = scalbn((double)m, sc - 52);  // outside the normal range
    return neg ? -d : d;
}

}  // namespace fx
}  // namespace sc
