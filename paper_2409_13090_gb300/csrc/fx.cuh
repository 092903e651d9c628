// FP64 values as 62-bit whole numbers in eight signed digits of base 256, and sums
// of digit products back to FP64: the arithmetic of the FP64 products on the tensor
// cores (split_gemm.cuh: tcgen05 tiles; sweep64.cuh: warp-level MMAs of the solve).
//
// x with |x| < 2^E is the whole number X = trunc(x 2^(62 - E)), |X| < 2^62,
//   X = sum_{i = 1..8} d_i 256^(8 - i),  d_i in [-128, 127],  |d_1| <= 65.
// A sum of products is
//   sum_k x_k y_k = 2^(E_x + E_y) sum_{g = 1..8} 2^(-4 - 8 g) G_g,
//   G_g = sum_k sum_{i + j = g + 1} d_i(x_k) d_j(y_k),
// with the groups g > 8 left out: seven products of at most 2^14 in units of 2^-76, and less
// after those, so below 2^-59.1 of 2^(E_x + E_y) per term (random operands: 2^-63 on average). The
// truncation leaves out less than 2^-62 of 2^E of each operand: all in all a term is below
// 2^-58.7 of 2^(E_x + E_y) off. Over at most
// 128 terms |G_g| <= 114944 * 128 < 2^24: FP32 accumulation of the FP16 digit
// products is exact.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace sc {
namespace fx {

constexpr int S = 8;  // digits
constexpr int32_t kBadExp = 1 << 20; // exponent of a row or column that holds an infinity or a NaN

// X + 0x8080808080808080 for a finite |x| < 2^E: its bytes, the highest first, are the
// digits d_1 .. d_8 plus 128.
__device__ __forceinline__ uint64_t split_bytes(double x, int E) {
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
    const int ex = (int)(hi >> 20) & 0x7ff;
    // |x| = M 2^(max(ex, 1) - 1085), M < 2^63; X = M >> n (towards zero)
    const uint32_t mh = (hi & 0xfffffu) | (ex ? 0x100000u : 0u);
    const uint64_t M = ((uint64_t)mh << 42) | ((uint64_t)lo << 10);
    const int n = E + 1023 - max(ex, 1);  // >= 1
    const uint64_t X = n < 64 ? M >> n : 0;
    const uint64_t s = (uint64_t)((int64_t)(int32_t)hi >> 31);  // all ones for a negative x
    return (X ^ s) + (0x8080808080808080ull - s);
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
// the accumulator, in units of 2^(e - 68), less 1
__device__ __forceinline__ void acc_sub_one(Acc96 &a, int e) {
    const int s = 68 - e;  // 1 is 2^s units
    if (s < 0 || s > 94) return;
    if (s >= 32) {
        a.t -= (int64_t)1 << (s - 32);
    } else {
        const uint32_t r = a.r;
        a.r = r - (1u << s);
        a.t -= a.r > r ? 1 : 0;
    }
}
// the accumulator times 2^(e - 68) when that is outside FP64's normal range
static __device__ __noinline__ double acc_value_slow(int64_t t, uint32_t r, int e) {
    return scalbn(scalbn((double)t, 32) + (double)r, e - 68);
}
// the accumulator times 2^(e - 68), rounded to FP64, in integer operations without
// branches (a conversion of a 64-bit whole number and a scaling take the FP64 pipe 64
// clocks each)
__device__ __forceinline__ double acc_value(const Acc96 &a, int e) {
    // magnitude (one's complement: off by at most the last of the 96 bits)
    const uint32_t s = (uint32_t)(a.t >> 63);
    uint32_t w2 = (uint32_t)(a.t >> 32) ^ s, w1 = (uint32_t)a.t ^ s, w0 = a.r ^ s;
    int sc = e - 68 + 32 + 62;
    // whole words of leading zeros (up to bit 62 of the upper two words)
#pragma unroll
    for (int i = 0; i < 2; i++) {
        const bool up = w2 == 0 && (w1 >> 31) == 0;
        w2 = up ? w1 : w2;
        w1 = up ? w0 : w1;
        w0 = up ? 0u : w0;
        sc -= up ? 32 : 0;
    }
    const bool zero = (w2 | w1) == 0;
    // w2 == 0 here means that bit 31 of w1 is set
    const int z = w2 ? __clz((int)w2) - 1 : 31;
    uint32_t hi = __funnelshift_l(w1, w2, z), lo = __funnelshift_l(w0, w1, z);
    sc -= z;
    // to nearest at bit 10: 53 bits from bit 62
    const uint32_t l2 = lo + 0x200u;
    hi += l2 < lo ? 1u : 0u;
    const uint32_t mh = hi >> 10, ml = __funnelshift_r(l2, hi, 10);  // 2^52 <= (mh, ml) <= 2^53
    if (zero) return 0.0;
    if ((unsigned)(sc + 1021) > 2043u) return acc_value_slow(a.t, a.r, e);
    return __hiloint2double((int)((mh + ((uint32_t)(sc + 1022) << 20)) | (s & 0x80000000u)), (int)ml);
}

// |x| 2^e as FP32, truncated (infinity from its range on)
__device__ __forceinline__ float size_of(double x, int e) {
    const int hi = __double2hiint(x), ex = (hi >> 20) & 0x7ff, f = ex + e - 896;
    if (ex == 0x7ff || f >= 255) return __int_as_float(0x7f800000);
    return f <= 0 ? 0.f : __int_as_float(f << 23 | (hi & 0xfffff) << 3);
}

}  // namespace fx
}  // namespace sc
