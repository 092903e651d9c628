// Triangular solve sweeps with an FP64 factor (included by solve.cu).
//
// The FP64 pipe of this chip takes 64 clocks for a warp's multiply-add, alone or in a chain;
// an FP16 MMA of 2048 multiply-adds takes 8. So the products of a sweep unit
// (64 rows of L, or the inverse of a diagonal block, times up to 64 right-hand
// sides) are formed from the 8-bit digits of fx.cuh by mma.sync: 36 MMAs per
// 16 x 8 x 16 block, 14 times fewer clocks than its multiply-adds take, and one
// rounding per result. The diagonal step y_c = L_cc^{-1} x_c is a product with the
// block's inverse (k_inverse64) in place of 64 dependent substitution steps.
// mma.sync and not tcgen05: a unit's operands are made of freshly loaded values
// in registers, its N is 8 to 64, and what counts is the latency of one
// unit on the chain of levels.
//
// Operands in shared memory as whole numbers (fx::split_bytes): a tile has a
// scale per row; a vector block [right-hand side][64 entries] a scale per
// right-hand side. Where the rows of a tile are the inner dimension (backward), the
// row scales go into the vector: L_ic z_i = X_ic (2^{E_i} z_i). An inverse also has a
// scale per column, 2^{-c_k} with 2^{c_k} the size of L_kk, which goes into the other factor or
// the result: the terms of a product then are of the size of their digits, also for
// D A D with any diagonal D.
//
// With W in FP64 the residual x_c - L_cc y_c would be of the size kappa u, kappa =
// || |W| |L_cc| ||_inf, where substitution leaves u; k_inverse64 gives W to the digits' 62 bits.
// In the chunks with kappa > kFixChunk, which it marks, y_c <- y_c + W (x_c - L_cc y_c)
// follows, likewise backward. Restated on the CPU (192 x 192 Gaussian kernels; mean backward error of
// the solution, eight right-hand sides): substitution 4e-17 to 1e-16; W in FP64 1e-16 at kappa =
// 29, 1e-15 at 270, 6e-15 at 2000; W in 62 bits 8e-18 to 8e-17 up to 2000, 3e-16 at 18000; with
// the step 8e-18 to 8e-17. Blocks of diffusion matrices have kappa 4 to 15, at most 71.
#pragma once
#include "fx.cuh"
#include "kernels.cuh"

namespace sc {

constexpr float kFixChunk = 1000.f;

namespace fx {

constexpr int kLd = 66;            // 64-bit words per row of a staged tile or vector (16 bytes of skew)
constexpr int kKeyNone = -(1 << 28), kKeyBad = 1 << 24;  // exponent keys: nothing yet; an infinity or a NaN

// exponent key of x 2^e
__device__ __forceinline__ int exp_key(double x, int e) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    return ex == 0x7ff || e == kBadExp ? kKeyBad : max(ex, 1) + e;
}

// Stages a rows x w block (row stride ld, w <= 64; kLower: its lower triangle) as a 64 x 64 tile
// of digits and its row exponents: 256 threads, four per row.
template <bool kLower = false>
__device__ __forceinline__ void stage_tile(uint64_t *T, int32_t *rowE, const double *__restrict__ src, int64_t ld,
                                           int rows, int w) {
    const int r = threadIdx.x / 4, q = threadIdx.x % 4;
    const double *p = src + (int64_t)r * ld;
    double v[16];
    if (((uintptr_t)src & 15) == 0 && ld % 2 == 0 && w % 2 == 0) {
#pragma unroll
        for (int j = 0; j < 8; j++) {
            const int c = 8 * j + 2 * q;
            const double2 d = r < rows && c < w ? *reinterpret_cast<const double2 *>(p + c) : make_double2(0.0, 0.0);
            v[2 * j] = d.x;
            v[2 * j + 1] = d.y;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 16; j++) {
            const int c = 8 * (j / 2) + 2 * q + j % 2;
            v[j] = r < rows && c < w ? p[c] : 0.0;
        }
    }
    if constexpr (kLower) {
#pragma unroll
        for (int j = 0; j < 16; j++)
            if (8 * (j / 2) + 2 * q + j % 2 > r) v[j] = 0.0;
    }
    uint32_t top = 0;
#pragma unroll
    for (int j = 0; j < 16; j++) top = max(top, (uint32_t)__double2hiint(v[j]) & 0x7fffffffu);
    top = max(top, __shfl_xor_sync(0xffffffffu, top, 1));
    top = max(top, __shfl_xor_sync(0xffffffffu, top, 2));
    const int ex = (int)(top >> 20), E = max(ex, 1) - 1022;
    const bool bad = ex == 0x7ff;
    if (q == 0) rowE[r] = bad ? kBadExp : E;
#pragma unroll
    for (int j = 0; j < 8; j++)
        *reinterpret_cast<ulonglong2 *>(T + r * kLd + 8 * j + 2 * q) =
            bad ? make_ulonglong2(0x8080808080808080ull, 0x8080808080808080ull)
                : make_ulonglong2(split_bytes(v[2 * j], E), split_bytes(v[2 * j + 1], E));
}

// Stages the digits of a chunk's inverse (k_inverse64), their row exponents and minus
// their column exponents: W_jk = X_jk 2^{rowE_j + colE_k}.
__device__ __forceinline__ void stage_inverse(uint64_t *T, int32_t *rowE, int32_t *colE,
                                              const uint64_t *__restrict__ inv, const int32_t *__restrict__ exps,
                                              const int32_t *__restrict__ cexps, int w) {
    constexpr int kIt = 64 * 64 / 256;
    uint64_t v[kIt];
#pragma unroll
    for (int i = 0; i < kIt; i++) {
        const int e = threadIdx.x + i * 256, r = e / 64, c = e % 64;
        v[i] = r < w && c < w ? inv[r * w + c] : 0x8080808080808080ull;
    }
#pragma unroll
    for (int i = 0; i < kIt; i++) {
        const int e = threadIdx.x + i * 256;
        T[e / 64 * kLd + e % 64] = v[i];
    }
    if (threadIdx.x < 64) {
        rowE[threadIdx.x] = (int)threadIdx.x < w ? exps[threadIdx.x] : -1021;
        colE[threadIdx.x] = (int)threadIdx.x < w ? cexps[threadIdx.x] : 0;
    }
}

// Digit s (0: the highest) of two staged values as FP16: 1024 + byte, less 1152.
template <int s>
__device__ __forceinline__ uint32_t digits(const ulonglong2 &x) {
    constexpr int b = 3 - s % 4, sel = b | b << 4 | (4 + b) << 8 | (4 + b) << 12;
    const uint32_t w0 = s < 4 ? (uint32_t)(x.x >> 32) : (uint32_t)x.x, w1 = s < 4 ? (uint32_t)(x.y >> 32) : (uint32_t)x.y;
    uint32_t h = (__byte_perm(w0, w1, sel) & 0x00ff00ffu) | 0x64006400u;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h) : "r"(h), "r"(0x64806480u));
    return h;
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
template <int i>
__device__ __forceinline__ void digit_row(float (&acc)[S][4], const ulonglong2 (&x)[4], const uint32_t (&b)[S][2]) {
    const uint32_t a[4] = {digits<i>(x[0]), digits<i>(x[1]), digits<i>(x[2]), digits<i>(x[3])};
#pragma unroll
    for (int j = 0; j < S - i; j++) mma_16816(acc[i + j], a, b[j]);
}

// The 36 MMAs of a 16 x 8 x 16 block: x the staged pairs of rows g, g + 8 at columns 2 t, and
// at columns 2 t + 8; y0, y1 those of the other operand's row g.
__device__ __forceinline__ void digit_product(float (&acc)[S][4], const ulonglong2 (&x)[4], const ulonglong2 &y0,
                                              const ulonglong2 &y1) {
    const uint32_t b[S][2] = {{digits<0>(y0), digits<0>(y1)}, {digits<1>(y0), digits<1>(y1)},
                              {digits<2>(y0), digits<2>(y1)}, {digits<3>(y0), digits<3>(y1)},
                              {digits<4>(y0), digits<4>(y1)}, {digits<5>(y0), digits<5>(y1)},
                              {digits<6>(y0), digits<6>(y1)}, {digits<7>(y0), digits<7>(y1)}};
    digit_row<0>(acc, x, b);
    digit_row<1>(acc, x, b);
    digit_row<2>(acc, x, b);
    digit_row<3>(acc, x, b);
    digit_row<4>(acc, x, b);
    digit_row<5>(acc, x, b);
    digit_row<6>(acc, x, b);
    digit_row<7>(acc, x, b);
}
// a += register e of a block's group sums over at most 64 columns: every pair of groups
// fits in 32 bits (|g_7| < 2^22.6)
__device__ __forceinline__ void acc_add64(Acc96 &a, const float (&acc)[S][4], int e) {
    auto pair = [&](int s) { return __float2int_rn(acc[s][e]) * 256 + __float2int_rn(acc[s + 1][e]); };
    const int64_t H = ((int64_t)pair(0) << 16) + pair(2), L = ((int64_t)pair(4) << 16) + pair(6);
    const uint32_t r = a.r + (uint32_t)L;
    a.t += H + (L >> 32) + (r < (uint32_t)L ? 1 : 0);
    a.r = r;
}

// Group sums of a 16 x 8 block of T V (or T^T V): rows 16 mb .. + 15 of the result,
// right-hand sides n0 .. n0 + 7, inner dimension 16 ks0 .. 16 ks1 - 1. Lane l holds rows l / 4
// (registers 0, 1) and l / 4 + 8 (2, 3), columns 2 (l % 4) and + 1.
template <bool kTrans>
__device__ __forceinline__ void product(const uint64_t *T, const uint64_t *V, int mb, int n0, int ks0, int ks1,
                                        float (&acc)[S][4]) {
    const int lane = threadIdx.x % 32, g = lane / 4, t = lane % 4;
#pragma unroll
    for (int s = 0; s < S; s++)
#pragma unroll
        for (int e = 0; e < 4; e++) acc[s][e] = 0.f;
#pragma unroll 1
    for (int ks = ks0; ks < ks1; ks++) {
        const int k = 16 * ks + 2 * t, m = 16 * mb + g;
        ulonglong2 x[4];
        if constexpr (kTrans) {
            const uint64_t *p = T + k * kLd + m;
            x[0] = make_ulonglong2(p[0], p[kLd]);
            x[1] = make_ulonglong2(p[8], p[kLd + 8]);
            x[2] = make_ulonglong2(p[8 * kLd], p[9 * kLd]);
            x[3] = make_ulonglong2(p[8 * kLd + 8], p[9 * kLd + 8]);
        } else {
            const uint64_t *p = T + m * kLd + k;
            x[0] = *reinterpret_cast<const ulonglong2 *>(p);
            x[1] = *reinterpret_cast<const ulonglong2 *>(p + 8 * kLd);
            x[2] = *reinterpret_cast<const ulonglong2 *>(p + 8);
            x[3] = *reinterpret_cast<const ulonglong2 *>(p + 8 * kLd + 8);
        }
        const uint64_t *v = V + (n0 + g) * kLd + k;
        const ulonglong2 y0 = *reinterpret_cast<const ulonglong2 *>(v), y1 = *reinterpret_cast<const ulonglong2 *>(v + 8);
        digit_product(acc, x, y0, y1);
    }
}
// value of register e of a block's group sums, times 2^(er + ec)
__device__ __forceinline__ double block_value(const float (&acc)[S][4], int e, int er, int ec) {
    if (er == kBadExp || ec == kBadExp) return __longlong_as_double(0x7ff8000000000000ll);
    Acc96 a{0, 0};
    acc_add64(a, acc, e);
    return acc_value(a, er + ec);
}

// A warp's part of a 64 x nb block of values, in the layout of the products: rows
// 16 (warp % 4) + g + 8 (e / 2), right-hand sides 8 (warp / 4 + 2 b) + 2 t + e % 2.
template <int NB>
struct Frag {
    double v[NB][4];
    static __device__ __forceinline__ int row(int e) {
        return 16 * ((int)threadIdx.x / 32 % 4) + (int)threadIdx.x % 32 / 4 + 8 * (e / 2);
    }
    static __device__ __forceinline__ int n0(int b) { return 8 * ((int)threadIdx.x / 128 + 2 * b); }
    static __device__ __forceinline__ int col(int b, int e) { return n0(b) + 2 * ((int)threadIdx.x % 4) + e % 2; }
    // v = f(row, column) inside rows x nb, 0 elsewhere
    template <typename F>
    __device__ __forceinline__ void load(int rows, int nb, F &&f) {
#pragma unroll
        for (int b = 0; b < NB; b++)
#pragma unroll
            for (int e = 0; e < 4; e++) v[b][e] = row(e) < rows && col(b, e) < nb ? f(row(e), col(b, e)) : 0.0;
    }
    template <typename F>
    __device__ __forceinline__ void each(int rows, int nb, F &&f) const {
#pragma unroll
        for (int b = 0; b < NB; b++)
#pragma unroll
            for (int e = 0; e < 4; e++)
                if (row(e) < rows && col(b, e) < nb) f(row(e), col(b, e), v[b][e]);
    }
    // Column exponents of the block, row r scaled by 2^{addE[r]} (addE NULL: by 1),
    // into key[] (set to kKeyNone before); barrier; then put() writes the digits.
    __device__ __forceinline__ void keys(int nb, const int32_t *addE, int *key) const {
        const int e0 = addE ? addE[row(0)] : 0, e1 = addE ? addE[row(2)] : 0;
#pragma unroll
        for (int b = 0; b < NB; b++) {
            if (n0(b) >= nb) break;
            int k0 = max(exp_key(v[b][0], e0), exp_key(v[b][2], e1)), k1 = max(exp_key(v[b][1], e0), exp_key(v[b][3], e1));
#pragma unroll
            for (int o = 4; o < 32; o *= 2) {
                k0 = max(k0, __shfl_xor_sync(0xffffffffu, k0, o));
                k1 = max(k1, __shfl_xor_sync(0xffffffffu, k1, o));
            }
            if (threadIdx.x % 32 < 4) {
                atomicMax(key + col(b, 0), k0);
                atomicMax(key + col(b, 1), k1);
            }
        }
    }
    __device__ __forceinline__ void put(int nb, const int32_t *addE, const int *key, uint64_t *V) const {
        const int e0 = addE ? addE[row(0)] : 0, e1 = addE ? addE[row(2)] : 0;
#pragma unroll
        for (int b = 0; b < NB; b++) {
            if (n0(b) >= nb) break;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int k = key[col(b, e)];
                V[col(b, e) * kLd + row(e)] =
                    k == kKeyBad ? 0x8080808080808080ull : split_bytes(v[b][e], k - 1022 - (e < 2 ? e0 : e1));
            }
        }
    }
    // v = T V (or T^T V); rowE: the exponents of the result's rows (NULL: none)
    template <bool kTrans, bool kAdd>
    __device__ __forceinline__ void mul(const uint64_t *T, const int32_t *rowE, const uint64_t *V, const int *key,
                                        int K, int M, int nb) {
        const int mb = (int)threadIdx.x / 32 % 4;
#pragma unroll
        for (int b = 0; b < NB; b++) {
            if (n0(b) >= nb || 16 * mb >= M) break;
            float acc[S][4];
            product<kTrans>(T, V, mb, n0(b), 0, (K + 15) / 16, acc);
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int k = key[col(b, e)];
                const double x = block_value(acc, e, rowE ? rowE[row(e)] : 0, k == kKeyBad ? kBadExp : k - 1022);
                v[b][e] = kAdd ? v[b][e] + x : x;
            }
        }
    }
};

// shared memory of a sweep CTA for blocks of nb right-hand sides: two tiles, one
// vector block (the narrow tiles' slices, 8 x 16 x nb values, fit in the tiles)
inline size_t sweep64_smem(int nb) { return 8 * (size_t)kLd * (128 + (nb + 7) / 8 * 8); }

}  // namespace fx
}  // namespace sc
