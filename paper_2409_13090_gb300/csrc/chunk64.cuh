// FP64 POTRF and TRSM of a chunk (at most 64 columns) in panels of 16 columns, products
// by digits (fx.cuh, sweep64.cuh) instead of the FP64 pipe, whose multiply-add takes a
// warp 64 clocks.
//
// Panel p, rows at or below it:
//   S_p <- S_p - sum_{q < p} X_q L_pq^T     mma.sync, one drain per q
//   diagonal 16 x 16 block (POTRF only)     L D L^T in FP64, then W = L_pp^{-1}
//   X_p = S_p W^T                           mma.sync
// Digits of a row's 16 columns have an exponent of their own, so no bound on the
// factor's entries is assumed (a matrix that is not positive definite reaches its
// failing pivot with the values it had). In S_p W^T the inner index runs over
// columns whose scales may differ by any amount (S_ik ~ s_k, W_jk ~ 1 / s_k in D A D): S's
// columns are taken times 2^{-c_k}, W's times 2^{c_k}, with 2^{c_k} the size of L_kk.
//
// The residual S_p - X_p L_pp^T of that product is of the size kappa u, kappa =
// || |W| |L_pp| ||_inf, where substitution leaves u. Where kappa > kFixPanel one step
//   X_p <- X_p + (S_p - X_p L_pp^T) W^T
// follows, whose residual is (kappa u)^2 + u (kappa < 1e8: L_pp is the factor of a matrix
// that FP64 can factor). Restated on the CPU (Gaussian kernels and chains, 192 points, kappa
// from 5 to 1e6; residual over sqrt(a_ii a_jj)): FP64 operations 2e-16 to 1.7e-15; without the
// step 2e-16 to 5e-16 up to kappa = 50, 7e-12 at 1e6, and pivots <= 0 in matrices that
// can be factored; with it 2e-16 to 6e-16. Diffusion matrices have kappa 5 to 10, at most 40.
// Forming kappa costs some 2 us a level (48^3 FP64 step 18.03 -> 18.33 ms, 64^2 0.761 -> 0.788).
//
// Measured, 64 columns: the FP64-pipe kernels took 70 us for the POTRF (64 pivots of some
// 900 clocks, and a rank-8 update of 27 us in all) and 19 us for a TRSM tile of
// 16 rows. This POTRF: some 97,000 clocks (51 us), between the barriers of a copy with clock
// stamps: the pivots 59,000, W's elimination 12,000, digits 14,000, products 7,000, the
// slot 3,600. The pivots' chain bounds it.
#pragma once
#include "sweep64.cuh"

namespace sc {

constexpr float kFixPanel = 32.f;

// dynamic shared memory: the L or X digits of 64 rows (two tiles in the TRSM) and the W digits
constexpr int kChunk64Smem = 8 * fx::kLd * (64 + 64 + 16);

namespace fx {

// Row exponent keys of a 16 x 8 block in fragment layout (rows g and g + 8 of block mb),
// its columns times 2^{e0} and 2^{e1}: into key[64].
__device__ __forceinline__ void row_keys(const double (&v)[4], int mb, int *key, int e0 = 0, int e1 = 0) {
    const int lane = threadIdx.x % 32;
    int k0 = max(exp_key(v[0], e0), exp_key(v[1], e1)), k1 = max(exp_key(v[2], e0), exp_key(v[3], e1));
#pragma unroll
    for (int o = 1; o < 4; o *= 2) {
        k0 = max(k0, __shfl_xor_sync(0xffffffffu, k0, o));
        k1 = max(k1, __shfl_xor_sync(0xffffffffu, k1, o));
    }
    if (lane % 4 == 0) {
        atomicMax(key + 16 * mb + lane / 4, k0);
        atomicMax(key + 16 * mb + lane / 4 + 8, k1);
    }
}
__device__ __forceinline__ int key_exp(int k) { return k == kKeyBad ? kBadExp : k - 1022; }
// digits of the block's values into columns c0 .. c0 + 7 of T
__device__ __forceinline__ void row_put(const double (&v)[4], int mb, int c0, const int *key, uint64_t *T, int e0 = 0,
                                        int e1 = 0) {
    const int lane = threadIdx.x % 32;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int r = 16 * mb + lane / 4 + 8 * h, k = key[r];
        const bool bad = k == kKeyBad;
        *reinterpret_cast<ulonglong2 *>(T + r * kLd + c0 + 2 * (lane % 4)) =
            make_ulonglong2(bad ? 0x8080808080808080ull : split_bytes(v[2 * h], k - 1022 - e0),
                            bad ? 0x8080808080808080ull : split_bytes(v[2 * h + 1], k - 1022 - e1));
    }
}
// v -= (panel q of rows 16 mb .. of T) (panel q of rows n0 .. n0 + 7 of V)^T
__device__ __forceinline__ void panel_sub(double (&v)[4], const uint64_t *T, const uint64_t *V, int mb, int n0, int q,
                                          const int *keyT, const int *keyV) {
    float acc[S][4];
    product<false>(T, V, mb, n0, q, q + 1, acc);
    const int lane = threadIdx.x % 32;
#pragma unroll
    for (int e = 0; e < 4; e++)
        v[e] -= block_value(acc, e, key_exp(keyT[16 * mb + lane / 4 + 8 * (e / 2)]),
                            key_exp(keyV[n0 + 2 * (lane % 4) + e % 2]));
}
// v = (panel p of rows 16 mb .. of T) (panel p of rows n0 .. of V)^T
__device__ __forceinline__ void panel_mul(double (&v)[4], const uint64_t *T, const uint64_t *V, int mb, int n0, int p,
                                          const int *keyT, const int *keyV) {
    float acc[S][4];
    product<false>(T, V, mb, n0, p, p + 1, acc);
    const int lane = threadIdx.x % 32;
#pragma unroll
    for (int e = 0; e < 4; e++)
        v[e] = block_value(acc, e, key_exp(keyT[16 * mb + lane / 4 + 8 * (e / 2)]),
                           key_exp(keyV[n0 + 2 * (lane % 4) + e % 2]));
}

// The second step for the rows of block mb, columns 8 nb .. + 7 of panel p (by every warp of
// the CTA; `on`: this one has rows): s holds X_p = S_p W^T, whose keys are in keyX, r holds
// S_p (its digits would not do: they are relative to the row's largest S_ik 2^{-c_k}, of any
// size beside the others). L: the rows of L_pp's digits. keyX of the rows from row0 on is left reset.
__device__ __forceinline__ void panel_fix(double (&s)[4], double (&r)[4], bool on, uint64_t *X, const uint64_t *W,
                                          const uint64_t *L, int mb, int nb, int p, int *keyS, int *keyX,
                                          const int *keyL, const int *keyW, int row0, int c0, int c1) {
    if (on) row_put(s, mb, 16 * p + 8 * nb, keyX, X);
    __syncthreads();
    if (threadIdx.x < 64) keyS[threadIdx.x] = kKeyNone;
    if (on) panel_sub(r, X, L, mb, 8 * nb, p, keyX, keyL);
    __syncthreads();  // keyS reset; X's digits and keys have been read
    if ((int)threadIdx.x >= row0 && threadIdx.x < 64) keyX[threadIdx.x] = kKeyNone;
    if (on) row_keys(r, mb, keyS, -c0, -c1);
    __syncthreads();
    if (on) row_put(r, mb, 16 * p + 8 * nb, keyS, X, -c0, -c1);
    __syncthreads();
    if (on) {
        panel_mul(r, X, W, mb, 8 * nb, p, keyS, keyW);
#pragma unroll
        for (int e = 0; e < 4; e++) s[e] += r[e];
    }
}

// L D L^T of a 16 x 16 block a (lower triangle) by the first four warps: u = the unit
// lower factor below the diagonal, d = the pivots. A thread holds one entry of the
// columns 1 .. 15 (120 of them, so every FP64 unit takes five multiply-adds a
// pivot and no more); the pivot's column goes through shared memory. 1 / d: the
// hardware's approximation y and 1 + e + e^2, e = 1 - d y (the geometric series;
// |e| < 2^-20, so what is left is below 2^-60). A pivot <= 0 sets info and counts as 1.
// 14,800 clocks for 16 pivots, 930 each: four dependent FP64 operations, the column through
// shared memory and a barrier.
__device__ __forceinline__ void ldl16(const double (*a)[17], double (*u)[17], double *d, double (*col)[16], int w,
                                      int col0, int32_t *__restrict__ info) {
    const int t = threadIdx.x;
    int i = 1;
    while (i * (i + 1) / 2 <= t) i++;  // rows 1 .. 15 hold 1 .. 15 entries
    const int j = t - i * (i - 1) / 2 + 1;
    const bool live = i < 16;
    double r = live ? a[i][j] : 0.0;
    if (t < 16) col[0][t] = a[t][0];
    asm volatile("bar.sync 1, 128;" ::: "memory");
    w = min(w, 16);  // past the chunk: the identity
    if (t < 16 && t >= w) d[t] = 1.0;
    for (int e = t; e < 256; e += 128)
        if (e % 16 >= w) u[e / 16][e % 16] = 0.0;
#pragma unroll 1
    for (int k = 0; k < w; k++) {
        const double *ck = col[k & 1];
        double dk = ck[k];
        const double aik = live ? ck[i] : 0.0, ajk = live ? ck[j] : 0.0;
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(dk));
        const double e = fma(-dk, y, 1.0), x = ajk * y;
        double uk = fma(x, fma(e, e, e), x);
        // outside 2^-991 <= dk < 2^993 (on the high word: a comparison in FP64 takes the
        // pipe 64 clocks too)
        if ((unsigned)(__double2hiint(dk) - 0x02000000) >= 0x7c000000u) {
            if (!(dk > 0.0)) {
                if (t == 0) atomicMin(info, col0 + k + 1);
                dk = 1.0;
            }
            uk = ajk / dk;
        }
        if (t == 0) d[k] = dk;
        if (live && j > k) {
            r -= aik * uk;
            if (i == j) u[j][k] = uk;
            if (j == k + 1) col[(k + 1) & 1][i] = r;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
    }
}

// || |W| |L| ||_inf of 16 x 16 blocks by one warp, sums in a fixed order
__device__ __forceinline__ float condition16(const float (*W)[17], const float (*L)[17]) {
    const int lane = threadIdx.x % 32, i = lane % 16, k0 = lane / 16 * 8;
    float rho = 0.f, kap = 0.f;
#pragma unroll
    for (int k = 0; k < 8; k++) rho += L[i][k0 + k];
    rho += __shfl_xor_sync(0xffffffffu, rho, 16);
#pragma unroll
    for (int k = 0; k < 8; k++) kap += W[i][k0 + k] * __shfl_sync(0xffffffffu, rho, k0 + k);
    kap += __shfl_xor_sync(0xffffffffu, kap, 16);
#pragma unroll
    for (int o = 1; o < 16; o *= 2) kap = fmaxf(kap, __shfl_xor_sync(0xffffffffu, kap, o));
    return kap;
}

// c with 2^c about sqrt(d)
__device__ __forceinline__ int half_exp(double d) { return (((__double2hiint(d) >> 20) & 0x7ff) - 1023) >> 1; }

}  // namespace fx

// POTRF of chunk list[blockIdx.x]; leaves L_cc's digits, the W digits and the exponent
// keys in the chunk's slot for the TRSM.
__global__ void __launch_bounds__(256) k_potrf64(double *__restrict__ lnz, const ChunkDev *__restrict__ chunks,
                                                 const int32_t *__restrict__ list, int32_t *__restrict__ info,
                                                 uint64_t *__restrict__ slots) {
    extern __shared__ __align__(16) unsigned char smem_chunk64[];
    uint64_t *X = reinterpret_cast<uint64_t *>(smem_chunk64), *W = X + 64 * fx::kLd;  // W: 16 rows
    __shared__ double blk[16][17], u[16][17], d[16], rs[16], col[2][16];
    __shared__ int keyS[4][64], keyX[4][64], keyW[64], cexp[64], fix[4];
    __shared__ float sizeL[16][17], sizeW[16][17];
    const ChunkDev ch = chunks[list[blockIdx.x]];
    const int w = ch.w, np = (w + 15) / 16;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, mb = warp % 4, nb = warp / 4;
    double *base = lnz + ch.off + (int64_t)ch.c0 * ch.ld + ch.c0;
    const int row0 = 16 * mb + lane / 4, colx = 8 * nb + 2 * (lane % 4);  // rows row0, + 8; columns 16 p + colx, + 1
    double s[4][4];
#pragma unroll
    for (int p = 0; p < 4; p++)
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int r = row0 + 8 * (e / 2), c = 16 * p + colx + e % 2;
            // past the chunk: the identity
            s[p][e] = r < w && c <= r ? base[(int64_t)r * ch.ld + c] : (r == c ? 1.0 : 0.0);
        }
    if (threadIdx.x < 64) {
#pragma unroll
        for (int p = 0; p < 4; p++) keyS[p][threadIdx.x] = keyX[p][threadIdx.x] = fx::kKeyNone;
        keyW[threadIdx.x] = fx::kKeyNone;
    }
    __syncthreads();
    // (p not unrolled, the panels move down instead: the code of one turn stays in the
    // instruction cache; unrolled, fetching it took longer than running it)
#pragma unroll 1
    for (int p = 0; p < np; p++) {
        double (&sp)[4] = s[0];
        if (mb >= p && mb < np)
#pragma unroll 1
            for (int q = 0; q < p; q++)
                fx::panel_sub(sp, X, X + 16 * p * fx::kLd, mb, 8 * nb, q, keyX[q], keyX[q] + 16 * p);
        if (mb == p) {
#pragma unroll
            for (int e = 0; e < 4; e++) blk[lane / 4 + 8 * (e / 2)][colx + e % 2] = sp[e];
        }
        __syncthreads();
        if (warp < 4) {
            fx::ldl16(blk, u, d, col, w - 16 * p, ch.col0 + 16 * p, info);
            if (threadIdx.x < 16) {
                rs[lane] = fast_rsqrt(d[lane]);
                cexp[16 * p + lane] = fx::half_exp(d[lane]);
            }
        }
        __syncthreads();
        const int c0 = cexp[16 * p + colx], c1 = cexp[16 * p + colx + 1];
        if (mb > p && mb < np) fx::row_keys(sp, mb, keyS[p], -c0, -c1);
        // L_pp = u D^{1/2} (thread: row i, column j); W = D^{-1/2} u^{-1} by rows of
        // elimination, columns 2 warp and 2 warp + 1 in a warp's two halves
        double wv;
        {
            const int i = lane % 16, j = 2 * warp + lane / 16;
            double ui[16];
#pragma unroll
            for (int k = 0; k < 15; k++) ui[k] = u[i][k];
            wv = i == j ? 1.0 : 0.0;
#pragma unroll
            for (int k = 0; k < 15; k++) {
                if (16 * p + k + 1 >= w) break;
                const double wk = __shfl_sync(0xffffffffu, wv, k + (lane & 16));
                if (i > k) wv -= ui[k] * wk;
            }
            wv *= rs[i];
            sizeW[i][j] = fx::size_of(wv, cexp[16 * p + j]);
            atomicMax(&keyW[16 * p + i], fx::exp_key(wv, cexp[16 * p + j]));
        }
        double lv[4] = {0.0, 0.0, 0.0, 0.0};
        if (mb == p) {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int i = lane / 4 + 8 * (e / 2), j = colx + e % 2;
                const double sq = d[j] * rs[j];
                lv[e] = i == j ? sq : i > j ? u[i][j] * sq : 0.0;
                sizeL[i][j] = fx::size_of(lv[e], -cexp[16 * p + i]);
                const int r = 16 * p + i, c = 16 * p + j;
                if (r < w && i >= j) base[(int64_t)r * ch.ld + c] = lv[e];
            }
            fx::row_keys(lv, mb, keyX[p]);
        }
        __syncthreads();
        {
            const int i = lane % 16, j = 2 * warp + lane / 16, k = keyW[16 * p + i];
            W[i * fx::kLd + 16 * p + j] =
                k == fx::kKeyBad ? 0x8080808080808080ull : fx::split_bytes(wv, k - 1022 - cexp[16 * p + j]);
        }
        if (mb == p) fx::row_put(lv, mb, 16 * p + 8 * nb, keyX[p], X);
        else if (mb > p && mb < np) fx::row_put(sp, mb, 16 * p + 8 * nb, keyS[p], X, -c0, -c1);
        __syncthreads();
        const bool on = mb > p && mb < np;
        double S[4] = {sp[0], sp[1], sp[2], sp[3]};
        if (on) {
            fx::panel_mul(sp, X, W, mb, 8 * nb, p, keyS[p], keyW + 16 * p);
            fx::row_keys(sp, mb, keyX[p]);
        } else if (warp == 0) {  // (never among these: it has the rows of panel 0)
            const float kap = fx::condition16(sizeW, sizeL);
            if (lane == 0) fix[p] = !(kap <= kFixPanel);
        }
        __syncthreads();
        if (fix[p] && p + 1 < np) {
            fx::panel_fix(sp, S, on, X, W, X + 16 * p * fx::kLd, mb, nb, p, keyS[p], keyX[p], keyX[p] + 16 * p,
                          keyW + 16 * p, 16 * p + 16, c0, c1);
            if (on) fx::row_keys(sp, mb, keyX[p]);
            __syncthreads();
        }
        if (on) {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int r = row0 + 8 * (e / 2), c = 16 * p + colx + e % 2;
                if (r < w && c < w) base[(int64_t)r * ch.ld + c] = sp[e];
            }
            fx::row_put(sp, mb, 16 * p + 8 * nb, keyX[p], X);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 3; q++)
#pragma unroll
            for (int e = 0; e < 4; e++) s[q][e] = s[q + 1][e];
    }
    // to the slot: L digits [16 np][16 np], W digits [np][16][16], keys of L [4][64], of W
    // [64], the columns' exponents [64], which panels take the second step [4]
    uint64_t *out = slots + (int64_t)ch.slot * 256;
    const int n = 16 * np;
    for (int e = threadIdx.x; e < n * n; e += 256) {
        const int r = e / n, c = e % n;
        out[e] = r / 16 >= c / 16 ? X[r * fx::kLd + c] : 0x8080808080808080ull;
    }
    out += n * n;
    for (int e = threadIdx.x; e < np * 256; e += 256) out[e] = W[e / 16 % 16 * fx::kLd + e / 256 * 16 + e % 16];
    int *ko = reinterpret_cast<int *>(out + np * 256);
    ko[threadIdx.x] = keyX[threadIdx.x / 64][threadIdx.x % 64];
    if (threadIdx.x < 64) {
        ko[256 + threadIdx.x] = keyW[threadIdx.x];
        ko[320 + threadIdx.x] = (int)threadIdx.x < n ? cexp[threadIdx.x] : 0;
        if (threadIdx.x < 4) ko[384 + threadIdx.x] = (int)threadIdx.x < np ? fix[threadIdx.x] : 0;
    }
}

// TRSM of up to 64 rows below a chunk's diagonal block.
__global__ void __launch_bounds__(256, 2) k_trsm64(double *__restrict__ lnz, const ChunkDev *__restrict__ chunks,
                                                   const TrsmTile *__restrict__ tiles,
                                                   const uint64_t *__restrict__ slots) {
    extern __shared__ __align__(16) unsigned char smem_chunk64[];
    uint64_t *X = reinterpret_cast<uint64_t *>(smem_chunk64), *L = X + 64 * fx::kLd, *W = L + 64 * fx::kLd;
    __shared__ int keyS[4][64], keyX[4][64], keyL[4][64], keyW[64], cexp[64], fix[4];
    __shared__ double keep[256][5];  // a thread's S_p (in registers it would spill)
    const TrsmTile tl = tiles[blockIdx.x];
    const ChunkDev ch = chunks[tl.chunk];
    const int w = ch.w, np = (w + 15) / 16, n = 16 * np, rows = min(kTrsm64Rows, ch.m - tl.r0);
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, mb = warp % 4, nb = warp / 4;
    const bool on = 16 * mb < rows;
    double *base = lnz + ch.off + (int64_t)tl.r0 * ch.ld + ch.c0;
    const int row0 = 16 * mb + lane / 4, colx = 8 * nb + 2 * (lane % 4);
    double s[4][4];
#pragma unroll
    for (int p = 0; p < 4; p++)
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const int r = row0 + 8 * (e / 2), c = 16 * p + colx + e % 2;
            s[p][e] = r < rows && c < w ? base[(int64_t)r * ch.ld + c] : 0.0;
        }
    const uint64_t *in = slots + (int64_t)ch.slot * 256;
    for (int e = threadIdx.x; e < n * n; e += 256) L[e / n * fx::kLd + e % n] = in[e];
    in += n * n;
    for (int e = threadIdx.x; e < np * 256; e += 256) W[e / 16 % 16 * fx::kLd + e / 256 * 16 + e % 16] = in[e];
    const int *ki = reinterpret_cast<const int *>(in + np * 256);
    keyL[threadIdx.x / 64][threadIdx.x % 64] = ki[threadIdx.x];
    keyS[threadIdx.x / 64][threadIdx.x % 64] = keyX[threadIdx.x / 64][threadIdx.x % 64] = fx::kKeyNone;
    if (threadIdx.x < 64) {
        keyW[threadIdx.x] = ki[256 + threadIdx.x];
        cexp[threadIdx.x] = ki[320 + threadIdx.x];
        if (threadIdx.x < 4) fix[threadIdx.x] = ki[384 + threadIdx.x];
    }
    __syncthreads();
#pragma unroll 1
    for (int p = 0; p < np; p++) {
        double (&sp)[4] = s[0];
        const int c0 = cexp[16 * p + colx], c1 = cexp[16 * p + colx + 1];
        if (on) {
#pragma unroll 1
            for (int q = 0; q < p; q++)
                fx::panel_sub(sp, X, L + 16 * p * fx::kLd, mb, 8 * nb, q, keyX[q], keyL[q] + 16 * p);
            fx::row_keys(sp, mb, keyS[p], -c0, -c1);
        }
        __syncthreads();
        if (on) fx::row_put(sp, mb, 16 * p + 8 * nb, keyS[p], X, -c0, -c1);
        __syncthreads();
        if (on) {
            if (fix[p]) {
#pragma unroll
                for (int e = 0; e < 4; e++) keep[threadIdx.x][e] = sp[e];
            }
            fx::panel_mul(sp, X, W, mb, 8 * nb, p, keyS[p], keyW + 16 * p);
            if (p + 1 < np || fix[p]) fx::row_keys(sp, mb, keyX[p]);
        }
        if (fix[p]) {
            __syncthreads();
            double S[4];
#pragma unroll
            for (int e = 0; e < 4; e++) S[e] = on ? keep[threadIdx.x][e] : 0.0;
            fx::panel_fix(sp, S, on, X, W, L + 16 * p * fx::kLd, mb, nb, p, keyS[p], keyX[p], keyL[p] + 16 * p,
                          keyW + 16 * p, 0, c0, c1);
            if (on) fx::row_keys(sp, mb, keyX[p]);
        }
        if (on) {
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int r = row0 + 8 * (e / 2), c = 16 * p + colx + e % 2;
                if (r < rows && c < w) base[(int64_t)r * ch.ld + c] = sp[e];
            }
        }
        if (p + 1 >= np) break;
        __syncthreads();
        if (on) fx::row_put(sp, mb, 16 * p + 8 * nb, keyX[p], X);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 3; q++)
#pragma unroll
            for (int e = 0; e < 4; e++) s[q][e] = s[q + 1][e];
    }
}

}  // namespace sc
