// Device-side RLB loops (Alg. 5's small products) of an FP64 factor, by digits (fx.cuh)
// and mma.sync. An item's rows -- block B, if the item starts with its SYRK, and the
// runs B' after it -- are consecutive in J's panel and meet the same rows of B, so the item is
// one product of all its rows, cut into 16 x 8 blocks, a warp each; only where a row of the
// result goes differs from block to block (row_blk: row -> block; relindB: block -> row
// of P). Product by product the blocks would be mostly padding: runs of a few rows
// against a few columns are what these loops hold.
// A block takes some 450 issue slots for 16 columns of K, where the FP64 pipe takes a warp
// 64 clocks for each multiply-add. Below kFxMinK columns splitting the operands would
// be most of the work: an output per thread. Loop class, before (FP64 pipe, product by
// product) and after: 48^3 3.17 -> 1.82 ms, 37x41x29 graph-ordered 3.18 -> 2.21,
// 80^3 27-point 47.5 -> 38.9.
#pragma once
#include "sweep64.cuh"

namespace sc {

constexpr int kFxMinK = 6;

namespace fx {

// Block of A B^T (A and B rows of one panel, row stride ld, K columns; ni <= 16 rows,
// nj <= 8 columns): put(e, i, j, v) for the lane's entries inside it, e < 2 in row l / 4, else in row l / 4 + 8.
template <typename Put>
__device__ __forceinline__ void loop_block(const double *__restrict__ A, const double *__restrict__ B, int64_t ld, int K,
                                           int ni, int nj, Put &&put) {
    const int lane = threadIdx.x % 32, g = lane / 4, t = lane % 4;
    const bool a0 = g < ni, a1 = g + 8 < ni, b0 = g < nj;
    const double *pa = A + g * ld, *pb = B + g * ld;
    // row exponents: the lane's rows g, g + 8 of A and g of B over all of K
    uint32_t ta0 = 0, ta1 = 0, tb = 0;
    auto hi = [](double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; };
#pragma unroll 2
    for (int k = t; k < K; k += 4) {
        if (a0) ta0 = max(ta0, hi(pa[k]));
        if (a1) ta1 = max(ta1, hi(pa[8 * ld + k]));
        if (b0) tb = max(tb, hi(pb[k]));
    }
#pragma unroll
    for (int o = 1; o < 4; o *= 2) {
        ta0 = max(ta0, __shfl_xor_sync(0xffffffffu, ta0, o));
        ta1 = max(ta1, __shfl_xor_sync(0xffffffffu, ta1, o));
        tb = max(tb, __shfl_xor_sync(0xffffffffu, tb, o));
    }
    auto exp_of = [](uint32_t h) { return h >= 0x7ff00000u ? kBadExp : max((int)(h >> 20), 1) - 1022; };
    const int ea0 = exp_of(ta0), ea1 = exp_of(ta1), eb = exp_of(tb);
    // digits of columns k and k + 1 of a row
    auto pair = [&](const double *p, bool on, int e, int k) {
        const bool ok = on && e != kBadExp;
        return make_ulonglong2(ok && k < K ? split_bytes(p[k], e) : 0x8080808080808080ull,
                               ok && k + 1 < K ? split_bytes(p[k + 1], e) : 0x8080808080808080ull);
    };
    Acc96 sum[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
#pragma unroll 1
    for (int kb = 0; kb < K; kb += 64) {
        float acc[S][4];
#pragma unroll
        for (int s = 0; s < S; s++)
#pragma unroll
            for (int e = 0; e < 4; e++) acc[s][e] = 0.f;
#pragma unroll 1
        for (int k0 = kb; k0 < min(K, kb + 64); k0 += 16) {
            const int k = k0 + 2 * t;
            const ulonglong2 x[4] = {pair(pa, a0, ea0, k), pair(pa + 8 * ld, a1, ea1, k), pair(pa, a0, ea0, k + 8),
                                     pair(pa + 8 * ld, a1, ea1, k + 8)};
            const ulonglong2 y0 = pair(pb, b0, eb, k), y1 = pair(pb, b0, eb, k + 8);
            digit_product(acc, x, y0, y1);
        }
#pragma unroll
        for (int e = 0; e < 4; e++) acc_add64(sum[e], acc, e);
    }
    // lane: rows g and g + 8, columns 2 t and 2 t + 1, whose exponents lanes 8 t and 8 t + 4 hold
    const int e0 = __shfl_sync(0xffffffffu, eb, 8 * t), e1 = __shfl_sync(0xffffffffu, eb, 8 * t + 4);
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const int i = g + 8 * (e / 2), j = 2 * t + e % 2, er = e < 2 ? ea0 : ea1, ec = e % 2 ? e1 : e0;
        if (i >= ni || j >= nj) continue;
        put(e, i, j, er == kBadExp || ec == kBadExp ? __longlong_as_double(0x7ff8000000000000ll)
                                                    : acc_value(sum[e], er + ec));
    }
}

}  // namespace fx

// One loop item, its blocks dealt to `nwarps` warps (this one is `warp`).
__device__ __forceinline__ void loop_item64(double *__restrict__ lnz, const LoopItem &it, const SnDev *__restrict__ sn,
                                            const BlkDev *__restrict__ blk, const int32_t *__restrict__ rb_val,
                                            const int32_t *__restrict__ row_blk, int warp, int nwarps) {
    const SnDev J = sn[it.sn];
    const BlkDev B = blk[it.b];
    const SnDev P = sn[B.owner];
    const int K = J.n, nb = B.size, lane = threadIdx.x % 32;
    const int64_t ld = J.ld;
    const double *src = lnz + J.off, *rowsB = src + (int64_t)B.pos * ld;
    // rows [r0, r1) of J's panel
    const int r0 = it.r_lo == it.b ? B.pos : it.r_lo < J.b1 ? blk[it.r_lo].pos : J.m;
    const int r1 = it.r_hi < J.b1 ? blk[it.r_hi].pos : J.m;
    double *C = lnz + P.off + (B.first - P.f);
    // target row of row r of J; columns from `lo` on are above the diagonal
    auto target = [&](int r, int &lo) {
        const int q = row_blk[J.gl + r], rowP = P.m - 1 - rb_val[B.rb + (q - B.bs)] + r - blk[q].pos;
        lo = q == it.b ? r - B.pos + 1 : nb;
        return C + (int64_t)rowP * P.ld;
    };
    if (K < kFxMinK) {
        for (int e = warp * 32 + lane; e < (r1 - r0) * nb; e += 32 * nwarps) {
            const int r = r0 + e / nb, j = e % nb;
            int lo;
            double *c = target(r, lo);
            if (j >= lo) continue;
            double acc = 0.0;
            for (int k = 0; k < K; k++) acc += src[r * ld + k] * rowsB[j * ld + k];
            atomicAdd(c + j, -acc);
        }
        return;
    }
    int task = 0;
#pragma unroll 1
    for (int i0 = r0; i0 < r1; i0 += 16) {
#pragma unroll 1
        for (int j0 = 0; j0 < nb; j0 += 8) {
            if (task++ % nwarps != warp) continue;
            const int ia = i0 + lane / 4, ib = ia + 8;
            int lo0 = 0, lo1 = 0;
            double *c0 = C, *c1 = C;
            // (entries from lo on are above the diagonal)
            if (ia < r1) c0 = target(ia, lo0);
            if (ib < r1) c1 = target(ib, lo1);
            fx::loop_block(src + i0 * ld, rowsB + j0 * ld, ld, K, min(16, r1 - i0), min(8, nb - j0),
                           [&](int e, int, int j, double v) {
                               if (j0 + j < (e < 2 ? lo0 : lo1)) atomicAdd((e < 2 ? c0 : c1) + j0 + j, -v);
                           });
        }
    }
}

__global__ void __launch_bounds__(256, 2) k_rlb_loop64(double *__restrict__ lnz, const LoopItem *__restrict__ items,
                                                       const SnDev *__restrict__ sn, const BlkDev *__restrict__ blk,
                                                       const int32_t *__restrict__ rb_val,
                                                       const int32_t *__restrict__ row_blk) {
    loop_item64(lnz, items[blockIdx.x], sn, blk, rb_val, row_blk, threadIdx.x / 32, 8);
}
__global__ void __launch_bounds__(256, 2) k_rlb_loop_warp64(double *__restrict__ lnz,
                                                            const LoopItem *__restrict__ items, int count,
                                                            const SnDev *__restrict__ sn,
                                                            const BlkDev *__restrict__ blk,
                                                            const int32_t *__restrict__ rb_val,
                                                            const int32_t *__restrict__ row_blk) {
    const int idx = blockIdx.x * 8 + threadIdx.x / 32;
    if (idx < count) loop_item64(lnz, items[idx], sn, blk, rb_val, row_blk, 0, 1);
}

// The product tiles of k_split_gemm (128 x 64) straight from the panels, for handles without
// a slice pool (no memory for it): a warp takes 16 rows, eight columns at a time. The digits, the rows'
// exponents and the sums are k_split_gemm's, and the sums are exact, so L has the same
// bits with and without the pool.
__global__ void __launch_bounds__(256, 2) k_digit_tiles(double *__restrict__ lnz, double *__restrict__ upool,
                                                        const Task *__restrict__ tasks,
                                                        const GemmTile *__restrict__ tiles) {
    const GemmTile tl = tiles[blockIdx.x];
    const Task tk = tasks[tl.task];
    const int i0 = tl.tm * 128 + threadIdx.x / 32 * 16, ni = min(16, tk.m - i0);
    if (ni <= 0) return;
    const bool lower = tk.flags & kTaskLower, store = tk.flags & kTaskStoreU, excl = tk.flags & kTaskExclusive;
    double *C = (store ? upool : lnz) + tk.c_off + (int64_t)i0 * tk.ldc;
#pragma unroll 1
    for (int j0 = tl.tn * 64; j0 < min(tk.n, tl.tn * 64 + 64); j0 += 8) {
        if (lower && i0 + ni - 1 < j0) break;
        fx::loop_block(lnz + tk.a_off + (int64_t)i0 * tk.lds, lnz + tk.b_off + (int64_t)j0 * tk.lds, tk.lds, tk.k, ni,
                       min(8, tk.n - j0), [&](int, int i, int j, double v) {
                           if (lower && j0 + j > i0 + i) return;
                           double *c = C + (int64_t)i * tk.ldc + j0 + j;
                           if (store) *c = -v;
                           else if (excl) *c -= v;
                           else atomicAdd(c, -v);
                       });
    }
}

}  // namespace sc
