// FP64 product tiles on the tensor cores (sm_103a): C[128 x 64 tile] -= A B^T
// with A, B row slabs of one FP64 supernode panel, formed from products of
// 8-bit slices (error-free splitting after Ozaki, Ogita, Oishi, Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numerical Algorithms 59, 2012).
//
// Why: the FP64 pipe of this chip makes 2 multiply-adds per clock and SM
// (1.255 TFLOP/s, which the SIMT tiles reached to 97 %), the tensor cores 4096
// FP16 ones, so 36 slice products in place of one FP64 product are still far
// cheaper.
//
// Splitting (k_split): row r of the source columns [kx0, kx0 + K) has the
// exponent E_r with max |x| < 2^E_r. X = x 2^(62 - E_r), truncated to a whole number
// (|X| < 2^62), is written in 8 signed digits of base 256,
//   X = sum_i d_i 256^(8 - i),  d_i in [-128, 127]  (|d_1| <= 65),
// which are the bytes of X + 0x8080808080808080 less 128, stored as FP16 (exact).
// Product: with G_g = sum over i + j = g + 1 of the slice products,
//   sum_k x_k y_k = 2^(E_r + E_c) sum_{g = 1..8} 2^(-4 - 8 g) G_g,
// the groups g > 8 left out (fx.cuh: with the truncation a term is below 2^-58.7 of
// 2^(E_r + E_c) off, random ones 2^-62 on average). A group's sum
// over 128 columns is a whole number of at most 114944 * 128 < 2^24, so FP32
// accumulation in TMEM is exact; every 128 columns the groups are added into
// a 96-bit whole number per entry, and that is rounded to FP64 once at the end.
// A product of K columns thus has one rounding and what the digits leave out, relative to its
// rows' largest entries, where the FMA chain has K roundings: against 113-bit sums the largest error is 4 to 15 times
// smaller than the FMA chain's (K = 64 .. 512).
//
// Tile 128 x 64: the eight groups' accumulators fill the 512 TMEM columns, so the
// next 128 columns wait for the drain. A slice of A is multiplied by up to four slices
// of B in one MMA (N = 256): they lie one after another in shared memory, and so do the
// groups that the products go to. The 36 products one by one (N = 64, some 70 clocks
// each, about twice their share of the peak: 128 rows of A are read for 64 of
// B) reached 11.7 TFLOP/s (FP64 operations) at K = 64, 17.3 at 128, 19.7 at 1024 on
// 10000 x 3000, against 1.2 for the SIMT tiles; by 12 MMAs the steps of 48^3
// 7-point take 18.1 instead of 18.9 ms, 80^3 27-point 178 instead of 197, with the same bits.
// Factorizations on the SIMT tiles: 77 and 1541 ms.
#pragma once
#include <cuda.h>
#include <cudaTypedefs.h>

#include "fx.cuh"
#include "kernels.cuh"
#include "tc_gemm.cuh"

namespace sc {
namespace sp {
using namespace fx;

constexpr int BM = 128, BN = 64;       // tile
constexpr int BK = 32;                 // columns of a stage: 64 bytes of FP16, one swizzle row
constexpr int kDrain = 4;              // stages between two drains of the accumulators (128 columns)
constexpr int STAGES = 2;
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2;  // one slice of a stage
constexpr int STAGE_BYTES = S * (A_BYTES + B_BYTES);
constexpr int SMEM = STAGES * STAGE_BYTES + 1024 /*alignment*/ + 128 /*barriers*/;
static_assert(SMEM <= 227 * 1024, "shared memory per CTA");
static_assert(S * BN <= 512, "TMEM columns per SM");
constexpr int kEpiWarps = 16;                   // four per TMEM lane quarter, each 16 columns
constexpr int kThreads = 32 * (4 + kEpiWarps);  // producer warp, MMA warp, two idle warps, epilogue warps
// 96 registers a thread, 132 bytes of spills. Eight epilogue warps with twice the entries spilled their
// accumulators, and a spill goes to L2 here: the stages leave L1 some 30 KB.

// instruction descriptor: kind::f16, D = F32, A = B = F16, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t idesc_f16(int n) {
    return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}
// shared-memory matrix descriptor: K-major, 64-byte swizzle, 8-row groups 512 B apart
__device__ __forceinline__ uint64_t umma_desc_sw64(uint32_t addr) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;
    return d;
}
__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
        : "memory");
}
// 16 rows x 8 columns of an accumulator: register 2 q + h of lane l holds row
// l / 4 + 8 h, column 4 q + l % 4 (four lanes cover 32 bytes of a row of C)
__device__ __forceinline__ void tmem_ld_16x8(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.16x128b.x2.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

// --------------------------------------------------------------------- splitting
// One CTA of 256 threads splits 64 rows of a source block, four lanes per row
// (8 columns of a 32-column piece each). Piece (kb, slice i, row r) is row
// piece0 + (kb * S + i) * rows + r of the slice pool (32 FP16 values each).
// 8 bytes read and 16 written per entry (a row's exponent takes a first pass over
// its columns, whose second reading is served by L1 / L2).
__global__ void __launch_bounds__(256) k_split(const double *__restrict__ lnz, const SplitBlk *__restrict__ blks,
                                               const SplitUnit *__restrict__ units, uint16_t *__restrict__ pool,
                                               int32_t *__restrict__ exps) {
    const SplitUnit u = units[blockIdx.x];
    const SplitBlk bk = blks[u.blk];
    const int r = u.row0 + (int)threadIdx.x / 4, q = threadIdx.x % 4;
    const bool live = r < bk.rows;
    const double *src = lnz + bk.src + (int64_t)(live ? r : 0) * bk.ld;
    auto load8 = [&](int kb, double (&x)[8]) {
        const int k = kb * BK + q * 8;
        if (live && k + 8 <= bk.k) {
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                const double2 v = *reinterpret_cast<const double2 *>(src + k + i);
                x[i] = v.x;
                x[i + 1] = v.y;
            }
        } else {
#pragma unroll
            for (int i = 0; i < 8; i++) x[i] = live && k + i < bk.k ? src[k + i] : 0.0;
        }
    };
    const int nkb = (bk.k + BK - 1) / BK;
    double x[8];
    uint32_t top = 0;  // largest high word of |x|
    for (int kb = 0; kb < nkb; kb++) {
        load8(kb, x);
#pragma unroll
        for (int i = 0; i < 8; i++) top = max(top, (uint32_t)__double2hiint(x[i]) & 0x7fffffffu);
    }
    top = max(top, __shfl_xor_sync(0xffffffffu, top, 1));
    top = max(top, __shfl_xor_sync(0xffffffffu, top, 2));
    const int ex = (int)(top >> 20);
    const bool bad = ex == 0x7ff;
    const int E = max(ex, 1) - 1022;  // |x| < 2^E
    if (live && q == 0) exps[bk.exp0 + r] = bad ? kBadExp : E;
    for (int kb = 0; kb < nkb; kb++) {
        if (nkb > 1) load8(kb, x);
        uint64_t y[8];
#pragma unroll
        for (int i = 0; i < 8; i++) y[i] = bad ? 0x8080808080808080ull : split_bytes(x[i], E);
        if (!live) continue;
#pragma unroll
        for (int s = 0; s < S; s++) {
            const int sh = 8 * (S - 1 - s);
            uint32_t w[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
                // two digits as FP16: 1024 + byte, less 1152
                const uint32_t lo = (uint32_t)(y[2 * i] >> sh) & 0xffu, hi = (uint32_t)(y[2 * i + 1] >> sh) & 0xffu;
                uint32_t h2 = 0x64006400u | lo | (hi << 16);
                asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h2) : "r"(h2), "r"(0x64806480u));
                w[i] = h2;
            }
            *reinterpret_cast<uint4 *>(pool + ((bk.piece0 + (int64_t)(kb * S + s) * bk.rows + r) * BK + q * 8)) =
                make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// --------------------------------------------------------------------- product tiles
__device__ __forceinline__ void red_sub(double *p, double a) {
    asm volatile("red.relaxed.gpu.global.add.f64 [%0], %1;" ::"l"(p), "d"(-a) : "memory");
}

__global__ void __launch_bounds__(kThreads, 1)
    k_split_gemm(double *__restrict__ lnz, double *__restrict__ upool, const Task *__restrict__ tasks,
                 const GemmTile *__restrict__ tiles, int ntiles, const int32_t *__restrict__ blk_of_task,
                 const SplitBlk *__restrict__ blks, const int32_t *__restrict__ exps,
                 const CUtensorMap *__restrict__ maps /* 128-row box, 64-row box */, int32_t *__restrict__ err,
                 long long spin_limit) {
    using namespace tc;
    extern __shared__ __align__(1024) unsigned char sp_smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)sp_smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES);
    uint64_t *full = bars, *empty = bars + STAGES, *accf = bars + 2 * STAGES, *acce = bars + 2 * STAGES + 1;
    uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + 2 * STAGES + 2);
    __shared__ volatile int abort_flag;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    if (threadIdx.x == 0) {
        abort_flag = 0;
        for (int s = 0; s < STAGES; s++) mbar_init(smem_u32(full + s), 1), mbar_init(smem_u32(empty + s), 1);
        mbar_init(smem_u32(accf), 1);
        mbar_init(smem_u32(acce), kEpiWarps);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                     "r"(S * BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_holder;

    if (warp == 0) {
        if (lane == 0) {
            // producer
            uint32_t g = 0;
            for (int t = blockIdx.x; t < ntiles && !abort_flag; t += gridDim.x) {
                const GemmTile tl = tiles[t];
                const Task tk = tasks[tl.task];
                const SplitBlk bk = blks[blk_of_task[tl.task]];
                const int nk = (tk.k + BK - 1) / BK;
                const int64_t ay = bk.piece0 + (tk.a_row - bk.row0) + tl.tm * BM;
                const int64_t by = bk.piece0 + (tk.b_row - bk.row0) + tl.tn * BN;
                for (int kb = 0; kb < nk; kb++, g++) {
                    const int s = g % STAGES;
                    if (g >= STAGES && !mbar_wait(smem_u32(empty + s), ((g / STAGES) & 1u) ^ 1u, spin_limit, err, 11)) {
                        abort_flag = 1;
                        break;
                    }
                    const uint32_t fb = smem_u32(full + s);
                    mbar_expect_tx(fb, STAGE_BYTES);
                    const uint32_t a0 = smem_u32(smem + s * STAGE_BYTES), b0 = a0 + S * A_BYTES;
                    for (int i = 0; i < S; i++) {
                        const int64_t off = (int64_t)(kb * S + i) * bk.rows;
                        tma_load_2d(a0 + i * A_BYTES, maps, 0, (int)(ay + off), fb);
                        tma_load_2d(b0 + i * B_BYTES, maps + 1, 0, (int)(by + off), fb);
                    }
                }
            }
            // the copies in flight (all of them have landed unless a wait ran out)
            for (uint32_t u = g > (uint32_t)STAGES ? g - STAGES : 0; u < g; u++)
                if (!mbar_wait(smem_u32(full + u % STAGES), (u / STAGES) & 1u, spin_limit, err, 15)) break;
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // MMA issuer
            uint32_t g = 0, drains = 0;
            for (int t = blockIdx.x; t < ntiles && !abort_flag; t += gridDim.x) {
                const GemmTile tl = tiles[t];
                const Task tk = tasks[tl.task];
                const int nk = (tk.k + BK - 1) / BK;
                for (int kb = 0; kb < nk; kb++, g++) {
                    const bool first = kb % kDrain == 0;
                    if (first && drains > 0 && !mbar_wait(smem_u32(acce), (drains - 1) & 1u, spin_limit, err, 12)) {
                        abort_flag = 1;
                        break;
                    }
                    const int s = g % STAGES;
                    if (!mbar_wait(smem_u32(full + s), (g / STAGES) & 1u, spin_limit, err, 13)) {
                        abort_flag = 1;
                        break;
                    }
                    fence_after();
                    const uint32_t a0 = smem_u32(smem + s * STAGE_BYTES), b0 = a0 + S * A_BYTES;
                    const int ksteps = min(BK / 16, (tk.k - kb * BK + 15) / 16);
                    for (int kk = 0; kk < ksteps; kk++) {  // 16 FP16 = 32 bytes along K inside the swizzle row
                        const uint64_t ad = umma_desc_sw64(a0 + kk * 32), bd = umma_desc_sw64(b0 + kk * 32);
                        // slice i of A times the slices j .. j + 3 of B at once: B's slices lie one
                        // after another, and so do the groups i + j that the products go to
#pragma unroll
                        for (int i = 0; i < S; i++)
#pragma unroll
                            for (int j = 0; j < S - i; j += 4)
                                mma_f16(tmem + (i + j) * BN, ad + (uint64_t)(i * (A_BYTES >> 4)),
                                        bd + (uint64_t)(j * (B_BYTES >> 4)), idesc_f16(BN * (S - i - j < 4 ? S - i - j : 4)),
                                        (first && kk == 0 && i == 0) ? 0u : 1u);
                    }
                    mma_commit(smem_u32(empty + s));
                    if (kb == nk - 1 || kb % kDrain == kDrain - 1) {
                        mma_commit(smem_u32(accf));
                        drains++;
                    }
                }
            }
            // the products in flight
            for (uint32_t u = g > (uint32_t)STAGES ? g - STAGES : 0; u < g; u++)
                if (!mbar_wait(smem_u32(empty + u % STAGES), (u / STAGES) & 1u, spin_limit, err, 16)) break;
        }
    } else if (warp >= 4) {
        // epilogue warps 4..19: TMEM lanes 32 (warp % 4) .. + 31, columns 16 (warp / 4 - 1) .. + 15.
        // Lane l holds rows l / 4 + 8 h (h < 4) and columns l % 4 + 4 q (q < 4).
        const int quarter = warp % 4, c0 = (warp / 4 - 1) * 16;
        const int lr = lane / 4, lc = lane % 4;
        uint32_t drains = 0;
        bool ok = true;
        for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
            // the task's fields are read again after the drains: they would only hold registers
            const GemmTile tl = tiles[t];
            const Task &tk = tasks[tl.task];
            const bool lower = tk.flags & kTaskLower;
            // does this warp's 32 x 16 part hold any entry that is written?
            const int wr = tl.tm * BM + quarter * 32, wc = tl.tn * BN + c0;
            const bool active = wr < tk.m && wc < tk.n && !(lower && min(wr + 31, tk.m - 1) < wc);
            const int nk = (tk.k + BK - 1) / BK, nd = (nk + kDrain - 1) / kDrain;
            Acc96 acc[4][4];
#pragma unroll
            for (int h = 0; h < 4; h++)
#pragma unroll
                for (int q = 0; q < 4; q++) acc[h][q].t = 0, acc[h][q].r = 0;
            for (int d = 0; d < nd; d++, drains++) {
                ok = mbar_wait(smem_u32(accf), drains & 1u, spin_limit, err, 14);
                ok = __all_sync(0xffffffffu, ok && !abort_flag);
                if (!ok) break;
                fence_after();
                if (active) {
#pragma unroll
                    for (int part = 0; part < 8; part++) {
                        // 16 rows, 8 columns, four groups at a time
                        const int hh = part / 4, qq = part / 2 % 2, half = part % 2;
                        uint32_t v[4][4];
#pragma unroll
                        for (int s = 0; s < 4; s++)
                            tmem_ld_16x8(tmem + ((uint32_t)(quarter * 32 + hh * 16) << 16) +
                                             (uint32_t)((half * 4 + s) * BN + c0 + qq * 8),
                                         v[s]);
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                        for (int e = 0; e < 4; e++) {
                            Acc96 &a = acc[hh * 2 + (e & 1)][qq * 2 + (e >> 1)];
                            if (half == 0) acc_add_high(a, v[0][e], v[1][e], v[2][e], v[3][e]);
                            else acc_add_low(a, v[0][e], v[1][e], v[2][e], v[3][e]);
                        }
                    }
                }
                fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(acce));
            }
            if (!ok || !active) continue;
            const SplitBlk &bk = blks[blk_of_task[tl.task]];
            const int32_t *ex = exps + bk.exp0 - bk.row0;
            const int gi0 = wr + lr, gj0 = wc + lc;
            const int flags = tk.flags, m = tk.m, n = tk.n;
            const bool excl = flags & kTaskExclusive, store = flags & kTaskStoreU;
            double *C = (store ? upool : lnz) + tk.c_off;
            int ebj[4];
#pragma unroll
            for (int q = 0; q < 4; q++) ebj[q] = gj0 + 4 * q < n ? ex[tk.b_row + gj0 + 4 * q] : 0;
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int gi = gi0 + 8 * h;
                if (gi >= m) continue;
                const int eai = ex[tk.a_row + gi];
                double *crow = C + (int64_t)gi * tk.ldc;
                double old[4];
                if (excl) {
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const int gj = gj0 + 4 * q;
                        old[q] = gj < n && (!(flags & kTaskLower) || gj <= gi) ? crow[gj] : 0.0;
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const int gj = gj0 + 4 * q;
                    if (gj >= n || ((flags & kTaskLower) && gj > gi)) continue;
                    double v = acc_value(acc[h][q], eai + ebj[q]);
                    if (eai == kBadExp || ebj[q] == kBadExp) v = __longlong_as_double(0x7ff8000000000000ll);
                    if (store) crow[gj] = -v;
                    else if (excl) crow[gj] = old[q] - v;
                    else red_sub(crow + gj, v);
                }
            }
        }
    }
    __syncwarp();
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S * BN) : "memory");
}

}  // namespace sp

// ---------------------------------------------------------------- host side
inline bool split_gemm_init() {
    return cudaFuncSetAttribute(sp::k_split_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, sp::SMEM) == cudaSuccess;
}

inline void split_tiles_of(const Task &t, int32_t id, std::vector<GemmTile> &out) {
    const int tm = (t.m + sp::BM - 1) / sp::BM, tn = (t.n + sp::BN - 1) / sp::BN;
    for (int i = 0; i < tm; i++)
        for (int j = 0; j < tn; j++) {
            if ((t.flags & kTaskLower) && (i * sp::BM + sp::BM - 1) < j * sp::BN) continue;  // above the diagonal
            out.push_back(GemmTile{id, i, j, -1});
        }
}

// Tensor maps of the slice pool (rows of 32 FP16): boxes of 128 and of 64 rows.
inline int split_encode_maps(uint16_t *pool, int64_t pieces, std::vector<CUtensorMap> &maps) {
    PFN_cuTensorMapEncodeTiled_v12000 encode = tc_map_encoder();
    if (!encode) return SC_ERR_CUDA;
    maps.clear();
    for (int rows : {sp::BM, sp::BN}) {
        CUtensorMap map;
        cuuint64_t dims[2] = {(cuuint64_t)sp::BK, (cuuint64_t)pieces};
        cuuint64_t strides[1] = {(cuuint64_t)sp::BK * 2};
        cuuint32_t box[2] = {(cuuint32_t)sp::BK, (cuuint32_t)rows};
        cuuint32_t estr[2] = {1, 1};
        if (encode(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (void *)pool, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return SC_ERR_CUDA;
        maps.push_back(map);
    }
    return SC_OK;
}

inline void launch_split(const double *lnz, const SplitBlk *blks, const SplitUnit *units, int32_t count, uint16_t *pool,
                         int32_t *exps, cudaStream_t st) {
    sp::k_split<<<count, 256, 0, st>>>(lnz, blks, units, pool, exps);
}
inline void launch_split_gemm(double *lnz, double *upool, const Task *tasks, const GemmTile *tiles, int32_t count,
                              const int32_t *blk_of_task, const SplitBlk *blks, const int32_t *exps,
                              const CUtensorMap *maps, int32_t *err, long long spin_limit, int num_sms,
                              cudaStream_t st) {
    sp::k_split_gemm<<<std::min<int>(count, num_sms), sp::kThreads, sp::SMEM, st>>>(
        lnz, upool, tasks, tiles, count, blk_of_task, blks, exps, maps, err, spin_limit);
}

}  // namespace sc

