// Numeric factorization of libsc on the GPU: builds the per-level launch plan
// from the host schedule, owns the device memory of a numeric handle, and
// runs the level sequence (Alg. 5 RLB or Alg. 4 RL, made level-parallel),
// replayed as one CUDA graph.
#include <algorithm>
#include <cstring>

#include "kernels.cuh"
#include "numeric.h"
#include "split_gemm.cuh"
#include "chunk64.cuh"
#include "loops64.cuh"
#include "sweep64.cuh"
#include "tc_gemm.cuh"

namespace sc {

#define SC_CUDA(x)                                  \
    do {                                            \
        cudaError_t e_ = (x);                       \
        if (e_ != cudaSuccess) return SC_ERR_CUDA;  \
    } while (0)

namespace {

constexpr int kBM = 64, kBN = 64, kBK = 16;

// diagonal of the input matrix in the final ordering: adiag[k] = A(perm[k], perm[k])
__global__ void k_diag(double *__restrict__ adiag, const int64_t *__restrict__ diag_pos,
                       const double *__restrict__ values, int64_t n) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) adiag[i] = values[diag_pos[i]];
}


template <typename U>
int upload(U *&dst, const std::vector<U> &src, int64_t &bytes) {
    size_t b = std::max<size_t>(1, src.size()) * sizeof(U);
    if (cudaMalloc((void **)&dst, b) != cudaSuccess) return SC_ERR_OOM;
    bytes += (int64_t)b;
    if (!src.empty() && cudaMemcpy(dst, src.data(), src.size() * sizeof(U), cudaMemcpyHostToDevice) != cudaSuccess)
        return SC_ERR_CUDA;
    return SC_OK;
}

bool is_small(const Task &t) { return (int64_t)t.m * t.n <= 64; }

// algorithmic flops of a product task: 2 k per entry written
double task_flops(const Task &t) {
    double e = (t.flags & kTaskLower) ? (double)t.n * (t.n + 1) / 2 + (double)(t.m - t.n) * t.n : (double)t.m * t.n;
    return 2.0 * e * t.k;
}

void tiles_of(const Task &t, int32_t id, std::vector<GemmTile> &out, bool no_split) {
    int tm = (t.m + kBM - 1) / kBM, tn = (t.n + kBN - 1) / kBN;
    // a task of few tiles with a long inner dimension is split along it, so its
    // tiles do not serialise a level; a critical task (the next level waits for
    // it) is split into slices of kSplitKCrit so its latency is short (an RL
    // update matrix is stored, not added: never split; nor is anything in a
    // deterministic plan, where the slices' atomic adds would land in any order)
    int slices = 0;
    if (!(t.flags & kTaskStoreU) && !no_split) {
        if ((t.flags & kTaskCrit) && t.k >= 2 * kSplitKCrit) slices = (t.k + kSplitKCrit - 1) / kSplitKCrit;
        else if (tm * tn <= 8 && t.k > 2 * kSplitK) slices = (t.k + kSplitK - 1) / kSplitK;
    }
    for (int i = 0; i < tm; i++)
        for (int j = 0; j < tn; j++) {
            if ((t.flags & kTaskLower) && (i * kBM + kBM - 1) < j * kBN) continue;  // above the diagonal
            if (!slices) out.push_back(GemmTile{id, i, j, -1});
            for (int q = 0; q < slices; q++) out.push_back(GemmTile{id, i, j, q});
        }
}

// FP32 inverses of the factored diagonal blocks of all chunks, for the solve
// sweeps of FP32 / TF32 factors (one launch after the last level, off the
// factorization's critical path).
__global__ void __launch_bounds__(256) k_inverse(const float *__restrict__ lnz, const ChunkDev *__restrict__ chunks,
                                                 const int32_t *__restrict__ list, float *__restrict__ inv) {
    extern __shared__ double smem_potrf[];
    const ChunkDev ch = chunks[list[blockIdx.x]];
    auto a = reinterpret_cast<float (*)[kMaxChunk + 1]>(smem_potrf);
    auto iv = a + kMaxChunk;
    load_block(a, lnz + ch.off + (int64_t)ch.c0 * ch.ld + ch.c0, ch.ld, ch.w);
    __syncthreads();
    tri_inverse<float>(a, ch.w, iv, inv + ch.inv);
}


// Inverses of the factored diagonal blocks of the chunks wider than kNarrowChunk, for
// the solve sweeps of FP64 factors: L_cc in 16 x 16 blocks; the diagonal ones W_ii by
// substitution (a warp each, a lane per column), then W_ij = -W_ii sum_{j <= k < i} L_ik W_kj
// by digits (fx.cuh) on mma.sync. A warp takes eight columns of W through all the block rows,
// so nothing but the digits of L and the W_ii passes between warps. An operand has an
// exponent per row or column of a 16-column panel; in W_ii S the inner index also carries
// the scale 2^{c_k}, the size of L_kk, as in chunk64.cuh. Stored as the digits of W's rows (columns
// times 2^{c_k}: where W is multiplied, its columns' scales
// cancel against those of the other operand, also for D A D), the rows' exponents
// and minus the columns'. With the products on the FP64 pipe a block took an SM
// some 41,000 clocks, 33,000 of them these products; by digits the 48^3 FP64 step takes 18.01
// instead of 18.12 ms, the 83 x 71 RL factor 0.670 instead of 0.681. What is left is the
// substitution (136 multiply-adds of a warp, 64 clocks each) and the launch.
//
// W rounded to FP64 would cost the sweeps' y = W x a residual of || |W| |L| || u = kappa u. The digits
// have nine bits more: R = I - L W is formed by digits (exact sums, the identity subtracted
// from the whole numbers), and W R in FP32 is added to the digits of W. The solution's backward
// error then is that of substitution up to kappa of some 2000 (sweep64.cuh); chunks above kFixChunk
// are marked in fix.
constexpr int kInv64Smem = 8 * (2 * 64 * fx::kLd + kMaxChunk * (kMaxChunk + 1));
__global__ void __launch_bounds__(256, 2) k_inverse64(const double *__restrict__ lnz, const ChunkDev *__restrict__ chunks,
                                                      const int32_t *__restrict__ list, uint64_t *__restrict__ inv,
                                                      int32_t *__restrict__ inv_exp, int32_t *__restrict__ inv_cexp,
                                                      int32_t *__restrict__ fix) {
    extern __shared__ __align__(16) unsigned char smem_inv64[];  // read 16 bytes at a time
    __shared__ double rinv[kMaxChunk];
    __shared__ int32_t e_c[kMaxChunk], e_l[kMaxChunk], e_d[kMaxChunk], e_v[4][kMaxChunk];
    __shared__ float size_l[kMaxChunk];  // row sums of |L| over the rows' sizes
    __shared__ int kappa;                // as FP32 bits (not negative, so they compare as whole numbers)
    const ChunkDev ch = chunks[list[blockIdx.x]];
    const int w = ch.w, nbk = (w + 15) / 16;
    // T: digits of L's rows left of the diagonal blocks, and of the W_ii there; V: digits of
    // the columns of W (and of S), in the place of L's values, which are only read before
    uint64_t *T = reinterpret_cast<uint64_t *>(smem_inv64), *V = T + 64 * fx::kLd;
    auto l = reinterpret_cast<double (*)[kMaxChunk + 1]>(V);
    auto v = reinterpret_cast<double (*)[kMaxChunk + 1]>(V + 64 * fx::kLd);
    auto put = [](double x, int key, int e) {
        return key == fx::kKeyBad ? 0x8080808080808080ull : fx::split_bytes(x, key - 1022 - e);
    };
    auto quad_max = [](int k) {
        k = max(k, __shfl_xor_sync(0xffffffffu, k, 1));
        return max(k, __shfl_xor_sync(0xffffffffu, k, 2));
    };
    auto quad_sum = [](float x) {
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        return x + __shfl_xor_sync(0xffffffffu, x, 2);
    };
    load_block(l, lnz + ch.off + (int64_t)ch.c0 * ch.ld + ch.c0, ch.ld, w);
    __syncthreads();
    if (threadIdx.x < kMaxChunk) {
        const double lk = l[threadIdx.x][threadIdx.x];
        rinv[threadIdx.x] = threadIdx.x < w ? 1.0 / lk : 0.0;
        e_c[threadIdx.x] = (int)threadIdx.x < w ? ((__double2hiint(lk) >> 20) & 0x7ff) - 1023 : 0;
    }
    // four threads per row: columns q, q + 4, ...
    const int r = threadIdx.x / 4, q = threadIdx.x % 4, ob = r / 16 * 16;
    {
        int key = fx::kKeyNone;
        for (int c = q; c < ob; c += 4) key = max(key, fx::exp_key(l[r][c], 0));
        key = quad_max(key);
        for (int c = q; c < ob; c += 4) T[r * fx::kLd + c] = put(l[r][c], key, 0);
        const int er = r < w ? 1023 - ((__double2hiint(l[r][r]) >> 20) & 0x7ff) : 0;
        float sum = 0.f;
        for (int c = q; c <= r; c += 4) sum += fx::size_of(l[r][c], er);
        sum = quad_sum(sum);
        if (q == 0) {
            e_l[r] = fx::key_exp(key);
            size_l[r] = sum;
        }
        if (threadIdx.x == 0) kappa = 0;
    }
    __syncthreads();
    if ((int)threadIdx.x / 32 < nbk && threadIdx.x % 32 < 16) {
        const int o = threadIdx.x / 32 * 16, j = threadIdx.x % 32;
        double x[16];
#pragma unroll
        for (int i = 0; i < 16; i++) {
            double s = i == j ? 1.0 : 0.0;
#pragma unroll
            for (int t = 0; t < i; t++) s -= l[o + i][o + t] * x[t];
            x[i] = s * rinv[o + i];
        }
#pragma unroll
        for (int i = 0; i < 16; i++) v[o + i][o + j] = i >= j ? x[i] : 0.0;
    }
    __syncthreads();
    if (ob < 16 * nbk) {
        // digits of the W_ii: rows (for W_ii S) and columns (for L_ki W_ii)
        int kd = fx::kKeyNone, kv = fx::kKeyNone;
#pragma unroll
        for (int t = ob + q; t < ob + 16; t += 4) {
            kd = max(kd, fx::exp_key(v[r][t], e_c[t]));
            kv = max(kv, fx::exp_key(v[t][r], 0));
        }
        kd = quad_max(kd);
        kv = quad_max(kv);
#pragma unroll
        for (int t = ob + q; t < ob + 16; t += 4) {
            T[r * fx::kLd + t] = put(v[r][t], kd, e_c[t]);
            V[r * fx::kLd + t] = put(v[t][r], kv, 0);
        }
        if (q == 0) {
            e_d[r] = fx::key_exp(kd);
            e_v[ob / 16][r] = fx::key_exp(kv);
        }
    }
    __syncthreads();
    // columns n0 .. n0 + 7 of W by this warp, block row by block row (lane: rows r0 and r0 + 8,
    // columns nc and nc + 1 of a product)
    const int lane = threadIdx.x % 32, n0 = threadIdx.x / 32 * 8, jb = n0 / 16, nc = n0 + 2 * (lane % 4);
#pragma unroll 1
    for (int i = jb + 1; i < nbk; i++) {
        const int r0 = 16 * i + lane / 4;
        float acc[fx::S][4];
        double x[4] = {0.0, 0.0, 0.0, 0.0};
        int k[2];  // exponent keys of the columns nc, nc + 1
        // digits of x, its rows times 2^{f0}, 2^{f1}, as columns of V
        auto put_columns = [&](int f0, int f1) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                k[h] = max(fx::exp_key(x[h], f0), fx::exp_key(x[2 + h], f1));
#pragma unroll
                for (int o = 4; o < 32; o *= 2) k[h] = max(k[h], __shfl_xor_sync(0xffffffffu, k[h], o));
                V[(nc + h) * fx::kLd + r0] = put(x[h], k[h], f0);
                V[(nc + h) * fx::kLd + r0 + 8] = put(x[2 + h], k[h], f1);
            }
            __syncwarp();
        };
        // S = sum_k L_ik W_kj
#pragma unroll 1
        for (int p = jb; p < i; p++) {
            fx::product<false>(T, V, i, n0, p, p + 1, acc);
#pragma unroll
            for (int e = 0; e < 4; e++) x[e] += fx::block_value(acc, e, e_l[r0 + 8 * (e / 2)], e_v[p][nc + e % 2]);
        }
        put_columns(-e_c[r0], -e_c[r0 + 8]);
        fx::product<false>(T, V, i, n0, i, i + 1, acc);
#pragma unroll
        for (int e = 0; e < 4; e++) {
            x[e] = -fx::block_value(acc, e, e_d[r0 + 8 * (e / 2)], fx::key_exp(k[e % 2]));
            v[r0 + 8 * (e / 2)][nc + e % 2] = x[e];
        }
        __syncwarp();  // S's digits have been read
        put_columns(0, 0);
        if (lane < 4) {
            e_v[i][nc] = fx::key_exp(k[0]);
            e_v[i][nc + 1] = fx::key_exp(k[1]);
        }
        __syncwarp();
    }
    __syncthreads();
    // R = I - L W, columns as above: L's rows and W's columns with one exponent each, so the
    // sums over all of the inner index are exact
    fx::stage_tile<true>(T, e_l, lnz + ch.off + (int64_t)ch.c0 * ch.ld + ch.c0, ch.ld, w, w);
    {
        int key = fx::kKeyNone;
        for (int t = r + q; t < w; t += 4) key = max(key, fx::exp_key(v[t][r], 0));
        key = quad_max(key);
        for (int t = q; t < kMaxChunk; t += 4)
            V[r * fx::kLd + t] = t >= r && t < w ? put(v[t][r], key, 0) : 0x8080808080808080ull;
        if (q == 0) e_v[0][r] = fx::key_exp(key);
    }
    __syncthreads();
    {
        float res[4][4];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            if (i < jb || i >= nbk) continue;
            float acc[fx::S][4];
            fx::product<false>(T, V, i, n0, jb, i + 1, acc);
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const int row = 16 * i + lane / 4 + 8 * (e / 2), col = nc + e % 2, E = e_l[row] + e_v[0][col];
                fx::Acc96 a{0, 0};
                fx::acc_add64(a, acc, e);
                if (row == col && row < w) fx::acc_sub_one(a, E);
                res[i][e] = -(float)fx::acc_value(a, E - e_c[row] + e_c[col]);
            }
        }
        __syncwarp();  // V's rows n0 .. + 7 are this warp's alone: R's columns take their place
#pragma unroll
        for (int i = 0; i < 4; i++) {
            if (i < jb || i >= nbk) continue;
#pragma unroll
            for (int e = 0; e < 4; e++)
                reinterpret_cast<float *>(V + (nc + e % 2) * fx::kLd)[16 * i + lane / 4 + 8 * (e / 2)] = res[i][e];
        }
    }
    __syncthreads();
    // W, columns times 2^{c_k}, in the place of L's digits; kappa
    float *wf = reinterpret_cast<float *>(T) + r * (kMaxChunk + 1);
    int key = fx::kKeyNone;
    float sum = 0.f;
    for (int c = q; c < kMaxChunk; c += 4) {
        const double x = c <= r && r < w ? v[r][c] : 0.0;
        const float f = fx::size_of(x, e_c[c]);
        wf[c] = __double2hiint(x) < 0 ? -f : f;
        sum += f * size_l[c];
        if (c <= r) key = max(key, fx::exp_key(x, e_c[c]));
    }
    key = quad_max(key);
    sum = quad_sum(sum);
    if (q == 0) atomicMax(&kappa, __float_as_int(sum));
    __syncthreads();
    if (threadIdx.x == 0) fix[list[blockIdx.x]] = !(__int_as_float(kappa) <= kFixChunk);
    if (r >= w) return;
    // W R, columns q, q + 4, ...
    float dw[kMaxChunk / 4];
#pragma unroll
    for (int m = 0; m < kMaxChunk / 4; m++) dw[m] = 0.f;
#pragma unroll
    for (int b = 0; b < 4; b++) {
        if (16 * b > r) break;
#pragma unroll 4
        for (int t = 16 * b; t < 16 * b + 16; t++) {
            const float x = wf[t];
#pragma unroll
            for (int m = 0; m < 4 * b + 4; m++) dw[m] += x * reinterpret_cast<const float *>(V + (q + 4 * m) * fx::kLd)[t];
        }
    }
    // digits of the rows of W + W R (the second term where it is the smaller by 2^8 and more)
    const int E = key - 1022;
    const float scale = __int_as_float(min(max(127 + 62 - E, 1), 254) << 23);
#pragma unroll
    for (int m = 0; m < kMaxChunk / 4; m++) {
        const int c = q + 4 * m;
        if (c >= w) continue;
        const float d = dw[m] * scale;
        const int64_t add = c <= r && fabsf(d) < 0x1p54f && key != fx::kKeyBad ? __float2ll_rn(d) : 0;
        inv[ch.inv + r * w + c] = c > r ? 0x8080808080808080ull : put(v[r][c], key, e_c[c]) + (uint64_t)add;
    }
    if (q == 0) {
        inv_exp[ch.col0 + r] = fx::key_exp(key);
        inv_cexp[ch.col0 + r] = -e_c[r];
    }
}

// ---- one persistent launch per level (SIMT precisions, RLB)
// Bounded wait until *flag >= target (acquire at GPU scope); gives up, setting
// *err, after spin_limit polls or once another CTA has given up.
__device__ bool flow_wait(const int32_t *flag, int32_t target, int32_t *err, long long spin_limit, int code) {
    for (long long i = 0; i < spin_limit; i++) {
        int32_t v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
        if (v >= target) return true;
        if (*(volatile int32_t *)err) return false;
        if (i > 64) __nanosleep(64);
    }
    atomicCAS(err, 0, code);
    return false;
}

template <typename T>
struct LevelArgs {
    T *lnz, *pool;
    const ChunkDev *chunks;
    const TrsmTile *trsm;
    const GemmTile *gemm;
    const Task *tasks;
    const ThinUnit *thin;
    const int32_t *small;
    const LoopItem *loops;
    const SnDev *sn;
    const BlkDev *blk;
    const int32_t *rbval;
    const double *adiag;
    int32_t *info, *low_pivots;
    double tau;
    const FlowUnit *units;
    int32_t nunits;
    int32_t *ctr;             // per chunk (kFlowStride apart): POTRF and TRSM units done
    const int32_t *need;      // per chunk: 1 + its TRSM tiles
    const int32_t *task_chunk;
    const int32_t *sn_chunk;
    int32_t *work;            // this launch's unit counter
    int32_t *err;
    long long spin_limit;
};

// All work of one level in one launch: CTAs take units in list order (POTRF of
// the level's chunks, their TRSM tiles, the previous level's lookahead
// products, this level's products, small tasks and device loops). A TRSM tile
// waits for its chunk's POTRF; a product, small task or loop item waits until
// the chunk it reads is factored (POTRF and every TRSM tile). Every wait is
// for a unit earlier in the list, taken by a running CTA, so the launch needs
// no co-residency; every wait is bounded (then *err is set and the CTAs stop).
// Product writes are atomic: units of one launch may update the same target.
template <typename T>
__global__ void __launch_bounds__(256, 2) k_level(LevelArgs<T> a) {
    __shared__ int s_u, s_ok;
    for (;;) {
        if (threadIdx.x == 0) s_u = *(volatile int32_t *)a.err ? a.nunits : atomicAdd(a.work, 1);
        __syncthreads();
        const int u = s_u;
        if (u >= a.nunits) break;
        const FlowUnit fu = a.units[u];
        // dependencies, checked by thread 0
        if (threadIdx.x == 0) {
            bool ok = true;
            auto src = [&](int32_t c) {
                if (ok) ok = flow_wait(a.ctr + (int64_t)c * kFlowStride, a.need[c], a.err, a.spin_limit, 9);
            };
            switch (fu.kind) {
                case kFlowTrsm:
                    ok = flow_wait(a.ctr + (int64_t)a.trsm[fu.idx].chunk * kFlowStride, 1, a.err, a.spin_limit, 9);
                    break;
                case kFlowGemm: src(a.task_chunk[a.gemm[fu.idx].task]); break;
                case kFlowThin:
                    for (int q = 0; q < fu.cnt; q++) src(a.task_chunk[a.thin[fu.idx + q].task]);
                    break;
                case kFlowSmall:
                    for (int q = 0; q < fu.cnt; q++) src(a.task_chunk[a.small[fu.idx + q]]);
                    break;
                case kFlowLoop: src(a.sn_chunk[a.loops[fu.idx].sn]); break;
                case kFlowLoopW:
                    for (int q = 0; q < fu.cnt; q++) src(a.sn_chunk[a.loops[fu.idx + q].sn]);
                    break;
                default: break;
            }
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) break;
        switch (fu.kind) {
            case kFlowPotrf:
                potrf_chunk<T>(a.lnz, a.chunks, fu.idx, a.adiag, a.info, a.low_pivots, a.tau, nullptr, nullptr);
                break;
            case kFlowTrsm: trsm_tile<T>(a.lnz, a.chunks, a.trsm[fu.idx], nullptr, nullptr); break;
            case kFlowGemm: gemm_tile<T, 64, 64, 16>(a.lnz, a.pool, a.tasks, a.gemm[fu.idx], true); break;
            case kFlowThin: {
                const int wq = threadIdx.x / 32 / kThinWarps;
                if (wq < fu.cnt) thin_warp<T>(a.lnz, a.tasks, a.thin[fu.idx + wq], (threadIdx.x / 32) % kThinWarps);
                break;
            }
            case kFlowSmall: small_tasks<T>(a.lnz, a.pool, a.tasks, a.small + fu.idx, fu.cnt, 0); break;
            case kFlowLoop: loop_item<T>(a.lnz, a.loops[fu.idx], a.sn, a.blk, a.rbval); break;
            case kFlowLoopW: loop_items_warp<T>(a.lnz, a.loops + fu.idx, fu.cnt, 0, a.sn, a.blk, a.rbval); break;
            default: break;
        }
        if (fu.kind == kFlowPotrf || fu.kind == kFlowTrsm) {
            // release: the barrier orders the CTA's stores before thread 0's fence
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                const int32_t c = fu.kind == kFlowPotrf ? fu.idx : a.trsm[fu.idx].chunk;
                atomicAdd(a.ctr + (int64_t)c * kFlowStride, 1);
            }
        }
        __syncthreads();
    }
}

// Optional per-kernel-class timing of one factorization (CUDA events around
// every launch; only used outside graph capture).
struct Prof {
    cudaStream_t st = nullptr;
    std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> ev;
    int cur = -1;
    void begin(int cls) {
        cudaEvent_t a, b;
        cudaEventCreate(&a);
        cudaEventCreate(&b);
        cudaEventRecord(a, st);
        ev.push_back({cls, {a, b}});
    }
    void end() { cudaEventRecord(ev.back().second.second, st); }
};

template <typename T>
// st2 (optional, graph capture only): a second stream on which each level's
// device RLB loops run concurrently with the level's tiled products.
int run_levels(sc_numeric *h, cudaStream_t st, Prof *prof = nullptr, cudaStream_t st2 = nullptr,
               cudaStream_t st3 = nullptr) {
    const sc_symbolic *s = h->sym;
    auto B = [&](int cls) {
        if (prof) prof->begin(cls);
    };
    auto E = [&]() {
        if (prof) prof->end();
    };
    T *lnz = (T *)h->d_lnz;
    T *pool = (T *)h->d_pool;
    int launches = 0;
    B(kProfK0);
    SC_CUDA(cudaMemsetAsync(h->d_lnz, 0, (size_t)s->lnz_size * sizeof(T), st));
    SC_CUDA(cudaMemsetAsync(h->d_info, 0x7f, sizeof(int32_t), st));
    SC_CUDA(cudaMemsetAsync(h->d_info + 1, 0, sizeof(int32_t), st));
    SC_CUDA(cudaMemsetAsync(h->d_err, 0, sizeof(int32_t), st));
    int64_t nnz = (int64_t)s->valmap.size();
    k_diag<<<(unsigned)((s->n + 255) / 256), 256, 0, st>>>(h->d_adiag, h->d_diagpos, h->d_values, s->n);
    k_scatter_values<T><<<(unsigned)std::min<int64_t>((nnz + 255) / 256, 152 * 16), 256, 0, st>>>(
        lnz, h->d_valmap, h->d_values, nnz);
    E();
    launches += 2;
    const double tau = s->opt.pivot_tau;
    // diagonal-block inverses for the solve, all chunks but k_narrow's in one launch
    auto launch_inverses = [&]() {
        const int32_t nch = sizeof(T) == 8 && h->fused ? 0 : h->inv_cnt;  // (FP64 operations only: substitution)
        const int32_t *list = h->d_potrf + h->inv_off;
        if (!nch) return;
        B(kProfPotrf);
        if constexpr (sizeof(T) == 4)
            k_inverse<<<nch, 256, kPotrfSmem, st>>>((const float *)lnz, h->d_chunks, list, (float *)h->d_inv);
        else
            k_inverse64<<<nch, 256, kInv64Smem, st>>>((const double *)lnz, h->d_chunks, list, (uint64_t *)h->d_inv,
                                                      h->d_inv_exp, h->d_inv_exp + s->n, h->d_inv_exp + 2 * s->n);
        E();
        launches++;
    };
    if (h->fused && !prof) {
        // one persistent launch per level, then the tail of lookahead products
        const size_t nch = s->chunks.size(), nlev = h->plans.size();
        SC_CUDA(cudaMemsetAsync(h->d_flow_ctr, 0, (nch * kFlowStride + nlev + 1) * sizeof(int32_t), st));
        LevelArgs<T> a{lnz, pool, h->d_chunks, h->d_trsm, h->d_gemm, h->d_tasks, h->d_thin, h->d_small, h->d_loops,
                       h->d_sn, h->d_blk, h->d_rbval, h->d_adiag, h->d_info, h->d_info + 1, tau, nullptr, 0,
                       h->d_flow_ctr, h->d_flow_need, h->d_task_chunk, h->d_sn_chunk, nullptr, h->d_err,
                       (long long)s->opt.spin_limit};
        int32_t *work = h->d_flow_ctr + nch * kFlowStride;
        for (size_t lv = 0; lv <= nlev; lv++) {
            const int32_t off = lv < nlev ? h->plans[lv].flow_off : h->flow_tail_off;
            const int32_t cnt = lv < nlev ? h->plans[lv].flow_cnt : h->flow_tail_cnt;
            if (!cnt) continue;
            a.units = h->d_flow + off;
            a.nunits = cnt;
            a.work = work + lv;
            const int grid = std::max(1, std::min(cnt, 2 * h->num_sms));
            k_level<T><<<grid, 256, kPotrfSmem, st>>>(a);
            launches++;
        }
        launch_inverses();
        SC_CUDA(cudaGetLastError());
        h->kernel_launches = launches;
        return SC_OK;
    }
    // tiled products of one dependency class on stream ps
    auto digit_products = [&](int32_t off, int32_t cnt, cudaStream_t ps) {
        if (h->d_slices)
            launch_split_gemm((double *)lnz, (double *)pool, h->d_tasks, h->d_gemm + off, cnt, h->d_split_of_task,
                              h->d_splits, h->d_exps, h->d_slice_maps, h->d_err, (long long)s->opt.spin_limit,
                              h->num_sms, ps);
        else
            k_digit_tiles<<<cnt, 256, 0, ps>>>((double *)lnz, (double *)pool, h->d_tasks, h->d_gemm + off);
    };
    auto products = [&](const ProdLists &pl, cudaStream_t ps) -> int {
        if (pl.gemm_cnt) {
            B(kProfGemm);
            k_gemm_tiles<T, kBM, kBN, kBK><<<pl.gemm_cnt, 256, 0, ps>>>(lnz, pool, h->d_tasks,
                                                                        h->d_gemm + pl.gemm_off);
            E();
            launches++;
        }
        if constexpr (sizeof(T) == 8) {
            if (pl.sp_cnt) {
                B(kProfTc);
                digit_products(pl.sp_off, pl.sp_cnt, ps);
                E();
                launches++;
            }
        }
        if constexpr (sizeof(T) == 4) {
            if (pl.tc_cnt) {
                B(kProfTc);
                launch_tc_gemm(128, h->precision == SC_TF32X3, (float *)lnz, h->d_tasks, h->d_gemm + pl.tc_off,
                               pl.tc_cnt, h->d_tmaps, h->nmaps, h->d_tmap_of_sn, h->d_err,
                               (long long)s->opt.spin_limit, h->num_sms, ps);
                E();
                launches++;
            }
            if (pl.tc256_cnt) {
                B(kProfTc);
                launch_tc_gemm(256, h->precision == SC_TF32X3, (float *)lnz, h->d_tasks, h->d_gemm + pl.tc256_off,
                               pl.tc256_cnt, h->d_tmaps, h->nmaps, h->d_tmap_of_sn, h->d_err,
                               (long long)s->opt.spin_limit, h->num_sms, ps, knobs_of(s->tune).tc_multicast);
                E();
                launches++;
            }
            if (pl.tc64_cnt) {
                B(kProfTc);
                launch_tc_gemm(64, h->precision == SC_TF32X3, (float *)lnz, h->d_tasks, h->d_gemm + pl.tc64_off,
                               pl.tc64_cnt, h->d_tmaps, h->nmaps, h->d_tmap_of_sn, h->d_err,
                               (long long)s->opt.spin_limit, h->num_sms, ps);
                E();
                launches++;
            }
        }
        if (pl.thin_cnt) {
            B(kProfGemm);
            k_thin_tasks<T><<<pl.thin_cnt, kThinWarps * 32, 0, ps>>>(lnz, h->d_tasks, h->d_thin + pl.thin_off);
            E();
            launches++;
        }
        return SC_OK;
    };
    const size_t nlev = h->plans.size();
    // FP64 by digits, except for a fused handle (here in its profile): its plan has the
    // FP64-pipe kernels' tiles, and it holds no digits
    const bool digits = sizeof(T) == 8 && !h->fused;
    for (size_t lv = 0; lv < nlev; lv++) {
        const LevelPlan &p = h->plans[lv];
        if (p.narrow_cnt) {
            B(kProfPotrf);
            k_narrow<T><<<(p.narrow_cnt + 7) / 8, 256, 0, st>>>(lnz, h->d_chunks, h->d_potrf + p.narrow_off,
                                                                p.narrow_cnt, h->d_adiag, h->d_info, h->d_info + 1, tau,
                                                                h->d_hi, h->d_lo, (T *)h->d_inv);
            E();
            launches++;
        }
        if (p.potrf_cnt) {
            B(kProfPotrf);
            if (digits)
                k_potrf64<<<p.potrf_cnt, 256, kChunk64Smem, st>>>((double *)lnz, h->d_chunks, h->d_potrf + p.potrf_off,
                                                                  h->d_info, h->d_chunk64);
            else
                k_potrf<T><<<p.potrf_cnt, 256, kPotrfSmem, st>>>(lnz, h->d_chunks, h->d_potrf + p.potrf_off, h->d_adiag,
                                                                  h->d_info, h->d_info + 1, tau, h->d_hi, h->d_lo);
            E();
            launches++;
        }
        if (p.trsm_cnt) {
            B(kProfTrsm);
            if (digits)
                k_trsm64<<<p.trsm_cnt, 256, kChunk64Smem, st>>>((double *)lnz, h->d_chunks, h->d_trsm + p.trsm_off,
                                                                h->d_chunk64);
            else
                k_trsm<T><<<p.trsm_cnt, trsm_rows<T>() * 4, 0, st>>>(lnz, h->d_chunks, h->d_trsm + p.trsm_off, h->d_hi,
                                                               h->d_lo);
            E();
            launches++;
        }
        if constexpr (sizeof(T) == 8) {
            // the level's half of the slice pool was last read by the products of level
            // lv - 2, which this stream has waited for (ev_rest, at level lv - 1)
            if (p.split_cnt && h->d_slices) {
                B(kProfTc);
                launch_split((const double *)lnz, h->d_splits, h->d_split_units + p.split_off, p.split_cnt,
                             h->d_slices, h->d_exps, st);
                E();
                launches++;
            }
        }
        // Lookahead: level lv's products into chunks two or more levels up run on
        // st3, overlapping level lv+1's POTRF, TRSM and device loops; level lv+1's
        // own products wait for them, so no target is written by two streams at
        // once (rest(lv) and crit(lv) have disjoint targets, and so have rest(lv)
        // and the device loops, which never target a supernode being factored).
        if (st3) {
            SC_CUDA(cudaEventRecord(h->ev_trsm, st));
            SC_CUDA(cudaStreamWaitEvent(st3, h->ev_trsm, 0));
            int rc = products(p.rest, st3);
            if (rc) return rc;
            SC_CUDA(cudaEventRecord(h->ev_rest[lv % 2], st3));
        }
        bool join = false;
        if (p.loop_cnt || p.loopw_cnt) {
            B(kProfLoop);
            cudaStream_t ls = st;
            if (st2 && (p.crit.any() || p.small_cnt)) {  // fork: loops and tiled products are independent
                SC_CUDA(cudaEventRecord(h->ev_fork, st));
                SC_CUDA(cudaStreamWaitEvent(st2, h->ev_fork, 0));
                ls = st2;
                join = true;
            }
            if (p.loop_cnt) {
                if (digits)
                    k_rlb_loop64<<<p.loop_cnt, 256, 0, ls>>>((double *)lnz, h->d_loops + p.loop_off, h->d_sn, h->d_blk,
                                                             h->d_rbval, h->d_row_blk);
                else
                    k_rlb_loop<T><<<p.loop_cnt, 256, 0, ls>>>(lnz, h->d_loops + p.loop_off, h->d_sn, h->d_blk,
                                                              h->d_rbval);
                launches++;
            }
            if (p.loopw_cnt) {
                if (digits)
                    k_rlb_loop_warp64<<<(p.loopw_cnt + 7) / 8, 256, 0, ls>>>(
                        (double *)lnz, h->d_loops + p.loopw_off, p.loopw_cnt, h->d_sn, h->d_blk, h->d_rbval,
                        h->d_row_blk);
                else
                    k_rlb_loop_warp<T><<<(p.loopw_cnt + 7) / 8, 256, 0, ls>>>(
                        lnz, h->d_loops + p.loopw_off, p.loopw_cnt, h->d_sn, h->d_blk, h->d_rbval);
                launches++;
            }
            if (join) SC_CUDA(cudaEventRecord(h->ev_join, st2));
            E();
        }
        {
            if (st3 && lv >= 1) SC_CUDA(cudaStreamWaitEvent(st, h->ev_rest[(lv - 1) % 2], 0));
            int rc = products(p.crit, st);
            if (rc) return rc;
            if (!st3 && (rc = products(p.rest, st))) return rc;
        }
        if (p.small_cnt) {
            B(kProfSmall);
            k_small_tasks<T><<<(p.small_cnt + 7) / 8, 256, 0, st>>>(lnz, pool, h->d_tasks, h->d_small + p.small_off,
                                                                    p.small_cnt);
            E();
            launches++;
        }
        if (p.rlg_cnt) {
            B(kProfRlUpd);
            k_gemm_tiles<T, kBM, kBN, kBK><<<p.rlg_cnt, 256, 0, st>>>(lnz, pool, h->d_tasks, h->d_gemm + p.rlg_off);
            E();
            launches++;
        }
        if constexpr (sizeof(T) == 8) {
            if (p.rlsp_cnt) {
                B(kProfRlUpd);
                digit_products(p.rlsp_off, p.rlsp_cnt, st);
                E();
                launches++;
            }
        }
        if (p.rls_cnt) {
            B(kProfRlUpd);
            k_small_tasks<T><<<(p.rls_cnt + 7) / 8, 256, 0, st>>>(lnz, pool, h->d_tasks, h->d_small + p.rls_off,
                                                                  p.rls_cnt);
            E();
            launches++;
        }
        if (join) SC_CUDA(cudaStreamWaitEvent(st, h->ev_join, 0));
        if (p.rlo_cnt) {
            B(kProfRlAsm);
            k_rl_assemble_ordered<T><<<p.rlo_cnt, 256, 0, st>>>(lnz, pool, h->d_rlpairs, h->d_rlslabs + p.rlo_off,
                                                                h->d_rlrelind);
            E();
            launches++;
        }
        for (int32_t q0 = 0; q0 < p.rlp_cnt && !p.rlo_cnt; q0 += 65535) {  // grid.y holds at most 65535 pairs
            unsigned gx = (unsigned)std::min<int64_t>((p.rlp_max + 255) / 256, 64);
            unsigned gy = (unsigned)std::min<int32_t>(65535, p.rlp_cnt - q0);
            B(kProfRlAsm);
            k_rl_assemble<T><<<dim3(gx, gy), 256, 0, st>>>(lnz, pool, h->d_rlpairs + p.rlp_off + q0, h->d_rlrelind);
            E();
            launches++;
        }
    }
    if (st3 && nlev) SC_CUDA(cudaStreamWaitEvent(st, h->ev_rest[(nlev - 1) % 2], 0));  // join the lookahead branch
    launch_inverses();
    SC_CUDA(cudaGetLastError());
    h->kernel_launches = launches;
    return SC_OK;
}

int set_smem_attrs() {
    static bool done = false;
    if (done) return SC_OK;
    SC_CUDA(cudaFuncSetAttribute(k_potrf<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPotrfSmem));
    SC_CUDA(cudaFuncSetAttribute(k_potrf<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPotrfSmem));
    SC_CUDA(cudaFuncSetAttribute(k_potrf64, cudaFuncAttributeMaxDynamicSharedMemorySize, kChunk64Smem));
    SC_CUDA(cudaFuncSetAttribute(k_trsm64, cudaFuncAttributeMaxDynamicSharedMemorySize, kChunk64Smem));
    SC_CUDA(cudaFuncSetAttribute(k_inverse64, cudaFuncAttributeMaxDynamicSharedMemorySize, kInv64Smem));
    SC_CUDA(cudaFuncSetAttribute(k_inverse, cudaFuncAttributeMaxDynamicSharedMemorySize, kPotrfSmem));
    SC_CUDA(cudaFuncSetAttribute(k_level<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPotrfSmem));
    SC_CUDA(cudaFuncSetAttribute(k_level<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPotrfSmem));
    if (!tc_gemm_init() || !split_gemm_init()) return SC_ERR_CUDA;
    done = true;
    return SC_OK;
}

// Host-only launch plan of one factorization for a precision: flat work lists
// with per-level offsets (no device memory touched).
struct Plan {
    std::vector<ChunkDev> cd;
    std::vector<int32_t> potrf, small;
    std::vector<ThinUnit> thin;
    std::vector<TrsmTile> trsm;
    std::vector<GemmTile> gemm;
    std::vector<Task> tasks;
    std::vector<RLPair> rlpairs;
    std::vector<RLSlab> rlslabs;
    std::vector<LoopItem> loops;
    std::vector<LevelPlan> levels;
    bool fused = false;    // for the per-level kernel: no k_narrow chunks (set before build_plan)
    int64_t inv_size = 0;  // elements of the diagonal-block inverses
    int32_t inv_off = 0, inv_cnt = 0;  // chunks of the inverse launch (in potrf)
    int32_t chunk64_units = 0;         // digits of a level's chunks (FP64), in 256-word units
    // FP64 products on the tensor cores (empty without them)
    std::vector<SplitBlk> splits;
    std::vector<SplitUnit> split_units;
    std::vector<int32_t> split_of_task;  // per task: its source block (0 where it has none)
    int64_t slice_pieces = 0;            // rows of the slice pool, both halves
    int64_t exps = 0;                    // row exponents, both halves
    double class_flops[kProfClasses] = {};
    // fused plans: the units of every level's k_level launch, then the tail launch's
    std::vector<FlowUnit> flow;
    int32_t flow_tail_off = 0, flow_tail_cnt = 0;
};

// Units of the per-level launches (fused plans): per level its POTRFs, TRSM
// tiles, the previous level's lookahead products (lookahead), its own products
// (with the rest as well when there is no lookahead), small tasks in eights,
// loop items, narrow loop items in eights; the last level's lookahead products
// form a tail launch.
void build_flow(Plan &P, bool lookahead) {
    P.flow.clear();
    auto products = [&](const ProdLists &pl) {
        for (int32_t i = 0; i < pl.gemm_cnt; i++) P.flow.push_back(FlowUnit{kFlowGemm, pl.gemm_off + i, 1, 0});
        for (int32_t i = 0; i < pl.thin_cnt; i += 2)
            P.flow.push_back(FlowUnit{kFlowThin, pl.thin_off + i, std::min<int32_t>(2, pl.thin_cnt - i), 0});
    };
    const size_t nlev = P.levels.size();
    for (size_t lv = 0; lv < nlev; lv++) {
        LevelPlan &p = P.levels[lv];
        p.flow_off = (int32_t)P.flow.size();
        for (int32_t i = 0; i < p.potrf_cnt; i++) P.flow.push_back(FlowUnit{kFlowPotrf, P.potrf[p.potrf_off + i], 1, 0});
        for (int32_t i = 0; i < p.trsm_cnt; i++) P.flow.push_back(FlowUnit{kFlowTrsm, p.trsm_off + i, 1, 0});
        if (lookahead && lv > 0) products(P.levels[lv - 1].rest);
        products(p.crit);
        if (!lookahead) products(p.rest);
        for (int32_t i = 0; i < p.small_cnt; i += 8)
            P.flow.push_back(FlowUnit{kFlowSmall, p.small_off + i, std::min<int32_t>(8, p.small_cnt - i), 0});
        for (int32_t i = 0; i < p.loop_cnt; i++) P.flow.push_back(FlowUnit{kFlowLoop, p.loop_off + i, 1, 0});
        for (int32_t i = 0; i < p.loopw_cnt; i += 8)
            P.flow.push_back(FlowUnit{kFlowLoopW, p.loopw_off + i, std::min<int32_t>(8, p.loopw_cnt - i), 0});
        p.flow_cnt = (int32_t)P.flow.size() - p.flow_off;
    }
    P.flow_tail_off = (int32_t)P.flow.size();
    if (lookahead && nlev) products(P.levels[nlev - 1].rest);
    P.flow_tail_cnt = (int32_t)P.flow.size() - P.flow_tail_off;
}

// lookahead: split each level's tiled products into those that target chunks
// of the next level (crit) and the rest (targets two or more levels up).
// split64: FP64 products on the tensor cores (split_route) instead of SIMT tiles.
void build_plan(const sc_symbolic *s, int precision, Plan &P, bool lookahead, bool split64) {
    const Knobs kn = knobs_of(s->tune);
    split64 = split64 && precision == SC_FP64;
    int64_t half_pieces[2] = {0, 0}, half_exps[2] = {0, 0};  // largest level of each parity
    std::vector<int32_t> split_of_sn(split64 ? s->nsuper : 0, -1);  // the level's block of a source supernode
    const bool det = s->opt.deterministic != 0;
    P.cd.resize(s->chunks.size());
    int64_t inv = 0;
    for (size_t c = 0; c < s->chunks.size(); c++) {
        const Chunk &ch = s->chunks[c];
        int32_t J = ch.sn;
        P.cd[c] = ChunkDev{s->lnz_off[J], s->gl_ptr[J], inv, s->lnz_ld[J], (int32_t)(s->gl_ptr[J + 1] - s->gl_ptr[J]),
                           ch.c0, ch.w, s->sup_ptr[J] + ch.c0, 0};
        inv += (int64_t)ch.w * ch.w;
    }
    P.inv_size = inv;
    const bool tc = precision == SC_TF32 || precision == SC_TF32X3;
    std::vector<int32_t> tmap_of_sn(s->nsuper, -1);
    {
        int32_t nm = 0;
        for (int64_t J = 0; J < s->nsuper; J++)
            if (s->sup_ptr[J + 1] - s->sup_ptr[J] >= 16) tmap_of_sn[J] = nm++;
    }
    P.levels.resize(s->levels.size());
    for (size_t lv = 0; lv < s->levels.size(); lv++) {
        const Level &L = s->levels[lv];
        LevelPlan &p = P.levels[lv];
        // chunks narrow and short enough for one warp, then the others; the per-level
        // kernel of a fused plan takes them all as the others
        auto small = [&](int32_t c) {
            const ChunkDev &ch = P.cd[c];
            return !P.fused && narrow_chunk(ch.w, ch.m - ch.c0 - ch.w, precision == SC_FP64);
        };
        // FP64: a level of few chunks gains nothing (a CTA takes a small chunk in about
        // the warp's time, and the level one launch less)
        const bool use_warps =
            precision != SC_FP64 || std::count_if(L.chunks.begin(), L.chunks.end(), small) >= kNarrowMin64;
        auto by_warp = [&](int32_t c) { return use_warps && small(c); };
        p.narrow_off = (int32_t)P.potrf.size();
        for (int32_t c : L.chunks) {
            if (by_warp(c)) P.potrf.push_back(c);
            double w = P.cd[c].w;
            P.class_flops[kProfPotrf] += w * w * w / 3.0;
            P.class_flops[kProfTrsm] += (double)(P.cd[c].m - P.cd[c].c0 - P.cd[c].w) * w * w;
        }
        p.narrow_cnt = (int32_t)P.potrf.size() - p.narrow_off;
        p.potrf_off = (int32_t)P.potrf.size();
        for (int32_t c : L.chunks)
            if (!by_warp(c)) P.potrf.push_back(c);
        p.potrf_cnt = (int32_t)P.potrf.size() - p.potrf_off;
        // FP64: where the POTRF leaves the chunk's digits for the TRSM (256-word units,
        // used again by the next level)
        int32_t slot = 0;
        for (int32_t i = 0; i < p.potrf_cnt; i++) {
            ChunkDev &ch = P.cd[P.potrf[p.potrf_off + i]];
            ch.slot = slot;
            slot += chunk64_units(ch.w);
        }
        P.chunk64_units = std::max(P.chunk64_units, slot);
        p.trsm_off = (int32_t)P.trsm.size();
        for (int32_t c : L.chunks) {
            if (by_warp(c)) continue;
            const ChunkDev &ch = P.cd[c];
            const int32_t rows = precision != SC_FP64 ? trsm_rows<float>() : P.fused ? trsm_rows<double>() : kTrsm64Rows;
            for (int32_t r0 = ch.c0 + ch.w; r0 < ch.m; r0 += rows) P.trsm.push_back(TrsmTile{c, r0});
        }
        p.trsm_cnt = (int32_t)P.trsm.size() - p.trsm_off;
        // product tasks: tensor-core tiles (TF32), SIMT tiles, warp tasks
        std::vector<int32_t> ids_small;
        std::vector<ThinUnit> units_thin[2];
        std::vector<GemmTile> g_simt[2], g_tc[2], g_tc64[2], g_tc256[2], g_sp[2];
        const bool split = lookahead;
        // the level's source blocks for FP64 products on the tensor cores: one per source
        // supernode (all of a level's products of a supernode read the same columns), its
        // rows from the first one that a routed product reads
        const size_t blk0 = P.splits.size();
        auto use_split = [&](const Task &t) {
            if (!split64 || is_small(t) || !split_route(t, s->sup_ptr[t.src + 1] - s->sup_ptr[t.src])) return false;
            const int32_t m = (int32_t)(s->gl_ptr[t.src + 1] - s->gl_ptr[t.src]), r = std::min(t.a_row, t.b_row);
            int32_t &b = split_of_sn[t.src];
            if (b < 0) {
                b = (int32_t)P.splits.size();
                P.splits.push_back(SplitBlk{s->lnz_off[t.src] + t.kx0, 0, s->lnz_ld[t.src], m - r, t.k, r, 0, 0});  // src, piece0, exp0: below
            } else if (r < P.splits[b].row0) {
                P.splits[b].rows = m - r;
                P.splits[b].row0 = r;
            }
            return true;
        };
        auto set_split = [&](const Task &t, int32_t id) {
            P.split_of_task.resize(id + 1, 0);
            P.split_of_task[id] = split_of_sn[t.src];
        };
        for (Task t : L.tasks) {
            int32_t id = (int32_t)P.tasks.size();
            const int cls = split && !(t.flags & kTaskCrit) ? 1 : 0;  // 0 crit, 1 rest
            P.tasks.push_back(t);
            int bn = tc ? tc_width(t, tmap_of_sn, s->sup_ptr[t.src + 1] - s->sup_ptr[t.src], kn.tc_min_k,
                                    kn.tc_wide_n, s->test_tc_ignore_tail)
                        : 0;
            if (bn == 128 && t.n >= kn.tc_wide256) bn = 256;
            if (is_small(t)) {
                ids_small.push_back(id);
                P.class_flops[kProfSmall] += task_flops(t);
            } else if (bn) {
                if (bn == 256 && kn.tc_multicast) tc_tile_pairs_of(t, id, g_tc256[cls]);
                else tc_tiles_of(t, id, bn, bn == 256 ? g_tc256[cls] : bn == 128 ? g_tc[cls] : g_tc64[cls]);
                P.class_flops[kProfTc] += task_flops(t);
            } else if (use_split(t)) {
                set_split(t, id);
                split_tiles_of(t, id, g_sp[cls]);
                P.class_flops[kProfTc] += task_flops(t);
            } else if (std::min(t.m, t.n) <= std::min(kn.thin_dim, kThinDim) && !(t.flags & kTaskStoreU)) {
                // a 64 x 64 tile would be mostly padding: warp blocks, kThinWarps per CTA
                const int ni = block_rows(t.m, t.n, precision == SC_FP64 ? 2 : 1, (t.flags & kTaskLower) != 0);
                const int nblk = ((t.m + ni - 1) / ni) * ((t.n + 32 / ni - 1) / (32 / ni));
                for (int b0 = 0; b0 < nblk; b0 += kThinWarps) units_thin[cls].push_back(ThinUnit{id, b0});
                P.class_flops[kProfGemm] += task_flops(t);
            } else {
                tiles_of(t, id, g_simt[cls], det);
                P.class_flops[kProfGemm] += task_flops(t);
            }
        }
        for (int cls = 0; cls < 2; cls++) {
            ProdLists &pl = cls == 0 ? p.crit : p.rest;
            pl.gemm_off = (int32_t)P.gemm.size();
            P.gemm.insert(P.gemm.end(), g_simt[cls].begin(), g_simt[cls].end());
            pl.gemm_cnt = (int32_t)g_simt[cls].size();
            pl.tc_off = (int32_t)P.gemm.size();
            P.gemm.insert(P.gemm.end(), g_tc[cls].begin(), g_tc[cls].end());
            pl.tc_cnt = (int32_t)g_tc[cls].size();
            pl.tc64_off = (int32_t)P.gemm.size();
            P.gemm.insert(P.gemm.end(), g_tc64[cls].begin(), g_tc64[cls].end());
            pl.tc64_cnt = (int32_t)g_tc64[cls].size();
            pl.tc256_off = (int32_t)P.gemm.size();
            P.gemm.insert(P.gemm.end(), g_tc256[cls].begin(), g_tc256[cls].end());
            pl.tc256_cnt = (int32_t)g_tc256[cls].size();
            pl.sp_off = (int32_t)P.gemm.size();
            P.gemm.insert(P.gemm.end(), g_sp[cls].begin(), g_sp[cls].end());
            pl.sp_cnt = (int32_t)g_sp[cls].size();
            pl.thin_off = (int32_t)P.thin.size();
            P.thin.insert(P.thin.end(), units_thin[cls].begin(), units_thin[cls].end());
            pl.thin_cnt = (int32_t)units_thin[cls].size();
        }
        p.small_off = (int32_t)P.small.size();
        P.small.insert(P.small.end(), ids_small.begin(), ids_small.end());
        p.small_cnt = (int32_t)ids_small.size();
        // device-side RLB loops
        // (items of supernodes narrower than 32 columns: one warp each)
        // (while a level has few of them a CTA each: a warp's chain of products would be
        // the level's time, 33 us a level of the 64 x 64 2D matrix)
        auto narrow = [&](const LoopItem &it) { return s->sup_ptr[it.sn + 1] - s->sup_ptr[it.sn] < 32; };
        const bool warp_items = std::count_if(L.loops.begin(), L.loops.end(), narrow) >= kLoopMinWarps;
        p.loop_off = (int32_t)P.loops.size();
        for (const LoopItem &it : L.loops)
            if (!warp_items || !narrow(it)) P.loops.push_back(it);
        p.loop_cnt = (int32_t)P.loops.size() - p.loop_off;
        p.loopw_off = (int32_t)P.loops.size();
        for (const LoopItem &it : L.loops)
            if (warp_items && narrow(it)) P.loops.push_back(it);
        p.loopw_cnt = (int32_t)P.loops.size() - p.loopw_off;
        P.class_flops[kProfLoop] += L.loop_flops;
        // RL update matrices and assembly
        std::vector<int32_t> rl_small;
        std::vector<GemmTile> rl_g, rl_sp;
        for (const Task &t : L.rl_tasks) {
            int32_t id = (int32_t)P.tasks.size();
            P.tasks.push_back(t);
            if (is_small(t)) {
                rl_small.push_back(id);
            } else if (use_split(t)) {
                set_split(t, id);
                split_tiles_of(t, id, rl_sp);
            } else {
                tiles_of(t, id, rl_g, det);
            }
            P.class_flops[kProfRlUpd] += task_flops(t);
        }
        p.rlsp_off = (int32_t)P.gemm.size();
        P.gemm.insert(P.gemm.end(), rl_sp.begin(), rl_sp.end());
        p.rlsp_cnt = (int32_t)rl_sp.size();
        // slices and exponents of the level's blocks, from the start of the level's half
        // (the offsets of odd levels get the even half's size added below)
        p.split_off = (int32_t)P.split_units.size();
        {
            int64_t piece = 0, exp = 0;
            for (size_t b = blk0; b < P.splits.size(); b++) {
                SplitBlk &bk = P.splits[b];
                bk.src += (int64_t)bk.row0 * bk.ld;
                bk.piece0 = piece;
                bk.exp0 = (int32_t)exp;
                bk.pad = (int32_t)(lv % 2);
                piece += (int64_t)((bk.k + sp::BK - 1) / sp::BK) * sp::S * bk.rows;
                exp += bk.rows;
                for (int32_t r = 0; r < bk.rows; r += kSplitRows) P.split_units.push_back(SplitUnit{(int32_t)b, r});
            }
            half_pieces[lv % 2] = std::max(half_pieces[lv % 2], piece);
            half_exps[lv % 2] = std::max(half_exps[lv % 2], exp);
            for (const Task &t : L.tasks)
                if (split64) split_of_sn[t.src] = -1;
            for (const Task &t : L.rl_tasks)
                if (split64) split_of_sn[t.src] = -1;
        }
        p.split_cnt = (int32_t)P.split_units.size() - p.split_off;
        p.rlg_off = (int32_t)P.gemm.size();
        P.gemm.insert(P.gemm.end(), rl_g.begin(), rl_g.end());
        p.rlg_cnt = (int32_t)rl_g.size();
        p.rls_off = (int32_t)P.small.size();
        P.small.insert(P.small.end(), rl_small.begin(), rl_small.end());
        p.rls_cnt = (int32_t)rl_small.size();
        p.rlp_off = (int32_t)P.rlpairs.size();
        for (const RLPair &pr : L.rl_pairs) {
            P.rlpairs.push_back(pr);
            p.rlp_max = std::max<int64_t>(p.rlp_max, (int64_t)(pr.c_end - pr.c_begin) * (pr.s - pr.c_begin));
            P.class_flops[kProfRlAsm] += (double)(pr.c_end - pr.c_begin) * (pr.s - pr.c_begin);
        }
        p.rlp_cnt = (int32_t)L.rl_pairs.size();
        if (det) {
            // target-owned assembly: the level's pairs grouped by target P, each
            // group in the order of its source supernodes (the order the level
            // lists them in), P's touched rows cut into slabs of kRLSlabRows
            auto first = P.rlpairs.begin() + p.rlp_off;
            std::stable_sort(first, P.rlpairs.end(),
                             [](const RLPair &a, const RLPair &b) { return a.p_off < b.p_off; });
            p.rlo_off = (int32_t)P.rlslabs.size();
            for (int32_t g0 = p.rlp_off, g1; g0 < (int32_t)P.rlpairs.size(); g0 = g1) {
                int32_t lo = INT32_MAX, hi = -1;
                for (g1 = g0; g1 < (int32_t)P.rlpairs.size() && P.rlpairs[g1].p_off == P.rlpairs[g0].p_off; g1++) {
                    const RLPair &pr = P.rlpairs[g1];
                    const int32_t *ri = s->rl_relind.data() + pr.ri_off;
                    // target rows mP - 1 - relind[r] of the pair's rows, ascending in r
                    lo = std::min(lo, pr.mP - 1 - ri[0]);
                    hi = std::max(hi, pr.mP - 1 - ri[pr.s - pr.c_begin - 1]);
                }
                for (int32_t r = lo; r <= hi; r += kRLSlabRows)
                    P.rlslabs.push_back(RLSlab{g0, g1 - g0, r, std::min(hi + 1, r + kRLSlabRows)});
            }
            p.rlo_cnt = (int32_t)P.rlslabs.size() - p.rlo_off;
            if (s->test_det_short_slab && p.rlo_cnt && !P.rlslabs.empty()) {
                RLSlab &last = P.rlslabs.back();  // its last row is a touched row (the group's hi)
                if (last.row1 - last.row0 > 1 && P.rlslabs.size() == (size_t)p.rlo_cnt) last.row1--;
            }
        }
    }
    // the chunks that the inverse launch takes: all but k_narrow's (FP64: the sweeps
    // substitute in the chunks up to kNarrowChunk)
    P.inv_off = (int32_t)P.potrf.size();
    for (const LevelPlan &p : P.levels)
        for (int32_t i = 0; i < p.potrf_cnt; i++) {
            const int32_t c = P.potrf[p.potrf_off + i];
            if (precision != SC_FP64 || P.cd[c].w > kNarrowChunk) P.potrf.push_back(c);
        }
    P.inv_cnt = (int32_t)P.potrf.size() - P.inv_off;
    for (SplitBlk &bk : P.splits)
        if (bk.pad) {
            bk.piece0 += half_pieces[0];
            bk.exp0 += (int32_t)half_exps[0];
        }
    P.slice_pieces = half_pieces[0] + half_pieces[1];
    P.exps = half_exps[0] + half_exps[1];
    P.split_of_task.resize(P.tasks.size(), 0);
}

}  // namespace

// one persistent launch per level (SIMT tiles only): FP64 and FP32, RLB schedule
static bool fused_plan(const sc_symbolic *s, int precision) {
    return knobs_of(s->tune).fused && s->opt.variant == SC_RLB && (precision == SC_FP64 || precision == SC_FP32);
}

int det_plan_check(const sc_symbolic *s, int64_t *bad_level) {
    for (int precision : {SC_FP64, SC_TF32}) {
        Plan P;
        build_plan(s, precision, P, false, true);
        for (size_t lv = 0; lv < P.levels.size(); lv++) {
            const LevelPlan &p = P.levels[lv];
            *bad_level = (int64_t)lv;
            auto split_in = [&](int32_t off, int32_t cnt) {
                for (int32_t i = off; i < off + cnt; i++)
                    if (P.gemm[i].ks >= 0) return true;
                return false;
            };
            for (const ProdLists *pl : {&p.crit, &p.rest})
                if (split_in(pl->gemm_off, pl->gemm_cnt) || split_in(pl->tc_off, pl->tc_cnt) ||
                    split_in(pl->tc64_off, pl->tc64_cnt) || split_in(pl->tc256_off, pl->tc256_cnt) ||
                    split_in(pl->sp_off, pl->sp_cnt))
                    return 13;
            if (split_in(p.rlg_off, p.rlg_cnt) || split_in(p.rlsp_off, p.rlsp_cnt)) return 13;
            if (!p.rlp_cnt) continue;
            // slabs: inside the level's pairs, one target each, sources ascending (pool offsets
            // follow the level's source order), groups disjoint and ascending, a group's row
            // ranges non-empty, ascending and disjoint
            const int32_t pe = p.rlp_off + p.rlp_cnt;
            for (int32_t q = p.rlo_off; q < p.rlo_off + p.rlo_cnt; q++) {
                const RLSlab &sl = P.rlslabs[q];
                if (sl.npairs < 1 || sl.pair0 < p.rlp_off || sl.pair0 + sl.npairs > pe || sl.row0 >= sl.row1) return 13;
                for (int32_t i = sl.pair0 + 1; i < sl.pair0 + sl.npairs; i++)
                    if (P.rlpairs[i].p_off != P.rlpairs[sl.pair0].p_off || P.rlpairs[i].u_off <= P.rlpairs[i - 1].u_off)
                        return 13;
                if (q > p.rlo_off) {
                    const RLSlab &pv = P.rlslabs[q - 1];
                    if (pv.pair0 == sl.pair0 ? (pv.npairs != sl.npairs || pv.row1 > sl.row0)
                                             : pv.pair0 + pv.npairs > sl.pair0)
                        return 13;
                }
            }
            // every target row of every pair lies in a slab of the pair's group
            int32_t q = p.rlo_off;
            for (int32_t i = p.rlp_off; i < pe; i++) {
                while (q < p.rlo_off + p.rlo_cnt && P.rlslabs[q].pair0 + P.rlslabs[q].npairs <= i) q++;
                if (q == p.rlo_off + p.rlo_cnt || P.rlslabs[q].pair0 > i) return 13;
                int32_t qe = q;
                while (qe < p.rlo_off + p.rlo_cnt && P.rlslabs[qe].pair0 == P.rlslabs[q].pair0) qe++;
                const RLPair &pr = P.rlpairs[i];
                const int32_t *ri = s->rl_relind.data() + pr.ri_off;
                for (int32_t r = 0, k = q; r < pr.s - pr.c_begin; r++) {
                    const int32_t row = pr.mP - 1 - ri[r];
                    while (k < qe && P.rlslabs[k].row1 <= row) k++;
                    if (k == qe || P.rlslabs[k].row0 > row) return 13;
                }
            }
        }
    }
    *bad_level = -1;
    return 0;
}

int split_plan_check(const sc_symbolic *s, int64_t *bad_level) {
    Plan P;
    build_plan(s, SC_FP64, P, false, true);
    std::vector<int64_t> half_end(2, 0);  // slice rows used by the levels of each parity
    int64_t odd0 = INT64_MAX;
    for (size_t lv = 0; lv < P.levels.size(); lv++) {
        const LevelPlan &p = P.levels[lv];
        *bad_level = (int64_t)lv;
        int64_t end = -1;
        for (int32_t u = p.split_off; u < p.split_off + p.split_cnt; u++) {
            const SplitUnit &su = P.split_units[u];
            const SplitBlk &b = P.splits[su.blk];
            // every row of a block once: its units in order, blocks one after another
            const bool head = u == p.split_off || P.split_units[u - 1].blk != su.blk;
            if (su.row0 != (head ? 0 : P.split_units[u - 1].row0 + kSplitRows) || su.row0 >= b.rows) return 14;
            const bool tail = u + 1 == p.split_off + p.split_cnt || P.split_units[u + 1].blk != su.blk;
            if (tail && su.row0 + kSplitRows < b.rows) return 14;
            if (!head) continue;
            // slices inside the pool, after the previous block's; exponents likewise
            if (b.rows < 1 || b.k < 1 || (end >= 0 && b.piece0 < end) || b.exp0 < 0 || b.exp0 + (int64_t)b.rows > P.exps)
                return 14;
            if (lv % 2) odd0 = std::min(odd0, b.piece0);
            end = b.piece0 + (int64_t)((b.k + sp::BK - 1) / sp::BK) * sp::S * b.rows;
            half_end[lv % 2] = std::max(half_end[lv % 2], end);
            if (b.piece0 < 0 || end > P.slice_pieces) return 14;
        }
        auto tiles_ok = [&](int32_t off, int32_t cnt) {
            for (int32_t i = off; i < off + cnt; i++) {
                const Task &t = P.tasks[P.gemm[i].task];
                const int32_t bi = P.split_of_task[P.gemm[i].task];
                if (bi < 0 || bi >= (int32_t)P.splits.size()) return false;
                const SplitBlk &b = P.splits[bi];
                const int32_t ld = s->lnz_ld[t.src];
                // the block is this level's, and holds the product's rows and columns, 16-byte aligned
                bool mine = false;
                for (int32_t u = p.split_off; !mine && u < p.split_off + p.split_cnt;
                     u += std::max(1, (P.splits[P.split_units[u].blk].rows + kSplitRows - 1) / kSplitRows))
                    mine = P.split_units[u].blk == bi;
                if (!mine || b.k != t.k || b.ld != ld ||
                    b.src != s->lnz_off[t.src] + (int64_t)b.row0 * ld + t.kx0 || b.src % 2 || ld % 2)
                    return false;
                for (int32_t r : {t.a_row, t.b_row})
                    if (r < b.row0) return false;
                if (t.a_row + t.m > b.row0 + b.rows || t.b_row + t.n > b.row0 + b.rows) return false;
                while (i + 1 < off + cnt && P.gemm[i + 1].task == P.gemm[i].task) i++;
            }
            return true;
        };
        if (!tiles_ok(p.crit.sp_off, p.crit.sp_cnt) || !tiles_ok(p.rest.sp_off, p.rest.sp_cnt) ||
            !tiles_ok(p.rlsp_off, p.rlsp_cnt))
            return 14;
    }
    // the two halves apart: a level's products may still read theirs while the next
    // level's are being written
    *bad_level = (int64_t)P.levels.size() - 1;
    if (odd0 != INT64_MAX && half_end[0] > odd0) return 14;
    *bad_level = -1;
    return 0;
}

int plan_stats(const sc_symbolic *s, int precision, int64_t *out, int nout) {
    Plan P;
    P.fused = fused_plan(s, precision);
    int64_t digit_tiles = 0;
    if (precision == SC_FP64 && !P.fused) {
        Plan D;
        build_plan(s, precision, D, false, true);
        for (const LevelPlan &l : D.levels) digit_tiles += l.crit.sp_cnt + l.rest.sp_cnt + l.rlsp_cnt;
    }
    build_plan(s, precision, P, false, false);  // FP64: the products as the SIMT tiles they cover
    int64_t small_tasks = 0, tile_tasks = 0;
    for (const LevelPlan &l : P.levels) small_tasks += l.small_cnt + l.rls_cnt;
    tile_tasks = (int64_t)P.tasks.size() - small_tasks;
    int64_t tc_tiles = 0, simt_tiles = 0, split_tiles = 0, tc256_tiles = 0;
    for (const LevelPlan &l : P.levels) {
        tc256_tiles += l.crit.tc256_cnt + l.rest.tc256_cnt;
        tc_tiles += l.crit.tc_cnt + l.crit.tc64_cnt + l.crit.tc256_cnt + l.rest.tc_cnt + l.rest.tc64_cnt +
                    l.rest.tc256_cnt;
        simt_tiles += l.crit.gemm_cnt + l.rest.gemm_cnt + l.rlg_cnt;
    }
    for (const GemmTile &g : P.gemm) split_tiles += g.ks >= 0;
    int64_t v[] = {(int64_t)P.levels.size(), (int64_t)P.cd.size(), (int64_t)P.tasks.size(), small_tasks, tile_tasks,
                   simt_tiles, tc_tiles, (int64_t)P.trsm.size(), (int64_t)P.rlpairs.size(), (int64_t)P.loops.size(),
                   (int64_t)P.thin.size(), split_tiles, (int64_t)P.rlslabs.size(), tc256_tiles, digit_tiles};
    for (int i = 0; i < nout && i < (int)(sizeof(v) / sizeof(v[0])); i++) out[i] = v[i];
    return SC_OK;
}

int numeric_create(sc_symbolic *s, int precision, sc_numeric **out) {
    if (precision < SC_FP64 || precision > SC_TF32X3) return -3;
    if (s->poisoned) return SC_ERR_INTERNAL;
    int rc = set_smem_attrs();
    if (rc) return rc;
    auto h = new sc_numeric();
    h->sym = s;
    s->refs++;  // released by numeric_free, also on the error paths below
    h->precision = precision;
    h->elt = precision == SC_FP64 ? 8 : 4;
    h->use_graph = s->opt.use_graph != 0;
    {
        int dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (h->num_sms < 1) h->num_sms = 1;
    }
    int64_t &bytes = h->device_bytes;
    auto fail = [&](int code) {
        numeric_free(h);
        return code;
    };
    if (cudaMalloc(&h->d_lnz, (size_t)s->lnz_size * h->elt) != cudaSuccess) return fail(SC_ERR_OOM);
    bytes += s->lnz_size * (int64_t)h->elt;
    if (cudaMalloc(&h->d_pool, (size_t)std::max<int64_t>(1, s->rl_pool_max) * h->elt) != cudaSuccess)
        return fail(SC_ERR_OOM);
    bytes += std::max<int64_t>(1, s->rl_pool_max) * (int64_t)h->elt;
    if ((rc = upload(h->d_valmap, s->valmap, bytes))) return fail(rc);
    if (cudaMalloc((void **)&h->d_values, std::max<size_t>(1, s->valmap.size()) * sizeof(double)) != cudaSuccess)
        return fail(SC_ERR_OOM);
    bytes += (int64_t)s->valmap.size() * 8;
    {
        std::vector<int64_t> dp(s->n);
        for (int64_t k = 0; k < s->n; k++) dp[k] = s->colptr[s->perm[k]];  // diagonal is first in its column
        if ((rc = upload(h->d_diagpos, dp, bytes))) return fail(rc);
    }
    if (cudaMalloc((void **)&h->d_adiag, (size_t)s->n * sizeof(double)) != cudaSuccess) return fail(SC_ERR_OOM);
    if (cudaMalloc((void **)&h->d_info, 2 * sizeof(int32_t)) != cudaSuccess) return fail(SC_ERR_OOM);
    if (cudaMalloc((void **)&h->d_err, sizeof(int32_t)) != cudaSuccess) return fail(SC_ERR_OOM);
    if (precision == SC_TF32X3) {
        // split copies of the factor: zero once, so padding columns stay zero
        for (float **p : {&h->d_hi, &h->d_lo}) {
            if (cudaMalloc((void **)p, (size_t)s->lnz_size * sizeof(float)) != cudaSuccess) return fail(SC_ERR_OOM);
            if (cudaMemset(*p, 0, (size_t)s->lnz_size * sizeof(float)) != cudaSuccess) return fail(SC_ERR_CUDA);
            bytes += s->lnz_size * 4;
        }
    }
    if (precision == SC_TF32 || precision == SC_TF32X3) {
        // TF32: maps over the factor; TF32x3: maps over hi, then maps over lo
        std::vector<CUtensorMap> maps, maps_lo;
        std::vector<int32_t> tmap_of_sn;
        if ((rc = tc_encode_maps(s, precision == SC_TF32 ? (float *)h->d_lnz : h->d_hi, maps, tmap_of_sn)))
            return fail(rc);
        h->nmaps = (int32_t)(maps.size() / 2);
        if (precision == SC_TF32X3) {
            if ((rc = tc_encode_maps(s, h->d_lo, maps_lo, tmap_of_sn))) return fail(rc);
            maps.insert(maps.end(), maps_lo.begin(), maps_lo.end());
        }
        if ((rc = upload(h->d_tmaps, maps, bytes))) return fail(rc);
        if ((rc = upload(h->d_tmap_of_sn, tmap_of_sn, bytes))) return fail(rc);
    }
    Plan P;
    const Knobs kn = knobs_of(s->tune);
    h->fused = P.fused = fused_plan(s, precision);
    // lookahead needs concurrent work: the captured graph's branches, or the fused launches
    h->lookahead = (h->use_graph || h->fused) && s->opt.variant == SC_RLB && kn.lookahead;
    build_plan(s, precision, P, h->lookahead, !h->fused);
    if (precision != SC_FP64) {
        if (cudaMalloc(&h->d_inv, (size_t)std::max<int64_t>(1, P.inv_size) * h->elt) != cudaSuccess) return fail(SC_ERR_OOM);
        bytes += P.inv_size * (int64_t)h->elt;
    } else if (!h->fused) {
        // what FP64 by digits holds beside the factor: the inverses and the digits between POTRF
        // and TRSM (4 to 17 % of the factor's size). Without room an RLB handle runs
        // by FP64 operations, which hold neither.
        const size_t b[3] = {(size_t)std::max<int64_t>(1, P.inv_size) * h->elt,
                             (size_t)std::max(1, P.chunk64_units) * 256 * sizeof(uint64_t),
                             ((size_t)s->n * 2 + s->chunks.size()) * sizeof(int32_t)};
        if (cudaMalloc(&h->d_inv, b[0]) == cudaSuccess && cudaMalloc((void **)&h->d_chunk64, b[1]) == cudaSuccess &&
            cudaMalloc((void **)&h->d_inv_exp, b[2]) == cudaSuccess) {
            bytes += (int64_t)(b[0] + b[1] + b[2]);
        } else {
            if (s->opt.variant != SC_RLB) return fail(SC_ERR_OOM);
            cudaGetLastError();
            for (void *p : {h->d_inv, (void *)h->d_chunk64, (void *)h->d_inv_exp})
                if (p) cudaFree(p);
            h->d_inv = nullptr;
            h->d_chunk64 = nullptr;
            h->d_inv_exp = nullptr;
            P = Plan();
            h->fused = P.fused = true;
            h->lookahead = kn.lookahead;
            build_plan(s, precision, P, h->lookahead, false);
        }
    }
    if (h->fused) {
        build_flow(P, h->lookahead);
        h->flow_tail_off = P.flow_tail_off;
        h->flow_tail_cnt = P.flow_tail_cnt;
        const size_t nch = s->chunks.size();
        std::vector<int32_t> need(nch, 1), task_chunk(P.tasks.size()), sn_chunk(s->nsuper);
        for (const TrsmTile &t : P.trsm) need[t.chunk]++;
        for (size_t i = 0; i < P.tasks.size(); i++) {
            const Task &t = P.tasks[i];
            task_chunk[i] = s->chunk_of_col[s->sup_ptr[t.src] + t.kx0 + t.k - 1];
        }
        for (int64_t J = 0; J < s->nsuper; J++) sn_chunk[J] = s->chunk_of_col[s->sup_ptr[J + 1] - 1];
        if ((rc = upload(h->d_flow, P.flow, bytes))) return fail(rc);
        if ((rc = upload(h->d_flow_need, need, bytes))) return fail(rc);
        if ((rc = upload(h->d_task_chunk, task_chunk, bytes))) return fail(rc);
        if ((rc = upload(h->d_sn_chunk, sn_chunk, bytes))) return fail(rc);
        const size_t words = nch * kFlowStride + P.levels.size() + 1;
        if (cudaMalloc((void **)&h->d_flow_ctr, words * sizeof(int32_t)) != cudaSuccess) return fail(SC_ERR_OOM);
        bytes += (int64_t)(words * sizeof(int32_t));
    }
    std::copy(P.class_flops, P.class_flops + kProfClasses, h->class_flops);
    h->plans = P.levels;
    h->inv_off = P.inv_off;
    h->inv_cnt = P.inv_cnt;
    h->ntasks = (int32_t)P.tasks.size();
    if ((rc = upload(h->d_chunks, P.cd, bytes))) return fail(rc);
    if ((rc = upload(h->d_potrf, P.potrf, bytes))) return fail(rc);
    if ((rc = upload(h->d_trsm, P.trsm, bytes))) return fail(rc);
    if ((rc = upload(h->d_gemm, P.gemm, bytes))) return fail(rc);
    if ((rc = upload(h->d_small, P.small, bytes))) return fail(rc);
    if ((rc = upload(h->d_thin, P.thin, bytes))) return fail(rc);
    if ((rc = upload(h->d_tasks, P.tasks, bytes))) return fail(rc);
    if ((rc = upload(h->d_rlpairs, P.rlpairs, bytes))) return fail(rc);
    if ((rc = upload(h->d_rlslabs, P.rlslabs, bytes))) return fail(rc);
    if ((rc = upload(h->d_rlrelind, s->rl_relind, bytes))) return fail(rc);
    if ((rc = upload(h->d_loops, P.loops, bytes))) return fail(rc);
    {
        std::vector<SnDev> snd(s->nsuper);
        for (int64_t J = 0; J < s->nsuper; J++)
            snd[J] = SnDev{s->lnz_off[J], s->lnz_ld[J], (int32_t)(s->gl_ptr[J + 1] - s->gl_ptr[J]), s->sup_ptr[J],
                           s->sup_ptr[J + 1] - s->sup_ptr[J], (int32_t)s->blk_ptr[J + 1], 0, s->gl_ptr[J]};
        std::vector<BlkDev> bd(s->blk_first.size());
        for (int64_t J = 0; J < s->nsuper; J++) {
            int64_t b0 = s->blk_ptr[J], b1 = s->blk_ptr[J + 1];
            int32_t q = s->sup_ptr[J + 1] - s->sup_ptr[J];
            for (int64_t b = b0; b < b1; b++) {
                bd[b] = BlkDev{q, s->blk_size[b], s->blk_first[b], s->blk_owner[b], 0, 0, 0};
                q += s->blk_size[b];
            }
            for (int64_t pq = s->rb_pair_ptr[J]; pq < s->rb_pair_ptr[J + 1]; pq++) {
                int64_t cnt = s->rb_val_ptr[pq + 1] - s->rb_val_ptr[pq];
                int64_t bs = b1 - cnt;
                for (int64_t b = bs; b < b1 && s->blk_owner[b] == s->rb_pair_P[pq]; b++) {
                    bd[b].rb = s->rb_val_ptr[pq];
                    bd[b].bs = (int32_t)bs;
                }
            }
        }
        if ((rc = upload(h->d_sn, snd, bytes))) return fail(rc);
        if ((rc = upload(h->d_blk, bd, bytes))) return fail(rc);
        if ((rc = upload(h->d_rbval, s->rb_val, bytes))) return fail(rc);
        if (precision == SC_FP64 && !h->fused && !P.loops.empty()) {
            std::vector<int32_t> rb(s->glbind.size(), 0);
            for (int64_t J = 0; J < s->nsuper; J++) {
                int64_t q = s->gl_ptr[J] + s->sup_ptr[J + 1] - s->sup_ptr[J];
                for (int64_t b = s->blk_ptr[J]; b < s->blk_ptr[J + 1]; b++)
                    for (int32_t i = 0; i < s->blk_size[b]; i++) rb[q++] = (int32_t)b;
            }
            if ((rc = upload(h->d_row_blk, rb, bytes))) return fail(rc);
        }
    }
    if (!P.splits.empty()) {
        // the slice pool, last. It takes at most half of what is free: a matrix whose factor and
        // solve vectors fit the device without the pool must not run out of memory because of it
        // (and a solve that does takes it back). Without it, or with more rows than a tensor
        // map's coordinate reaches, k_digit_tiles forms the same products to the same bits:
        // 27-point 40^3 factor 13.3 ms with the pool, 27.5 without; 7-point 48^3 16.3 and 49.9.
        const size_t pool = (size_t)P.slice_pieces * sp::BK * sizeof(uint16_t);
        size_t free_bytes = 0, total_bytes = 0;
        if (cudaMemGetInfo(&free_bytes, &total_bytes) != cudaSuccess) return fail(SC_ERR_CUDA);
        if (P.slice_pieces <= INT32_MAX && pool <= free_bytes / 2 &&
            cudaMalloc((void **)&h->d_slices, pool) == cudaSuccess) {
            h->slice_bytes = (int64_t)pool;
            bytes += h->slice_bytes;
            std::vector<CUtensorMap> maps;
            if ((rc = split_encode_maps(h->d_slices, P.slice_pieces, maps))) return fail(rc);
            if (cudaMalloc((void **)&h->d_exps, (size_t)P.exps * sizeof(int32_t)) != cudaSuccess) return fail(SC_ERR_OOM);
            bytes += P.exps * (int64_t)sizeof(int32_t);
            if ((rc = upload(h->d_slice_maps, maps, bytes))) return fail(rc);
            if ((rc = upload(h->d_splits, P.splits, bytes))) return fail(rc);
            if ((rc = upload(h->d_split_units, P.split_units, bytes))) return fail(rc);
            if ((rc = upload(h->d_split_of_task, P.split_of_task, bytes))) return fail(rc);
        } else {
            cudaGetLastError();
        }
    }
    *out = h;
    return SC_OK;
}

int numeric_factor(sc_numeric *h, const double *values, int on_device, cudaStream_t st, sc_factor_info *info) {
    const sc_symbolic *s = h->sym;
    int64_t nnz = (int64_t)s->valmap.size();
    h->last_stream = st;
    if (h->stall_factor_chunk >= 0) {
        // test hook: this factorization's units that read the chunk wait for one
        // more POTRF / TRSM completion than will come; their bounded waits give up
        const int32_t c = h->stall_factor_chunk;
        h->stall_factor_chunk = -1;
        if (!h->fused || c >= (int32_t)s->chunks.size()) return SC_ERR_UNSUPPORTED;
        int32_t need = 0;
        SC_CUDA(cudaMemcpy(&need, h->d_flow_need + c, sizeof(need), cudaMemcpyDeviceToHost));
        const int32_t raised = need + 1;
        SC_CUDA(cudaMemcpy(h->d_flow_need + c, &raised, sizeof(raised), cudaMemcpyHostToDevice));
        const int rc = numeric_factor(h, values, on_device, st, info);
        cudaStreamSynchronize(st);
        SC_CUDA(cudaMemcpy(h->d_flow_need + c, &need, sizeof(need), cudaMemcpyHostToDevice));
        return rc;
    }
    SC_CUDA(cudaMemcpyAsync(h->d_values, values, nnz * sizeof(double),
                            on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st));
    cudaEvent_t e0, e1;
    SC_CUDA(cudaEventCreate(&e0));
    SC_CUDA(cudaEventCreate(&e1));
    SC_CUDA(cudaEventRecord(e0, st));
    int rc = SC_OK;
    if (h->use_graph) {
        if (!h->gexec) {
            // captured once on the handle's own stream (the legacy default stream
            // cannot be captured), then replayed on the caller's stream
            if (!h->cap_stream) SC_CUDA(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
            if (!h->cap_stream2) SC_CUDA(cudaStreamCreateWithFlags(&h->cap_stream2, cudaStreamNonBlocking));
            if (!h->ev_fork) SC_CUDA(cudaEventCreateWithFlags(&h->ev_fork, cudaEventDisableTiming));
            if (!h->ev_join) SC_CUDA(cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming));
            cudaStream_t st3 = nullptr;
            if (h->lookahead) {
                if (!h->cap_stream3) SC_CUDA(cudaStreamCreateWithFlags(&h->cap_stream3, cudaStreamNonBlocking));
                if (!h->ev_trsm) SC_CUDA(cudaEventCreateWithFlags(&h->ev_trsm, cudaEventDisableTiming));
                for (auto &e : h->ev_rest)
                    if (!e) SC_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
                st3 = h->cap_stream3;
            }
            cudaGraph_t g;
            SC_CUDA(cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal));
            rc = h->precision == SC_FP64 ? run_levels<double>(h, h->cap_stream, nullptr, h->cap_stream2, st3)
                                         : run_levels<float>(h, h->cap_stream, nullptr, h->cap_stream2, st3);
            cudaError_t ce = cudaStreamEndCapture(h->cap_stream, &g);
            if (rc) return rc;
            SC_CUDA(ce);
            SC_CUDA(cudaGraphInstantiate(&h->gexec, g, 0));
            cudaGraphDestroy(g);
        }
        SC_CUDA(cudaGraphLaunch(h->gexec, st));
    } else {
        rc = h->precision == SC_FP64 ? run_levels<double>(h, st) : run_levels<float>(h, st);
        if (rc) return rc;
    }
    SC_CUDA(cudaEventRecord(e1, st));
    int32_t hinfo[2], herr = 0;
    SC_CUDA(cudaMemcpyAsync(hinfo, h->d_info, sizeof(hinfo), cudaMemcpyDeviceToHost, st));
    SC_CUDA(cudaMemcpyAsync(&herr, h->d_err, sizeof(herr), cudaMemcpyDeviceToHost, st));
    SC_CUDA(cudaStreamSynchronize(st));
    if (herr) return SC_ERR_TIMEOUT;
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    int64_t failed = 0;
    if (hinfo[0] != 0x7f7f7f7f) failed = (int64_t)s->perm[hinfo[0] - 1] + 1;
    if (info) {
        info->failed_col = failed;
        info->precision = h->precision;
        info->pivot_fallbacks = hinfo[1];
        info->flops = s->flops;
        info->factor_ms = ms;
        info->device_bytes = h->device_bytes;
        info->kernel_launches = h->kernel_launches;
    }
    return failed ? (int)std::min<int64_t>(failed, INT32_MAX) : SC_OK;
}

int numeric_profile(sc_numeric *h, const double *values, int on_device, cudaStream_t st, double *ms, double *flops,
                    int32_t *launches) {
    const sc_symbolic *s = h->sym;
    int64_t nnz = (int64_t)s->valmap.size();
    h->last_stream = st;
    SC_CUDA(cudaMemcpyAsync(h->d_values, values, nnz * sizeof(double),
                            on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st));
    Prof prof;
    prof.st = st;
    int rc = h->precision == SC_FP64 ? run_levels<double>(h, st, &prof) : run_levels<float>(h, st, &prof);
    SC_CUDA(cudaStreamSynchronize(st));
    for (int c = 0; c < kProfClasses; c++) {
        ms[c] = 0.0;
        flops[c] = h->class_flops[c];
        launches[c] = 0;
    }
    for (auto &e : prof.ev) {
        float t = 0.f;
        cudaEventElapsedTime(&t, e.second.first, e.second.second);
        ms[e.first] += t;
        launches[e.first]++;
        cudaEventDestroy(e.second.first);
        cudaEventDestroy(e.second.second);
    }
    return rc;
}

int numeric_export_L(const sc_numeric *h, double *out) {
    const sc_symbolic *s = h->sym;
    if (h->last_stream) SC_CUDA(cudaStreamSynchronize(h->last_stream));
    std::vector<unsigned char> buf((size_t)s->lnz_size * h->elt);
    SC_CUDA(cudaMemcpy(buf.data(), h->d_lnz, buf.size(), cudaMemcpyDeviceToHost));
    int64_t o = 0;
    for (int64_t J = 0; J < s->nsuper; J++) {
        int32_t w = s->sup_ptr[J + 1] - s->sup_ptr[J];
        int64_t m = s->gl_ptr[J + 1] - s->gl_ptr[J];
        for (int64_t r = 0; r < m; r++)
            for (int32_t c = 0; c < w; c++) {
                int64_t e = s->lnz_off[J] + r * s->lnz_ld[J] + c;
                double v = h->elt == 8 ? ((const double *)buf.data())[e] : (double)((const float *)buf.data())[e];
                out[o++] = r >= c ? v : 0.0;
            }
    }
    return SC_OK;
}

bool drop_slices(sc_numeric *h) {
    if (!h->d_slices) return false;
    if (h->gexec) cudaGraphExecDestroy(h->gexec);
    h->gexec = nullptr;
    cudaFree(h->d_slices);
    h->d_slices = nullptr;
    h->device_bytes -= h->slice_bytes;
    return true;
}

void numeric_free(sc_numeric *h) {
    if (!h) return;
    if (h->gexec) cudaGraphExecDestroy(h->gexec);
    for (auto &g : h->sg)
        if (g) cudaGraphExecDestroy(g);
    if (h->cap_stream) cudaStreamDestroy(h->cap_stream);
    if (h->cap_stream2) cudaStreamDestroy(h->cap_stream2);
    if (h->cap_stream3) cudaStreamDestroy(h->cap_stream3);
    for (cudaEvent_t e : {h->ev_fork, h->ev_join, h->ev_trsm, h->ev_rest[0], h->ev_rest[1]})
        if (e) cudaEventDestroy(e);
    void *ptrs[] = {h->d_lnz, h->d_pool, h->d_valmap, h->d_values, h->d_diagpos, h->d_adiag, h->d_info,
                    h->d_chunks, h->d_potrf, h->d_trsm, h->d_gemm, h->d_small, h->d_tasks, h->d_rlpairs,
                    h->d_rlslabs, h->d_rlrelind, h->d_glbind, h->d_perm, h->d_csr_ptr, h->d_csr_col, h->d_csr_val,
                    h->d_csr_map, h->d_counters, h->d_xw, h->d_solve_tiles, h->d_sn, h->d_blk, h->d_rbval,
                    h->d_loops, h->d_tmaps, h->d_tmap_of_sn, h->d_err, h->d_inv, h->d_x, h->d_r, h->d_b, h->d_xbest, h->d_y, h->d_z, h->d_acc, h->d_red,
                    h->d_dep_ptr, h->d_dep, h->d_sync, h->d_serr, h->d_hi, h->d_lo, h->d_thin,
                    h->d_cgz, h->d_cgp, h->d_cgq, h->d_cgs, h->d_solve_units, h->d_flow, h->d_flow_ctr,
                    h->d_flow_need, h->d_task_chunk, h->d_sn_chunk, h->d_splits, h->d_split_units, h->d_split_of_task,
                    h->d_slices, h->d_exps, h->d_slice_maps, h->d_inv_exp, h->d_chunk64, h->d_row_blk};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (h->sym) h->sym->refs--;
    delete h;
}

}  // namespace sc
