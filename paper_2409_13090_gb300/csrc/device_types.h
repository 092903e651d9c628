// Plain data types shared by the host launch plan and the device kernels.
#pragma once
#include <cstdint>

#include "sc_internal.h"

namespace sc {

// Per-chunk data needed on the device.
struct ChunkDev {
    int64_t off;   // offset of the supernode's panel
    int64_t gl;    // offset of glbind(J)
    int64_t inv;   // offset of the chunk's w x w diagonal-block inverse (FP32 / TF32 factors)
    int32_t ld;    // panel leading dimension
    int32_t m;     // rows of the panel (m_J)
    int32_t c0;    // first local column of the chunk
    int32_t w;     // chunk width
    int32_t col0;  // global column of the chunk's first column
    int32_t slot;  // FP64: offset of the chunk's digits (chunk64.cuh)
};

// One tile of the row-wise TRSM: rows [r0, min(r0+rows, m)) of chunk c.
struct TrsmTile {
    int32_t chunk, r0;
};

// What a CTA of a persistent solve sweep takes at once: tile t0 alone (cnt 0:
// the first tile of a wide chunk), narrow tiles t0 .. t0 + cnt - 1, one per
// warp (cnt 1..8), or -cnt further tiles t0 .. t0 - cnt - 1 of one wide chunk,
// one after another (cnt -1..-solve_group, a launch-plan setting).
struct SolveUnit {
    int32_t t0, cnt;
};

// One output tile of a product task. ks < 0: the whole inner dimension;
// ks >= 0: only its slice [ks * S, (ks + 1) * S), added atomically, with
// S = kSplitKCrit for a critical task and kSplitK otherwise (SIMT tiles of
// critical tasks, and of tasks with few tiles and a long inner dimension).
struct GemmTile {
    int32_t task, tm, tn, ks;
};
constexpr int kSplitK = 256;
constexpr int kSplitKCrit = 32;  // slice width of split critical tasks (kTaskCrit)

// Work of one CTA of the thin-product kernel: warp blocks blk0 .. blk0 + 3 of
// a task (blocks numbered row-major over the task's NI x NJ block grid).
struct ThinUnit {
    int32_t task, blk0;
};
constexpr int kThinWarps = 4;

// Warp-block shape for a rows x nb product: the NI in {ni_min, ..., 8}
// (powers of two; NJ = 32 / NI) with the fewest blocks, ties to the smaller
// NI + NJ (fewer loads per step). Lower (triangular) products use 4 x 8.
SC_HD inline int block_rows(int rows, int nb, int ni_min, bool lower) {
    if (lower) return 4;
    int best = ni_min, bestn = 1 << 30;
    for (int ni = ni_min; ni <= 8; ni *= 2) {
        const int nj = 32 / ni;
        const int cnt = ((rows + ni - 1) / ni) * ((nb + nj - 1) / nj);
        if (cnt < bestn || (cnt == bestn && ni + nj < best + 32 / best)) {
            best = ni;
            bestn = cnt;
        }
    }
    return best;
}

constexpr int kMaxChunk = 64;
// Loop items of narrow supernodes of a level from which a warp takes one. FP64 factorizations at
// 304 / 1216 / 4864: 64^2 0.491 / 0.503 / 0.504 ms, 300 x 280 2.44 / 2.38 / 2.40, 48^3 16.28 / 16.29 / 16.21,
// 37x41x29 graph-ordered 7.86 / 7.82 / 7.71, 24x22x25 27-point 3.41 / 3.27 / 3.19.
constexpr int kLoopMinWarps = 1216;
// Small chunks of a level from which FP64 takes them by warps. At 256 / 1024 / 4096: 300 x 280 2.36 /
// 2.38 / 2.63 ms, 64 2D matrices 3.65 / 3.64 / 3.68, 48^3 and the others within 0.1 %.
constexpr int kNarrowMin64 = 1024;

// FP64 POTRF to TRSM: 256-word units of a chunk's digits -- L_cc, the inverses of its
// 16 x 16 diagonal blocks, exponents.
SC_HD inline int chunk64_units(int w) {
    const int nb = (w + 15) / 16;
    return nb * nb + nb + 1;
}
constexpr int kTrsm64Rows = 64;
constexpr int kNarrowChunk = 16;  // solve tiles of chunks up to this width take a warp, wider ones a CTA

// Is a chunk of w columns and `rows` rows below factored by one warp (k_narrow)?
// FP32: up to 16 columns and 128 rows. FP64, where a warp's multiply-add takes 64 clocks:
// while it has at most 200 of them in line (7 us; the CTA-wide POTRF and TRSM
// take some 32 us in two launches) -- w^2 / 2 + 6 w for the pivots and w^2 / 2 for 32 rows.
// With the line at 100 / 200 / 400: 300 x 280 2.46 / 2.38 / 2.32 ms, 64 2D matrices 4.00 / 3.64 / 3.59, the
// 3D ones within 0.1 %.
SC_HD inline bool narrow_chunk(int w, int rows, bool fp64) {
    if (w > kNarrowChunk || rows > 128) return false;
    return !fp64 || w * w / 2 * (1 + (rows + 31) / 32) + 6 * w <= 200;
}

// Supernode descriptor for the device-side RLB loops.
struct SnDev {
    int64_t off;  // offset of Lnz(J)
    int32_t ld;   // leading dimension of Lnz(J)
    int32_t m;    // m_J = |glbind(J)|
    int32_t f;    // first column
    int32_t n;    // |J|
    int32_t b1;   // one past J's last block
    int32_t pad;
    int64_t gl;   // offset of glbind(J)
};

// Block descriptor (Sec. 1 / Alg. 5): rows pos..pos+size-1 of Lnz(J) hold the
// global rows first..first+size-1, which are columns of supernode owner.
// relindB(J, owner) starts at rb_val[rb] and covers J's blocks bs.. onward.
struct BlkDev {
    int32_t pos, size, first, owner;
    int64_t rb;
    int32_t bs, pad;
};

// Source block of FP64 products on the tensor cores (split_gemm.cuh): rows
// row0 .. row0 + rows - 1 and columns kx0 .. kx0 + k - 1 of a panel, cut into FP16
// slices in the level's half of the slice pool.
struct SplitBlk {
    int64_t src;     // offset of (row0, kx0) in the factor storage
    int64_t piece0;  // first row of the slice pool (rows of 32 values)
    int32_t ld, rows, k, row0;
    int32_t exp0;    // first row exponent
    int32_t pad;
};
// 64 rows of a source block: the work of one CTA of the splitting kernel.
struct SplitUnit {
    int32_t blk, row0;
};
constexpr int kSplitRows = 64;

constexpr int kLoopSmemBytes = 48 * 1024;

// Target-owned RL assembly (deterministic plans): rows [row0, row1) of Lnz(P)
// receive the update matrices of pairs pair0 .. pair0 + npairs - 1 (all with
// target P, in the order of their source supernodes) from one CTA.
struct RLSlab {
    int32_t pair0, npairs, row0, row1;
};
constexpr int kRLSlabRows = 64;

// One unit of the per-level persistent kernel (k_level): a POTRF of a chunk, a
// TRSM tile, a product tile, one or two thin units, up to eight small tasks, a
// device-loop item or up to eight narrow loop items. idx indexes the list of
// its kind (for small tasks and narrow loop items: the first of cnt entries).
struct FlowUnit {
    int32_t kind, idx, cnt, pad;
};
enum : int32_t { kFlowPotrf = 0, kFlowTrsm, kFlowGemm, kFlowThin, kFlowSmall, kFlowLoop, kFlowLoopW };
// one counter word per 128-byte line in the per-chunk arrays of k_level
constexpr int kFlowStride = 32;

}  // namespace sc
