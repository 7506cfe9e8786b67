// Sizes and splits that the host decides before a launch, in plain C++ so that they can be checked without a GPU
// (tests/test_host_plans.py walks them over every size the entry points accept).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace bwla {

constexpr int kLowrankPad = 64;          // T is kept as bf16 [3][M][64] (T = hi + mid + lo), zero beyond r <= 64

#ifdef __CUDACC__
#define BWLA_HOST_DEVICE __host__ __device__
#else
#define BWLA_HOST_DEVICE
#endif
BWLA_HOST_DEVICE inline int lowrank_cols(int r) { return r > kLowrankPad ? (r + 1) / 2 * 2 : kLowrankPad; }

// ---- T = V x by the mma.sync blocks beside the rotation (prologue_roles.cuh) ----
// With few tokens V is read by several blocks that each take a part of K; their partial sums of T meet in the workspace and
// the last block to arrive adds them in a fixed order (counters: status words 4..11, one per tile of T).
constexpr int kLrKSplitMax = 16;
constexpr int kLrSplitTiles = 8;
constexpr int kLrTileTok = 16;           // tokens of a tile

inline int lowrank_tile_cols(int64_t M) { return M > 32 ? 32 : 16; }
inline int64_t lowrank_tiles(int64_t M, int lr_cols) {
    const int cols = lowrank_tile_cols(M);
    return ((lr_cols + cols - 1) / cols) * ((M + kLrTileTok - 1) / kLrTileTok);
}
// Parts of K a tile is split into, given the warps of a block: so many that a warp has about as many chunks of 32 as it can request
// at once (a block that read all of V alone would stream it, cold, through one SM).  1 where there are more tiles than counters.
inline int lowrank_ksplit(int64_t M, int64_t K, int lr_cols, int warps) {
    if (lowrank_tiles(M, lr_cols) > kLrSplitTiles) return 1;
    const int64_t per = warps * (lowrank_tile_cols(M) == 32 ? 2 : 4);
    return (int)std::min<int64_t>(kLrKSplitMax, std::max<int64_t>(1, (K / 32 + per / 2) / per));
}
// Bytes of partial sums, fp32 [tile][part][16][columns of a tile], that M tokens or any smaller number need: a workspace made for
// M tokens serves fewer.  (A tile is whole also where lr_cols is no multiple of its columns.)
inline size_t lowrank_split_bytes(int64_t M, int lr_cols) {
    size_t most = 0;
    for (int64_t t = kLrTileTok; t < M + kLrTileTok && t <= kLrSplitTiles * kLrTileTok; t += kLrTileTok) {
        const int64_t tiles = lowrank_tiles(t, lr_cols);
        if (tiles <= kLrSplitTiles) most = std::max(most, (size_t)tiles * kLrKSplitMax * kLrTileTok * lowrank_tile_cols(t) * 4);
    }
    return most;
}

// ---- T = V x for many tokens on tcgen05 (lowrank_umma.cu) ----
constexpr int kLruTok = 128, kLruCols = 64, kLruBlockK = 64;        // tokens and columns of a tile, values of k per stage
constexpr int kLruMaxParts = 16;         // parts of K per token tile
constexpr int kLruTargetCtas = 160;      // parts are chosen so that tiles x parts comes near this, every part at least eight stages long
inline int64_t lowrank_umma_tiles(int64_t M) { return (M + kLruTok - 1) / kLruTok; }
inline int lowrank_umma_parts(int64_t M, int64_t K) {
    int64_t ks = std::max<int64_t>(1, kLruTargetCtas / lowrank_umma_tiles(M));
    ks = std::min<int64_t>(ks, kLruMaxParts);
    return (int)std::min<int64_t>(ks, std::max<int64_t>(1, K / (8 * kLruBlockK)));
}
// (from 50 tokens where the rotation of a token takes a cluster of three, 160 x 160: it goes to rot_umma.cu then, which has no
// blocks for T beside it)
inline bool lowrank_umma_supports(int64_t M, int64_t K, int r) {
    return (M > 64 || (K > 128 * 128 && 3 * M > 148)) && r > 0 && r <= kLruCols && K % kLruBlockK == 0;
}
// Bytes of its partial sums.  They lie where the rotation that follows it leaves the codes (or the rotated values) and are never
// larger than those: 256 bytes a column of 128 tokens against 128 values of K / 512 parts at the least.
inline size_t lowrank_umma_part_bytes(int64_t M, int64_t K, int r) {
    if (!lowrank_umma_supports(M, K, r)) return 0;
    const int ks = lowrank_umma_parts(M, K);
    return ks > 1 ? (size_t)lowrank_umma_tiles(M) * ks * kLruCols * kLruTok * 4 : 0;
}

// ---- the weight-only operating point ----
// Up to how many tokens it runs on three int8 digits per value (gemm_small.cu)
constexpr int kDigitTokens = 32;
constexpr int kQsumParts = 8;            // partial sums a token's code sum is kept as (one per CTA of its cluster)
// bf16 values, or three digits of few tokens, and the sums of either: never less than fewer tokens need
inline size_t a16_value_bytes(int64_t M, int64_t K) { return std::max((size_t)(M * K * 2), (size_t)(std::min<int64_t>(M, kDigitTokens) * K * 3)); }
inline size_t a16_sum_bytes(int64_t M) { return std::max((size_t)M * 4, (size_t)std::min<int64_t>(M, kDigitTokens) * 3 * kQsumParts * 4); }

}  // namespace bwla
