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
// Bytes of partial sums, fp32 [tile][part][16][columns of a tile].  (A tile is whole also where lr_cols is no multiple of its columns.)
inline size_t lowrank_split_bytes(int64_t M, int lr_cols) {
    const int64_t tiles = lowrank_tiles(M, lr_cols);
    return tiles <= kLrSplitTiles ? (size_t)tiles * kLrKSplitMax * kLrTileTok * lowrank_tile_cols(M) * 4 : 0;
}

}  // namespace bwla
