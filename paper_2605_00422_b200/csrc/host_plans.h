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

// (beyond 64 tokens K is not split, and narrow tiles fill more SMs)
inline int lowrank_tile_cols(int64_t M) { return M > 32 && M <= 64 ? 32 : 16; }
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
// Up to eight are added up in a cluster's shared memory; more, which a second kernel adds, only for a K above kLruClusterK: a call of 129 | 333
// tokens, rank 64, 5120 outputs, us, eight in a cluster and up to sixteen apart: K = 8192 40.2, 40.8 | 44.6, 45.4; 11008 49.5, 49.9 | 54.4, 53.7; 12288 50.6, 50.7 |
// 57.7, 56.3; 13824 58.2, 57.3 | 61.9, 59.7; 25600 94.3, 90.0 | 118.3, 113.4 (1024 tokens: 108.8, 110.6 at 11008, 126.2, 127.0 at 13824, 262, 259 at 25600).
constexpr int kLruClusterParts = 8;
constexpr int kLruClusterK = 12288;
constexpr int kLruTargetCtas = 160;      // parts are chosen so that tiles x parts comes near this, every part at least eight stages long
inline int64_t lowrank_umma_tiles(int64_t M) { return (M + kLruTok - 1) / kLruTok; }
inline int lowrank_umma_parts(int64_t M, int64_t K) {
    const int64_t tiles = lowrank_umma_tiles(M);
    int64_t ks = std::min<int64_t>(std::max<int64_t>(1, kLruTargetCtas / tiles), kLruMaxParts);
    ks = std::min<int64_t>(ks, std::max<int64_t>(1, K / (8 * kLruBlockK)));
    if (ks > kLruClusterParts && K <= kLruClusterK) ks = kLruClusterParts;
    return (int)std::min<int64_t>(ks, std::max<int64_t>(1, M * K / (tiles * kLruCols * kLruTok * 4)));      // (their room: below)
}
// Which problems it takes; which of them go to it, launch_rot decides.
inline bool lowrank_umma_supports(int64_t K, int r) { return r > 0 && r <= kLruCols && K % kLruBlockK == 0; }
// Bytes of its partial sums.  They lie where the rotation that follows it leaves the codes (or the rotated values) and are never
// larger than those.
inline size_t lowrank_umma_part_bytes(int64_t M, int64_t K) {
    const int ks = lowrank_umma_parts(M, K);
    return ks > 1 ? (size_t)lowrank_umma_tiles(M) * ks * kLruCols * kLruTok * 4 : 0;
}

// ---- rotation + quantiser on mma.sync (rot_mma.cu) ----
constexpr int kRotMaxWarps = 16;          // per CTA
constexpr int kRotMaxSmem = 232448 - 128; // the 227 KB a block may have, less the static shared memory of the roles
constexpr int kRotHeader = 256;           // prepared factors: exponents, then the terms
constexpr int kRotRedBytes = 3072;        // per group: RotShared

// Geometry of the kernel for one pair of Kronecker factor sizes; computed on the host, passed to the kernels by value.
struct RotGeom {
    int n1, n2, K;
    int n2p;                // n2 rounded up to 16
    int na;                 // 8-column tiles of a and c: n1 rounded up to 16, in eighths
    int cw, ntw;            // warps the column tiles are dealt to (1, 2 or 4), tiles per warp
    int dtc, dc;            // 16-row tiles of d per CTA, CTAs per token (cluster size, up to 8)
    int warps;              // warps of one token in a CTA: a group
    int max_groups;         // groups a CTA can hold
    int s2, s1;             // bytes per row of operands contracted over b / over a
    int p1_off, group_off, group_bytes;     // shared memory: P2^T terms at 0, P1^T terms, then per group
    int z_rel, red_rel;                     // ... x at 0, Z^T, RotShared
    int alias_z;            // Z^T takes the place of x
    int pad;                // bytes added to every row against bank conflicts
};
inline int round_to(int v, int m) { return (v + m - 1) / m * m; }

// A warp may have ntw column tiles at most; `alias`: Z^T takes the place of x, which is dead by then (the next token's x then
// arrives late, which costs about a fifth).  Fills in what follows from dc and alias; false when it does not fit.
inline bool rot_layout(RotGeom& g, int dc, int alias, int pad) {
    const int tiles = g.n2p / 16;
    g.dtc = (tiles + dc - 1) / dc;
    g.warps = g.dtc * g.cw;
    if (g.warps > kRotMaxWarps || (dc - 1) * g.dtc >= tiles || dc * g.warps > 64) return false;
    // Rows of an odd number of 16-byte chunks (pad 16): the eight rows of an ldmatrix then fall into different banks.  The
    // largest factors only fit without that padding, and without the rows of x beyond n1.
    g.pad = pad;
    g.s2 = g.n2p * 2 + pad; g.s1 = g.na * 16 + pad;
    const int x = (pad ? g.cw * g.ntw * 8 : g.n1) * g.s2, z = g.cw > 1 ? 2 * g.dtc * 16 * g.s1 : 0;
    g.dc = dc; g.alias_z = alias;
    g.p1_off = 3 * g.dtc * 16 * g.s2;
    g.group_off = g.p1_off + 2 * g.na * 8 * g.s1;
    // (a warp's column tiles beyond n1 are read all the same and dropped: they must lie inside the block, 180 x 136)
    g.group_bytes = std::max((alias ? std::max(x, z) : x + z) + kRotRedBytes, g.cw * g.ntw * 8 * g.s2);
    g.z_rel = alias ? 0 : x; g.red_rel = g.group_bytes - kRotRedBytes;
    if (g.group_off + g.group_bytes > kRotMaxSmem) return false;
    g.max_groups = dc == 1 ? std::min(std::min(kRotMaxWarps / g.warps, 8), (kRotMaxSmem - g.group_off) / g.group_bytes) : 1;   // (barriers 1..8)
    return true;
}

// Chooses the split of a token over warps and CTAs: the one that keeps most warps busy on an SM (16 is what the registers
// allow), counting that the last CTA of a cluster may have fewer rows.
inline bool rot_geometry(int n1, int n2, RotGeom* out) {
    if (n1 < 1 || n2 < 8 || n2 % 8 != 0 || n2 > 256 || n1 > 192) return false;
    RotGeom g{};
    g.n1 = n1; g.n2 = n2; g.K = n1 * n2;
    g.n2p = round_to(n2, 16); g.na = round_to(n1, 16) / 8;
    g.cw = g.na <= 8 ? 1 : g.na <= 16 ? 2 : 4;
    g.ntw = (g.na + g.cw - 1) / g.cw;                         // (the last warp may have tiles beyond na, which it ignores)
    double best = 0.0;
    for (int pad = 16; pad >= 0 && best == 0.0; pad -= 16)
        for (int dc = 1; dc <= 8; ++dc)
            for (int alias = 0; alias <= (g.cw > 1 ? 1 : 0); ++alias) {
                RotGeom t = g;
                if (!rot_layout(t, dc, alias, pad)) continue;
                const int ctas = dc == 1 ? 1 : std::min(kRotMaxWarps / t.warps, (kRotMaxSmem + 1024) / (t.group_off + t.group_bytes + 1024));
                const double score = (double)(g.n2p / 16) * g.cw / dc * t.max_groups * ctas * (alias ? 0.8 : 1.0);
                if (score > best * 1.001) { best = score; *out = t; }
            }
    return best != 0.0;
}

// Few tokens: what counts is the time of one token, so it is spread over more warps (up to 64 columns: two warps instead of
// one) and over more CTAs: MMAs of a CTA at 2 cycles each, against about 5000 cycles for the cluster's barriers and its later start
// (64 x 128, one token: 6.7 us on eight CTAs, 5.2 on one).  `resident(geometry)`: every token finds a cluster at once; false when no
// split has that (a second round of clusters doubles the time: 128 x 128, 16 tokens in clusters of eight 23.6 us).  `raw`: every CTA
// splits all of P1 and its rows of P2 first, a pair of values in about 220 cycles a thread (one token of 108 x 128: 23 us on two warps in
// each of eight CTAs, 14 on sixteen warps in one).
template <typename Resident>
inline bool few_tokens_geometry(const RotGeom& base, bool raw, RotGeom* out, Resident resident) {
    double best_cost = 0.0;
    const int ksteps = base.n2p / 16 + base.na / 2;
    for (int dc = 1; dc <= 8; ++dc) {
        RotGeom t = base;
        if (t.na > 4 && t.na <= 8) { t.cw = 2; t.ntw = 4; }
        if (!rot_layout(t, dc, 0, base.pad) && (t.cw == 1 || !rot_layout(t, dc, 1, base.pad))) continue;
        const int pairs = t.dtc * 8 * t.n2p + 32 * t.na * t.na;
        const double cost = 2.0 * 3.0 * t.dtc * t.na * ksteps + (dc > 1 ? 5000.0 + 300.0 * dc : 0.0) + (raw ? 220.0 * pairs / (32 * t.warps) : 0.0);
        if ((best_cost == 0.0 || cost < best_cost) && resident(t)) { best_cost = cost; *out = t; }
    }
    return best_cost != 0.0;
}

inline size_t rot_prepared_bytes(const RotGeom& g) {
    return kRotHeader + (size_t)3 * g.n2p * g.s2 + (size_t)2 * g.na * 8 * g.s1;
}

// ---- which kernel rotates many tokens (more than the device holds clusters for) ----
// The kernel alone, us at 150, 1024 and 4096 tokens of one linear, and the error of 300 tokens against 64 bits in 1e-7 of a row's 2-norm:
//                the other kernel                   rot_rows.cu
//    48 x  64    13    21    46   1.35   rot_mma    13    19    41   1.34
//    64 x  64    15    25    58   1.40   rot_mma    13    19    42   1.38
//    64 x  80    17    33    86   1.43   rot_mma    13    21    50   1.40
//    64 x 128    19    36    93   1.59   rot_umma   15    25    68   1.55
//    86 x 128    21    44   137   2.45   okt_umma   17    36   113   1.83
//   108 x 128    23    52   166   2.48   okt_umma   17    38   117   1.89
//   128 x 128    23    50   162   2.64   okt_umma   19    39   124   1.9
// rot_rows.cu where it can (n1 in (32, 128], n2 a multiple of 16 up to 128) and is the faster one (rot_rows_faster).  For the rest: mma.sync where one warp holds all columns of
// a token and a CTA several tokens; okt_umma.cu for 81 to 128 columns, where a step of rot_umma.cu would hold one token in half of its
// columns, and for n2 that is no multiple of 16; rot_umma.cu (160 x 160: 100 | 296 us at 150 and 1024 tokens on mma.sync, 81 | 156 here).
// (As many tokens as the device holds at once stay on mma.sync, 1.45e-7 for every size: rot_rows.cu has 86 x 128 in 14.6 us of a call for
// one token's 17.6, but 1.8e-7.)
// With T = V x as blocks of the same launch (up to 64 tokens of several linears, or ranks that lowrank_umma.cu does not take) the kernel before was
// rot_mma.cu unless okt_umma.cu took the factors, and its error is smaller beyond 80 columns or 64 rows (64 x 128: 1.44, 72 x 96: 1.49): they stay
// there (rot_rows_exact).
inline bool rot_mma_always(const RotGeom& g) { return g.cw == 1 && g.n2p <= 80; }
inline bool rot_okt_factors(const RotGeom& g) {
    return !rot_mma_always(g) && g.na <= 16 && g.n2 <= 128 && (g.na > 10 || g.n2 % 16 != 0);
}

// Whether rot_rows.cu's error is no larger than that of the kernel these factors would go to otherwise.  beside: T in the same launch.
inline bool rot_rows_exact(const RotGeom& g, bool beside) { return !beside || rot_mma_always(g) || rot_okt_factors(g); }
// Whether it is the faster one for more tokens than rot_mma.cu has places for at once; t: tokens x linears.  A step of rot_rows.cu takes its time
// whatever n1 and n2 are, and all SMs take a multiple of two tokens (n1 <= 64), so that it pays where the lanes are full and either the first
// step or many steps count.  A call with it in percent of a call with the other kernel (1536 outputs, one linear, r = 0; calls repeat to 1 %):
//     tokens          149 185 200 260 296 333 400 450 512 600 1024 2048
//    64 x 64           91  90 100  96 100 104 100 100  96  87   89   85        rank 32      96  96  99  99  99 100  98  98  96  88   91   87
//    64 x 64, raw      93  91  97 101 106 108  93  95  92  93   88   86        bf16 values  90  93  97  93  94  97  98  95  96  86   90   86
//    64 x 80           96  95  97  99  99 101  97  83  84  85   81   79        rank 32      98  97  98  99 100  98  96  86  86  84   83   81
//    64 x 80, raw      98  97  98  96  95 110  93  92  92  96   87   81        bf16 values 102 101 101 101 102 108 107  93  93 101   99   95
//    48 x 64           99  97 108 106 108 115 107 108 104  97  100   98        48 x 80     102 102 104 105 105 112 104  95  95  96   95   93
//    72 x 96          104 104 103  99 103  97  99 104 102  99  100  103        80 x 64     101 101 101  98 101  90  90  95  94  89   91   92
//    64 x 96           98  98  99  96  99  91  93  93  92  90   85   83        48 x 48, 64 x 48, 64 x 32: 100 to 145 up to 600 tokens
// (64 x 128 and more than 80 rows: 67 to 100.  With T beside, three linears of 64 x 64 and 64 tokens take 108 % of the time; without 95.)
// t_first: T = V x in a launch of its own before.
inline bool rot_rows_faster(const RotGeom& g, bool values, bool raw, bool beside, bool t_first, int64_t t, int sms) {
    if (rot_mma_always(g)) {
        if (g.n1 < 48 || g.n2 < 64) return false;          // (36 x 80 has 1.45e-7 here and 1.44e-7 on rot_mma.cu)
        if (values) return g.n2 % 32 == 0 ? g.K >= 4096 || t > 4 * sms : g.K >= 5120 && t > 3 * sms;
        if (g.K < 4096) return t > (g.n2 >= 80 ? 3 : 4) * sms;
        if (beside && g.K < 5120) return 4 * t <= 5 * sms;
        return t_first || 2 * t > 5 * sms || 4 * t <= (raw ? 7 : 8) * sms;
    }
    if (g.n1 > 64 && !rot_okt_factors(g)) return (values || g.n2 <= 80) && 2 * t > 3 * (int64_t)sms;
    return true;
}
// The same for t tokens that rot_mma.cu has places for (on `few_sms` SMs), raw factors.  It is the faster one by 5 to 10 % unless its blocks do not
// find SMs beside those of the contraction behind it (`behind`), as which the call after it takes 4 to 6 us more; rot_rows.cu has half
// as many.  us, rot_mma.cu | rot_rows.cu, 64 x 80 to 4096 outputs (128 blocks): 20 tokens 14.6 | 16.9, 25 20.2 | 16.5, 40 20.9 | 17.2, 64 22.2 | 21.3; to
// 4700 (148 blocks): 25 tokens 21.8 | 22.4; to 8192 (64 blocks): 80 tokens 25.2 | 27.9, 100 31.4 | 27.9, 128 31.3 | 27.9.  64 x 64 to 5120, 4 tokens
// (148 blocks): 15.5 | 13.7.  With t_first most of it is hidden up to one tile of 128 tokens (64 x 80 to 5120, 128 tokens 101 %, 140 92 %).
inline bool rot_rows_crowded(const RotGeom& g, bool t_first, int64_t t, int few_sms, int behind, int sms) {
    if (!rot_mma_always(g) || g.n1 < 48 || g.n2 < 64 || t < 3 || behind == 0) return false;
    if (behind + few_sms <= sms || (t_first && (g.K < 5120 || t <= 128))) return false;
    return t <= 16 || t > 64 || (behind < sms - 2 && behind + (t + 1) / 2 <= sms + 24);
}

// ---- rotation of many tokens on tcgen05 (rot_umma.cu) ----
constexpr int kRotUmmaSharedBytes = 1792;      // its barriers and small per-CTA state
struct RotUmmaGeom {
    int n1, n2, K;
    int nc;                 // columns of a token's Y: n1 rounded up to 16
    int np;                 // columns of a token in the accumulators
    int tps, ntot;          // tokens of a step, tps * np
    int dc, dt;             // CTAs of a token, rows d of each
    int atoms2, atoms1;     // K atoms of 32 elements over b / over a
    int xb;                 // buffers of x
    int staged;             // outputs of a step go through shared memory (two buffers of out_bytes)
    int out_bytes;
    int p1_off, x_off, st_off, sh_off, total;
    int s2, s1;             // row strides of the prepared factors
};

// False when the sizes are outside what the kernel takes: whole 16-byte pieces of the codes' order (n2 a multiple of 16), three
// times n1 columns of tensor memory, at most 128 rows and the factors' terms in the shared memory of one CTA or of two; both
// contractions at least two steps of 16 values deep (the second chain of sums would have none).
inline bool rot_umma_geometry(const RotGeom& g, int out_size, RotUmmaGeom* out) {
    if (g.n2 % 16 != 0 || g.n2 < 32 || g.na < 4 || g.n1 > 160) return false;
    RotUmmaGeom u{};
    u.n1 = g.n1; u.n2 = g.n2; u.K = g.K; u.s2 = g.s2; u.s1 = g.s1;
    u.nc = g.na * 8;
    u.tps = u.nc <= 32 ? 4 : u.nc <= 80 ? 2 : 1;
    u.np = u.tps == 1 ? (u.nc + 31) / 32 * 32 : u.nc;
    u.ntot = u.tps * u.np;
    u.atoms2 = (g.n2 + 31) / 32; u.atoms1 = (u.nc + 31) / 32;
    for (u.dc = 1; u.dc <= 2; ++u.dc) {
        u.dt = u.dc == 1 ? g.n2 : (g.n2 / 2 + 15) / 16 * 16;
        if (u.dt > 128) continue;
        // Outputs of whole tokens are contiguous: they are staged where two buffers fit, at the price of the second x if need
        // be (stored from registers, a sector of 32 bytes is written in two or four pieces: 64 x 80, 4096 tokens 54 us).
        for (int option = u.dc == 1 ? 0 : 2; option < 4; ++option) {
            u.xb = 2 - (option & 1);
            u.staged = option < 2;
            u.out_bytes = u.tps * u.K * out_size;
            u.p1_off = 3 * u.atoms2 * u.dt * 64;
            u.x_off = u.p1_off + 2 * u.atoms1 * u.nc * 64;
            u.st_off = u.x_off + u.xb * u.atoms2 * u.ntot * 64;
            u.sh_off = (u.st_off + (u.staged ? 2 * u.out_bytes : 0) + 127) / 128 * 128;
            u.total = u.sh_off + kRotUmmaSharedBytes;
            // (an MMA reads 128 rows from the first row of any block of P2's terms)
            if (u.total <= kRotMaxSmem && u.p1_off - u.dt * 64 + 128 * 64 <= u.total) { *out = u; return true; }
        }
    }
    return false;
}

// ---- rotation of many tokens on tcgen05, output rows on the lanes (rot_rows.cu) ----
constexpr int kRotRowsSharedBytes = 2048;      // its barriers and small per-CTA state
struct RotRowsGeom {
    int n1, n2, K;
    int lanes, tps;         // tensor-memory lanes of a token (n1 rounded up to 64 or 128), tokens of a step
    int groups, chunks;     // warps the columns are dealt to in every lane quarter, 16-column chunks of a warp
    int nv;                 // accumulators for the first contraction
    int y_chains;           // chains of sums of the second
    int ks1, ks2;           // steps of 16 over a and over b
    int atoms1, atoms2;     // K atoms of 32 elements
    int xb;                 // buffers of x
    int staged, out_bytes;  // outputs of a step go through shared memory (two buffers of out_bytes)
    int p1_off, x_off, st_off, sh_off, total;   // the terms of P2^T at 0
};
// What follows the factors, with xb buffers of x.
inline bool rot_rows_places(RotRowsGeom& g, int xb, int x_terms) {
    g.xb = xb;
    g.st_off = g.x_off + xb * x_terms * g.atoms2 * 128 * 64;
    g.sh_off = (g.st_off + (g.staged ? 2 * g.out_bytes : 0) + 127) / 128 * 128;
    g.total = g.sh_off + kRotRowsSharedBytes;
    return g.total <= kRotMaxSmem;
}
// n1 in (32, 128] on the lanes; n2 a multiple of 16 up to 128: two accumulators for either contraction fill four (or six, up to 80
// columns: two steps' V) times n2 columns of tensor memory.  A third chain of Y lies where V was, so that with one V the next step's V waits for it:
// two chains for codes from 81 rows on, where okt_umma.cu was before (108 x 128, 4096 tokens: 121 us with three chains, 117 with two, 1.73e-7 and
// 1.89e-7, 2.48e-7 there), three where rot_umma.cu was: bf16 values, whose error was 1.87e-7 there, and fewer rows (80 x 128: 1.84e-7 with two, 1.78e-7).  x_terms: 3 where rows are fp32.
inline bool rot_rows_geometry(int n1, int n2, int out_size, RotRowsGeom* out, int x_terms = 1) {
    if (n2 % 16 != 0 || n2 < 32 || n2 > 128 || n1 <= 32 || n1 > 128) return false;
    RotRowsGeom g{};
    g.n1 = n1; g.n2 = n2; g.K = n1 * n2;
    g.lanes = n1 <= 64 ? 64 : 128; g.tps = 128 / g.lanes;
    g.chunks = n2 <= 80 ? 1 : 2; g.groups = (n2 + 16 * g.chunks - 1) / (16 * g.chunks); g.nv = n2 <= 80 ? 2 : 1;
    g.ks1 = (n1 + 15) / 16; g.ks2 = n2 / 16;
    g.y_chains = g.ks2 == 2 || (g.nv == 1 && n1 > 80 && out_size == 1) ? 2 : 3;
    g.atoms1 = (n1 + 31) / 32; g.atoms2 = (n2 + 31) / 32;
    // Rows of a whole number of 32 outputs leave in 16-byte pieces from registers; others (half of a group of the codes' order would be
    // two bytes of every four) through shared memory.
    g.staged = n2 % 32 != 0;
    g.out_bytes = g.tps * g.K * out_size;
    g.p1_off = 2 * g.atoms2 * n2 * 64;         // (an MMA of the step's second token reads from 64 rows before P1's terms)
    g.x_off = g.p1_off + 3 * g.atoms1 * g.lanes * 64;
    for (int xb = x_terms == 1 ? 2 : 1; xb >= 1; --xb)
        if (rot_rows_places(g, xb, x_terms)) { *out = g; return true; }
    return false;
}
// Whether rows of weights are binarised there and not by rot_mma.cu: up to 80 columns (its error is smaller then), more rows than half of the SMs, and
// factors for which a step, whose time does not depend on n1, is the shorter one.  us of 4000 to 5120 rows, rot_mma.cu | rot_rows.cu, fp32 and bf16:
//    64 x 64  94 |  85   64 | 51      64 x 48  76 | 75   55 | 45      48 x 48  58 | 70   42 | 43      64 x 32  49 | 66   36 | 39
//    64 x 80 187 | 128  117 | 73      56 x 64  93 | 84   64 | 51      48 x 64  91 | 99   62 | 61      36 x 64  71 | 78   50 | 49
//    48 x 80 110 |  89   74 | 57
inline bool rot_rows_binarizes(const RotGeom& g, bool f32, int64_t rows, int sms) {
    return 2 * rows > sms && g.n1 <= 64 && g.n2 >= 48 && g.n2 <= 80 && (g.n1 > 48 || g.n2 >= (f32 ? 80 : 64));
}
// CTAs a problem gets, of as many as registers, threads and shared memory would let stay (`resident`): one an SM, because each takes all of
// its tensor memory (384 threads, of factors with 32 columns, would fit twice).
inline int rot_rows_ctas(int resident, int sms, int n_problems, int64_t steps) {
    return (int)std::min<int64_t>(steps, std::min(resident, sms) / n_problems);
}
// once per layer: a header with the exponent of P2's scale, then both factors' terms as they lie in shared memory
inline size_t rot_rows_prepared_bytes(const RotRowsGeom& g) { return kRotHeader + (size_t)g.x_off; }

// Up to how many tokens the warp-level MMA kernel (gemm_small.cu) runs the int8 contraction.
constexpr int kSmallTokens = 16;

// ---- the weight-only operating point ----
// Up to how many tokens it runs on three int8 digits per value: gemm_umma.cu, whose MMAs of 128 rows take 51 cycles whatever the 3 M columns
// are up to 64 (mma.sync: 12 a column tile of 8, and 3.4 times as long for two of them), or gemm_small.cu for very few tokens where the codes
// fit one CTA and the rows fill the device.  A call, us, gemm_small.cu | gemm_umma.cu, rank 32:
//                       1 token      4            8            16           32
//    4096 -> 4096      13.8 14.2   13.8 14.2    14.7 14.6    23.0 15.4    23.3 17.1
//    5120 -> 25600     25.8 29.9   27.9 28.3    28.5 23.9    43.2 23.8   143.7 36.7
//    5120 -> 1024      16.5 14.2   16.8 14.4    17.4 14.8    20.3 15.6    24.2 17.1     (split over clusters on gemm_small.cu)
//   25600 -> 5120      45.2 29.5   45.7 32.3    46.0 32.3    69.1 33.5   115.7 46.4     (the same)
constexpr int kDigitTokens = 32, kSmallDigitTokens = 4;
constexpr int kQsumParts = 8;            // partial sums a token's code sum is kept as (one per CTA of its cluster)
// bf16 values, or three digits of few tokens, and the sums of either: never less than fewer tokens need
inline size_t a16_value_bytes(int64_t M, int64_t K) { return std::max((size_t)(M * K * 2), (size_t)(std::min<int64_t>(M, kDigitTokens) * K * 3)); }
inline size_t a16_sum_bytes(int64_t M) { return std::max((size_t)M * 4, (size_t)std::min<int64_t>(M, kDigitTokens) * 3 * kQsumParts * 4); }

}  // namespace bwla
