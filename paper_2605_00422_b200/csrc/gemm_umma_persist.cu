// The binary-weight contraction for many tokens: the arithmetic of gemm_umma.cu (sign words expanded into tensor memory
// as the A operand of tcgen05.mma kind::i8, low-rank term as kind::f16 MMAs, fused epilogue) in pairs of CTAs that stay on their
// SMs and take tiles of 256 output rows x 128 tokens in turn.
//
// A pair (cta_group::2, clusters of two) is one tensor core to the MMAs: each CTA holds 128 of the rows, in its own tensor memory, and
// half of the tokens' codes, in its own shared memory.  One CTA alone needs 16 KB of codes for the 256 cycles of a k-block's MMAs, 64
// bytes a cycle and SM, which is what the L2 delivers; a CTA of a pair needs half of that.  4096 tokens of 25600 -> 5120: 469 us in single
// CTAs, 394 in pairs (2730 TOP/s, about what the power limit leaves: twice the sustained bf16 rate of cuBLAS).
//
// One CTA per tile pays its set-up (barriers, tensor memory, the first loads from HBM) and its epilogue (read-back,
// scaling, 32 KB of output) with the tensor core idle: at 128 tokens that was more than the tile's K loop.  Here the
// producers, the expanders and the MMA issuer run on into the next tile while eight epilogue warps finish the last one:
//   warp 0        packed sign words by TMA (a unit of 1024 weights x 128 rows per stage), all tiles back to back
//   warp 1        per tile: the codes k-block by k-block by TMA, then the three bf16 terms of T (64 tokens of either)
//   warp 2        in the even CTA, MMA issue: the tile's K loop into the int32 accumulator, then the low-rank MMAs, one commit per tile
//   warp 3        per tile: the tokens' scales, code sums and zero points into shared memory
//   warps 4..11   epilogue: stage the tile's rows of U, read the accumulators back (64 tokens each), scale, write bf16 straight from
//                 registers; the accumulator is handed back as soon as it has been read
//   warps 12..27  expansion of sign bits into the tensor-memory operand ring (as in gemm_umma.cu), tile boundaries unseen
// What the issuer waits for arrives on barriers of the even CTA, from both; its commits arrive in both.  Every wait is bounded
// (umma_wait.cuh).
#include <cuda_bf16.h>

#include <algorithm>

#include "bwla_common.cuh"
#include "umma_ptx.cuh"
#include "umma_wait.cuh"
#include "rot_mma.cuh"
#include "tensor_map.cuh"

namespace bwla {

using namespace ptx;

namespace persist {
constexpr int kRows = 128;                // output rows per tile and CTA (256 a pair)
constexpr int kTok = 128;                 // tokens per tile
constexpr int kHalfTok = kTok / 2;        // of which a CTA loads the codes and T
constexpr int kUnitK = 1024;              // weights per row in one sign-word stage
constexpr int kBlockK = 128;              // K per code stage and per operand stage
// A stage is a k-block's codes in shared memory and its expanded signs in tensor memory, under one pair of barriers: the issuing
// thread runs one wait and one commit per k-block.  (With a ring and barriers for each operand the loop took 590 cycles per
// k-block, 500 of them also without any of the copies, stores and MMAs: the issuing thread's waits and commits were the bound.)
constexpr int WS = 3, BS = 8, AS = 4, EW = 4;
static_assert(AS % EW == 0 && BS % AS == 0, "an operand stage must keep one owner among the expander parts");
// Two epilogue warps per lane quarter, 64 tokens each: one warp needs about eight cycles an instruction beside the expanders, and
// with four warps the epilogue of a tile took 8 us, more than the K loop of 5120 it runs under.
constexpr int kEpiFirst = 128, kExpFirst = 384;
constexpr int kThreads = kExpFirst + 128 * EW;       // 896
// registers: 72 a thread at launch (896 x 72 = 64512); 128 x 40 + 256 x 88 + 512 x 72 = 64512 after the split
constexpr int kRegsControl = 40, kRegsEpilogue = 88;
constexpr int w_bytes = kRows * 128, b_bytes = kHalfTok * 128;
constexpr int u_off = WS * w_bytes + BS * b_bytes;
constexpr int t_off = u_off + kRows * 128;
constexpr int bars_off = t_off + 3 * b_bytes;
constexpr int n_bars = 2 * WS + 2 * BS + 12;
constexpr int misc_off = bars_off + n_bars * 8;
constexpr int tok_off = (misc_off + 31) / 16 * 16;   // [2][scales, code sums, zero points, corrections][kTok]
constexpr int used = tok_off + 2 * 16 * kTok;
constexpr int total = used + 1024;
// tensor memory: two int32 accumulators (tiles alternate, so the MMAs of a tile never wait for the epilogue of the one
// before), one fp32 low-rank accumulator (written at the very end of a tile's MMAs, long after the previous epilogue has
// read it), then the operand ring
constexpr int D_COL = 0, LR_COL = 2 * kTok, A_COL = 3 * kTok, TMEM_COLS = 512;
static_assert(A_COL + 32 * AS <= TMEM_COLS, "tensor memory");
static_assert(total <= 232448, "shared memory");
}  // namespace persist

// One linear of a launch (linears of a group have M, K and the presence of a low-rank branch in common).
struct PersistProblem {
    int N, row_tiles, r;
    int fast;                    // no zero points, no row shift, no accumulators wanted, sums below 2^22: the short epilogue
    const float* scales; const int32_t* qsum; const int32_t* zp;
    const float* alpha; const float* mu; const int32_t* rowsum;
    const __nv_bfloat16* U;
    __nv_bfloat16* out; int64_t ldo;
    int32_t* acc_debug;
};
// NP: 1, or up to kRotMaxProblems (a lone linear launched with the parameters of four starts 1 us later)
template <int NP>
struct PersistParams {
    int M, K, tok_tiles;
    int lowrank;
    int tile_begin[NP + 1];     // tiles of problem i: [tile_begin[i], tile_begin[i + 1])
    PersistProblem prob[NP];
    uint32_t* status;
};
template <int NP>
struct PersistMaps { CUtensorMap w[NP], b[NP], t[NP]; };

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint4 lds_words(const uint8_t* p) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(smem_u32(p)) : "memory");
    return v;
}

template <int NP>
__global__ void __launch_bounds__(persist::kThreads, 1)
umma_w1a_persistent_kernel(const __grid_constant__ PersistMaps<NP> maps, const __grid_constant__ PersistParams<NP> p) {
    using namespace persist;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* wbuf = smem;
    uint8_t* bbuf = smem + WS * w_bytes;
    uint8_t* ubuf = smem + u_off;
    uint8_t* tbuf = smem + t_off;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + bars_off);
    uint64_t* w_full = bars;                 // [WS]
    uint64_t* w_empty = w_full + WS;
    uint64_t* s_full = w_empty + WS;         // [BS] codes landed and signs expanded, in both CTAs (the even CTA's are used)
    uint64_t* s_empty = s_full + BS;         // [BS] the MMAs that read both have completed
    uint64_t* d_full = s_empty + BS;         // the tile's MMAs (low-rank ones included) have completed
    uint64_t* acc_free = d_full + 1;         // the epilogue has read the tile's accumulators
    uint64_t* u_full = acc_free + 1;         // the tile's rows of U are staged
    uint64_t* u_empty = u_full + 1;          // the low-rank MMAs have read them
    uint64_t* t_full = u_empty + 1;
    uint64_t* t_empty = t_full + 1;
    uint64_t* tok_full = t_empty + 1;        // [2] per-token scales ... staged (by tile parity)
    uint64_t* epi_done = tok_full + 2;       // [2] the epilogue is through with them
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + misc_off);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + misc_off + 4);
    // per token: scale, sum of the codes, zero point, and the bits of the float 1.5 * 2^23 less the sum of the codes (p.fast) or,
    // as a float, what meets mu (the sum of the codes less K zero points)
    auto tok_scale = [&](int buf) { return reinterpret_cast<float*>(smem + tok_off + buf * 16 * kTok); };
    auto tok_qsum = [&](int buf) { return reinterpret_cast<int32_t*>(smem + tok_off + buf * 16 * kTok + 4 * kTok); };
    auto tok_zp = [&](int buf) { return reinterpret_cast<int32_t*>(smem + tok_off + buf * 16 * kTok + 8 * kTok); };
    auto tok_corr = [&](int buf) { return reinterpret_cast<float*>(smem + tok_off + buf * 16 * kTok + 12 * kTok); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), pairs = (int)(gridDim.x >> 1);
    const int tiles = p.tile_begin[NP];
    const int my_tiles = pair < tiles ? (tiles - pair + pairs - 1) / pairs : 0;
    const int units = (p.K + kUnitK - 1) / kUnitK;
    const int kblocks = p.K / kBlockK;
    // Pairs that work on the same token tile read the same codes: each starts at a unit of its own and goes round (the sums are
    // integers, the order does not matter), so that they do not all ask the same slices of the L2 at the same time.
    const int u0 = (int)(((int64_t)pair * units) / pairs);
    auto unit_at = [&](int j) { const int u = u0 + j; return u < units ? u : u - units; };
    const bool lowrank = p.lowrank != 0;
    // tile i of this pair: one problem after the other, row tiles fastest, so that the CTAs working at the same time share a token
    // tile's codes in the L2
    struct Tile { int pi, n0, t0; };
    auto tile_at = [&](int i) -> Tile {
        int g = pair + i * pairs, pi = 0;
        if (NP > 1)
            while (pi + 1 < NP && g >= p.tile_begin[pi + 1]) ++pi;
        g -= p.tile_begin[pi];
        const int rows = p.prob[pi].row_tiles;
        return Tile{pi, (g % rows) * 2 * kRows + rank * kRows, (g / rows) * kTok};
    };

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int i = 0; i < WS; ++i) { mbar_init(&w_full[i], 1); mbar_init(&w_empty[i], 4 * EW); }
        for (int i = 0; i < BS; ++i) { mbar_init(&s_full[i], 9); mbar_init(&s_empty[i], 1); }      // four expander warps a CTA, and the copies
        mbar_init(d_full, 1); mbar_init(acc_free, 16);
        mbar_init(u_full, 16); mbar_init(u_empty, 1);
        mbar_init(t_full, 1); mbar_init(t_empty, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&tok_full[i], 1); mbar_init(&epi_done[i], 8); }
        fence_barrier_init();
        fence_proxy_async();
    }
    if (warp == 2) {
        tmem_alloc_pair(tmem_slot, TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive_release();                 // the other CTA's barriers stand
    cluster_wait_acquire();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    griddep_launch_dependents();
    // what the MMA thread, in the even CTA, waits for
    auto issuer = [&](uint64_t* bar) { return map_shared_rank(smem_u32(bar), 0u); };

    if (warp < 4) {
    set_regs_dec<kRegsControl>();
    if (warp == 0) {
        // ---------------- packed sign words (independent of the preceding kernel) ----------------
        if (elect_one()) {
#pragma unroll
            for (int i = 0; i < NP; ++i) tma_prefetch_desc(&maps.w[i]);
            // one token tile: every word is read once; more: once per token tile, so they may stay
            const uint64_t stream_once = l2_policy_evict_first();
            const bool once = p.tok_tiles == 1;
            int ws = 0; uint32_t wph = 0;
            for (int i = 0; i < my_tiles && !*abort_flag; ++i) {
                const Tile at = tile_at(i);
                const int n0 = at.n0;
                for (int u = 0; u < units && !*abort_flag; ++u) {
                    if (!mbar_test_wait(&w_empty[ws], wph ^ 1)) {
                        griddep_wait();
                        if (!wait_or_abort(&w_empty[ws], wph ^ 1, abort_flag)) { give_up(p.status, abort_flag, 0x110); break; }
                    }
                    mbar_expect_tx(&w_full[ws], w_bytes);
                    if (once) tma_load_2d_hint(wbuf + ws * w_bytes, &maps.w[at.pi], unit_at(u) * (kUnitK / 32), n0, &w_full[ws], stream_once);
                    else tma_load_2d(wbuf + ws * w_bytes, &maps.w[at.pi], unit_at(u) * (kUnitK / 32), n0, &w_full[ws]);
                    if (++ws == WS) { ws = 0; wph ^= 1; }
                }
            }
            if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);
        }
    } else if (warp == 1) {
        // ---------------- codes and T ----------------
        griddep_wait();
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < NP; ++i) {
                tma_prefetch_desc(&maps.b[i]);
                if (lowrank) tma_prefetch_desc(&maps.t[i]);
            }
            if (p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0) *abort_flag = 1;   // the call already failed
        }
        __syncwarp();
        if (lane == 0) {
            int bs = 0; uint32_t bph = 0;
            bool ok = true;
            for (int i = 0; i < my_tiles && ok && !*abort_flag; ++i) {
                const Tile at = tile_at(i);
                const int t0 = at.t0 + rank * kHalfTok;
                int kb = u0 * (kUnitK / kBlockK);
                for (int c = 0; c < kblocks; ++c) {
                    if (!wait_or_abort(&s_empty[bs], bph ^ 1, abort_flag)) { give_up(p.status, abort_flag, 0x121); ok = false; break; }
                    if (rank == 0) mbar_expect_tx(&s_full[bs], 2 * b_bytes);
                    tma_load_2d_pair(bbuf + bs * b_bytes, &maps.b[at.pi], kb * kBlockK, t0, issuer(&s_full[bs]));
                    if (++bs == BS) { bs = 0; bph ^= 1; }
                    if (++kb == kblocks) kb = 0;
                }
                // T is first needed when the K loop is over; the previous tile's low-rank MMAs have long read theirs
                if (ok && lowrank) {
                    if (i >= 1 && !wait_or_abort(t_empty, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x122); ok = false; }
                    if (ok) {
                        if (rank == 0) mbar_expect_tx(t_full, 6 * b_bytes);
                        for (int h = 0; h < 3; ++h) tma_load_3d_pair(tbuf + h * b_bytes, &maps.t[at.pi], 0, t0, h, issuer(t_full));
                    }
                }
            }
            if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);
        }
    } else if (warp == 3) {
        // ---------------- per-token scalars (a warp of its own: in the codes' warp their load latency, 2 us a tile, held up the
        // codes of the tile) ----------------
        griddep_wait();
        for (int i = 0; i < my_tiles && !*abort_flag; ++i) {
            const Tile at = tile_at(i);
            const PersistProblem& pr = p.prob[at.pi];
            const int t0 = at.t0, buf = i & 1;
            if (i >= 2 && !warp_wait(&epi_done[buf], (uint32_t)(((i >> 1) - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x120); break; }
            for (int j = lane; j < kTok; j += 32) {
                const int t = t0 + j;
                tok_scale(buf)[j] = t < p.M ? pr.scales[t] : 0.f;
                int32_t qs = 0;
                if (t < p.M) {
                    const int4* parts = reinterpret_cast<const int4*>(pr.qsum + (size_t)t * kQsumParts);
                    const int4 a = parts[0], b = parts[1];
                    qs = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
                }
                tok_qsum(buf)[j] = qs;
                const int32_t zp = (pr.zp && t < p.M) ? pr.zp[t] : 0;
                tok_zp(buf)[j] = zp;
                tok_corr(buf)[j] = pr.fast ? __int_as_float(0x4B400000 - qs) : (float)(qs - p.K * zp);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&tok_full[buf]);
        }
    } else if (warp == 2) {
        // ---------------- MMA issue, for both CTAs ----------------
        if (rank == 0 && elect_one()) {
            const uint32_t idesc = (2u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTok >> 3) << 17) | ((256u >> 4) << 24);
            const uint32_t idesc_lr = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTok >> 3) << 17) | ((256u >> 4) << 24);
            const uint32_t a_base = tmem_base + A_COL;
            const uint64_t desc_hi = smem_desc_sw128(0u, 0u);
            const uint32_t b_lo0 = (smem_u32(bbuf) & 0x3FFFFu) >> 4;
            int bs = 0; uint32_t bph = 0;
            bool ok = true;
            griddep_wait();                           // everything this thread waits for follows the preceding kernel
            for (int i = 0; i < my_tiles && ok; ++i) {
                // accumulator i & 1 was last used by tile i - 2, whose epilogue this thread has seen finish at the end of tile
                // i - 1 (below)
                tc_fence_after();
                const uint32_t d_addr = tmem_base + D_COL + (uint32_t)(i & 1) * kTok;
                uint32_t acc = 0;
                for (int kb = 0; kb < kblocks && ok; ++kb) {
                    if (!wait_or_abort(&s_full[bs], bph, abort_flag)) { give_up(p.status, abort_flag, 0x132); ok = false; break; }
                    tc_fence_after();
                    const uint64_t desc = desc_hi | (uint64_t)(b_lo0 + (uint32_t)bs * (b_bytes >> 4));
                    const uint32_t a_addr = a_base + 32 * (bs % AS);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        mma_i8_ts_pair(d_addr, a_addr + 8 * j, desc + 2 * j, idesc, acc);
                        acc = 1u;
                    }
                    tc_commit_pair(&s_empty[bs]);
                    if (++bs == BS) { bs = 0; bph ^= 1u; }
                }
                // The epilogue of the tile before has had this tile's whole K loop to read its accumulators; it is waited for
                // here, before this tile's MMAs are committed, so that completions of acc_free are seen strictly in order
                // (a parity wait only tells the current phase from the one before it).  It frees the low-rank accumulator
                // for this tile and the int32 accumulator for the next.
                if (ok && i >= 1 && !wait_or_abort(acc_free, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x130); ok = false; }
                if (ok && lowrank) {
                    if (!wait_or_abort(u_full, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x133); ok = false; }
                    if (ok && !wait_or_abort(t_full, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x134); ok = false; }
                    if (ok) {
                        tc_fence_after();
                        const uint32_t u_addr = smem_u32(ubuf);
                        const int r = p.prob[tile_at(i).pi].r;      // (zeros beyond)
#pragma unroll
                        for (int h = 0; h < 3; ++h) {
                            const uint32_t t_addr = smem_u32(tbuf + h * b_bytes);
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if (16 * j < r) mma_f16_ss_pair(tmem_base + LR_COL, smem_desc_sw128(u_addr, 32 * j), smem_desc_sw128(t_addr, 32 * j),
                                           idesc_lr, (h | j) ? 1u : 0u);
                        }
                        tc_commit_pair(u_empty);
                        tc_commit_pair(t_empty);
                    }
                }
                tc_commit_pair(d_full);
            }
        }
    }
    } else if (warp < 12) {
        set_regs_inc<kRegsEpilogue>();
        // ---------------- epilogue ----------------
        const int q = warp & 3;
        const int e = (threadIdx.x - kEpiFirst) & 127;        // output row of the tile
        const int half = (warp - 4) >> 2;             // of the tile's tokens
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        bool ok = true;
        for (int i = 0; i < my_tiles; ++i) {
            const Tile at = tile_at(i);
            const PersistProblem& pr = p.prob[at.pi];
            const int n0 = at.n0, t0 = at.t0, buf = i & 1;
            const int n = n0 + e;
            const bool valid_row = n < pr.N;
            const float alpha_n = valid_row ? __ldg(pr.alpha + n) : 0.f;
            const float mu_n = (pr.mu && valid_row) ? __ldg(pr.mu + n) : 0.f;
            const int32_t rs_n = (pr.zp && valid_row) ? __ldg(pr.rowsum + n) : 0;
            if (lowrank) {
                // this tile's rows of U: 128 rows x 8 chunks of 16 bytes, 128B-swizzled K-major, zero beyond N and r
                if (ok && i >= 1 && !warp_wait(u_empty, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x140); ok = false; }
                if (ok) {
                    const bool vec = (pr.r % 8 == 0) && ((reinterpret_cast<uintptr_t>(pr.U) & 15) == 0);
#pragma unroll
                    for (int it = 0; it < 4; ++it) {
                        const int idx = it * 256 + half * 128 + e;
                        const int ur = idx >> 3, ch = idx & 7;
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        const int un = n0 + ur;
                        if (un < pr.N && ch * 8 < pr.r) {
                            const __nv_bfloat16* src = pr.U + (int64_t)un * pr.r + ch * 8;
                            if (vec) {
                                v = __ldg(reinterpret_cast<const uint4*>(src));
                            } else {
                                uint32_t w[4] = {0u, 0u, 0u, 0u};
                                for (int c = 0; c < 8 && ch * 8 + c < pr.r; ++c)
                                    w[c >> 1] |= (uint32_t)__bfloat16_as_ushort(src[c]) << (16 * (c & 1));
                                v = make_uint4(w[0], w[1], w[2], w[3]);
                            }
                        }
                        *reinterpret_cast<uint4*>(ubuf + ur * 128 + ((ch ^ (ur & 7)) << 4)) = v;
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_pair(issuer(u_full));
                }
            }
            if (i == 0) griddep_wait();                       // nothing is stored before the preceding kernel has completed
            if (ok && !warp_wait(&tok_full[buf], (uint32_t)((i >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x141); ok = false; }
            if (ok && !warp_wait(d_full, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x142); ok = false; }
            if (ok) {
                tc_fence_after();
                const float4* sc_s = reinterpret_cast<const float4*>(tok_scale(buf));
                const float4* co_s = reinterpret_cast<const float4*>(tok_corr(buf));
                const int4* qs_s = reinterpret_cast<const int4*>(tok_qsum(buf));
                const int4* zp_s = reinterpret_cast<const int4*>(tok_zp(buf));
                // Finished values go straight to global memory: a lane has one row and two tokens in a word, its neighbour the
                // other row of the pair; they swap halves, and a store instruction writes 64 bytes of each token's outputs.
                // (Through a shared-memory tile, one 16-bit store a value with three scalar loads and two conversions beside
                // it, four warps took 10.8 us a tile.)
                const int odd = lane & 1;
                const uint32_t sel = odd ? 0x3276u : 0x5410u;
                const int n_pair = n & ~1;
                const bool pair_ok = ((reinterpret_cast<uintptr_t>(pr.out) & 3) == 0) && (pr.ldo & 1) == 0 && n_pair + 1 < pr.N;
                const bool pairs_ok = __all_sync(0xFFFFFFFFu, pair_ok);
                const uint32_t acc_addr = tmem_base + lane_addr + D_COL + (uint32_t)(i & 1) * kTok;
                auto put = [&](uint32_t word, int tok) {          // word: tokens tok (low half) and tok + 1 of this lane's row
                    const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, word, 1);
                    if (pair_ok) {
                        const int t = t0 + tok + odd;
                        if (t < p.M) *reinterpret_cast<uint32_t*>(pr.out + (int64_t)t * pr.ldo + n_pair) = __byte_perm(word, other, sel);
                    } else if (valid_row) {
#pragma unroll
                        for (int h = 0; h < 2; ++h)
                            if (t0 + tok + h < p.M) pr.out[(int64_t)(t0 + tok + h) * pr.ldo + n] = __ushort_as_bfloat16((unsigned short)(word >> (16 * h)));
                    }
                };
#pragma unroll 1
                for (int c = half * (kTok / 32); c < (half + 1) * (kTok / 32); ++c) {
                    uint32_t v[16], l[16];
                    tmem_ld_32x16(acc_addr + 16 * c, v);
                    if (lowrank) tmem_ld_32x16(tmem_base + lane_addr + LR_COL + 16 * c, l);
                    tc_wait_ld();
                    if (c == (half + 1) * (kTok / 32) - 1) {
                        // both accumulators are in registers: the next tile's MMAs may start
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_pair(issuer(acc_free));
                    }
                    if (t0 + 16 * c >= p.M) continue;            // warp-uniform; nothing of this chunk is stored
                    if (pr.fast && pairs_ok && t0 + 16 * c + 16 <= p.M) {
                        // The usual case, a whole chunk: no conditions on single stores, a pointer that steps, packed additions.  A short K loop waits for
                        // its epilogue, 2400 cycles a chunk without this (270 instructions beside the expanders): 4096 tokens of 2048 -> 25600 279 us,
                        // 207 with it; of 5120 -> 25600, where most of it is hidden, 449 and 422.
                        __nv_bfloat16* at = pr.out + (int64_t)(t0 + 16 * c + odd) * pr.ldo + n_pair;
                        const int64_t step = 2 * pr.ldo;
#pragma unroll
                        for (int j = 0; j < 16; j += 4) {
                            const float4 sc = sc_s[4 * c + (j >> 2)], co = co_s[4 * c + (j >> 2)];
                            const float scs[4] = {sc.x, sc.y, sc.z, sc.w}, cos[4] = {co.x, co.y, co.z, co.w};
                            float y[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h) y[h] = __int_as_float(__float_as_int(cos[h]) - ((int32_t)v[j + h] >> 6));
                            add2(y[0], y[1], -12582912.f, -12582912.f);
                            add2(y[2], y[3], -12582912.f, -12582912.f);
                            // (the product is rounded before the addition: the scalar multiplication is not contracted)
#pragma unroll
                            for (int h = 0; h < 4; ++h) y[h] = __fmul_rn(__fmul_rn(alpha_n, scs[h]), y[h]);
                            add2(y[0], y[1], lowrank ? __uint_as_float(l[j]) : 0.f, lowrank ? __uint_as_float(l[j + 1]) : 0.f);
                            add2(y[2], y[3], lowrank ? __uint_as_float(l[j + 2]) : 0.f, lowrank ? __uint_as_float(l[j + 3]) : 0.f);
#pragma unroll
                            for (int h = 0; h < 4; h += 2) {
                                const uint32_t word = pack_bf16x2(y[h], y[h + 1]);
                                const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, word, 1);
                                *reinterpret_cast<uint32_t*>(at) = __byte_perm(word, other, sel);
                                at += step;
                            }
                        }
                    } else if (pr.fast) {
                        // the raw sum is -2^7 times the sum over the set bits; 1.5 * 2^23 + integer (below 2^22) is a float by its
                        // bits, and taking 1.5 * 2^23 off again is exact
#pragma unroll
                        for (int j = 0; j < 16; j += 4) {
                            const float4 sc = sc_s[4 * c + (j >> 2)], co = co_s[4 * c + (j >> 2)];
                            const float scs[4] = {sc.x, sc.y, sc.z, sc.w}, cos[4] = {co.x, co.y, co.z, co.w};
                            float y[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                const float acc = __int_as_float(__float_as_int(cos[h]) - ((int32_t)v[j + h] >> 6)) - 12582912.f;
                                y[h] = __fmul_rn(__fmul_rn(alpha_n, scs[h]), acc) + (lowrank ? __uint_as_float(l[j + h]) : 0.f);
                            }
                            put(pack_bf16x2(y[0], y[1]), 16 * c + j);
                            put(pack_bf16x2(y[2], y[3]), 16 * c + j + 2);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; j += 4) {
                            const float4 sc = sc_s[4 * c + (j >> 2)], co = co_s[4 * c + (j >> 2)];
                            const int4 qs = qs_s[4 * c + (j >> 2)], zp = zp_s[4 * c + (j >> 2)];
                            const float scs[4] = {sc.x, sc.y, sc.z, sc.w}, cos[4] = {co.x, co.y, co.z, co.w};
                            const int32_t qss[4] = {qs.x, qs.y, qs.z, qs.w}, zps[4] = {zp.x, zp.y, zp.z, zp.w};
                            float y[4];
#pragma unroll
                            for (int h = 0; h < 4; ++h) {
                                const int32_t acc = -((int32_t)v[j + h] >> 6) - qss[h] - zps[h] * rs_n;
                                if (pr.acc_debug && valid_row && t0 + 16 * c + j + h < p.M) pr.acc_debug[(int64_t)(t0 + 16 * c + j + h) * pr.N + n] = acc;
                                y[h] = fmaf(__fmul_rn(mu_n, scs[h]), cos[h], __fmul_rn(__fmul_rn(alpha_n, scs[h]), (float)acc) + (lowrank ? __uint_as_float(l[j + h]) : 0.f));
                            }
                            if (pr.out) {
                                put(pack_bf16x2(y[0], y[1]), 16 * c + j);
                                put(pack_bf16x2(y[2], y[3]), 16 * c + j + 2);
                            }
                        }
                    }
                }
            } else if (!*abort_flag) {
                *abort_flag = 1;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&epi_done[buf]);
        }
    } else {
        // ---------------- expansion of sign bits into the operand ring (tile boundaries do not matter here) ----------------
        const int q = warp & 3;
        const int part = (warp - 12) >> 2;             // which of the EW warps of the lane quarter
        const int row = q * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        // A warp's words of a unit (two blocks of eight) go to registers, a unit ahead, and the stage is let go at once: the copies
        // then have three units of MMA time to arrive instead of one.  (Held until the unit was expanded, the two stages made the
        // loop wait for the L2: 537 us for 4096 x 5120 x 25600 with and without MMAs, stores and code copies.)
        // Block g of this CTA (a running count over its tiles) belongs to part g % EW and to stage g % AS.  AS is a multiple of
        // EW, so a stage always has the same owner and the owner is never more than one phase ahead of the stage's consumer: a
        // parity wait cannot tell a phase from the one two before it.  (The last unit of a row may hold fewer than eight
        // blocks, which is why neither follows from the position inside the unit.)
        constexpr int PER = kUnitK / kBlockK / EW;
        const uint32_t filled = issuer(s_full);
        int ws = 0; uint32_t wph = 0;
        const int total = my_tiles * units;
        int c = 0, u_nxt = 0;                         // next unit to take: running number, position in its row
        int base_nxt = 0;                             // blocks of this CTA before it
        uint4 nxt[PER];
        int ns_nxt = 0, first_nxt = 0, g_nxt = 0;
        bool ok = true;
        auto take = [&]() {                           // (the unit's stage is full)
            ns_nxt = min(kUnitK / kBlockK, (p.K - unit_at(u_nxt) * kUnitK) / kBlockK);
            first_nxt = (part + EW - base_nxt % EW) % EW;
            g_nxt = base_nxt + first_nxt;
            const uint8_t* wrow = wbuf + ws * w_bytes + row * 128;
#pragma unroll
            for (int q = 0; q < PER; ++q) nxt[q] = lds_words(wrow + (((first_nxt + EW * q) ^ (row & 7)) << 4));
            // (behind the loads' data: see release_stage)
            uint32_t seen = 0u;
#pragma unroll
            for (int q = 0; q < PER; ++q) seen ^= nxt[q].x ^ nxt[q].y ^ nxt[q].z ^ nxt[q].w;
            release_stage(&w_empty[ws], seen);
            if (++ws == WS) { ws = 0; wph ^= 1u; }
            base_nxt += ns_nxt;
            if (++u_nxt == units) u_nxt = 0;
            ++c;
        };
        if (total > 0) {
            if (!warp_wait(&w_full[ws], wph, abort_flag)) { give_up(p.status, abort_flag, 0x150); ok = false; }
            else take();
        }
        for (int i = 0; i < total && ok; ++i) {
            uint4 cur[PER];
#pragma unroll
            for (int q = 0; q < PER; ++q) cur[q] = nxt[q];
            const int ns = ns_nxt, first = first_nxt, g = g_nxt;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                if (c == i + 1 && c < total && __all_sync(0xFFFFFFFFu, mbar_test_wait(&w_full[ws], wph))) take();
                if (first + EW * q < ns && ok) {
                    uint32_t v[32];
                    const uint32_t w[4] = {cur[q].x, cur[q].y, cur[q].z, cur[q].w};
#pragma unroll
                    for (int k = 0; k < 4; ++k)
#pragma unroll
                        for (int j = 0; j < 8; ++j) v[8 * k + j] = (w[k] << (7 - j)) & 0x80808080u;
                    const int as = (g + EW * q) % AS, bs = (g + EW * q) % BS;
                    // the block that used the operand stage before: AS blocks ago, under the barrier of its own code stage
                    const int before = g + EW * q - AS;
                    const int gone = before & (BS - 1);
                    const uint32_t gone_ph = (uint32_t)((before / BS) & 1);
                    if (before >= 0 && !__all_sync(0xFFFFFFFFu, mbar_test_wait(&s_empty[gone], gone_ph))) {
                        griddep_wait();
                        if (!warp_wait(&s_empty[gone], gone_ph, abort_flag)) { give_up(p.status, abort_flag, 0x151); ok = false; }
                    }
                    if (ok) {
                        tc_fence_after();
                        tmem_st_32x32(tmem_base + lane_addr + A_COL + 32 * as, v);
                        tc_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_pair(filled + 8u * (uint32_t)bs);
                    }
                }
            }
            if (c == i + 1 && c < total && ok) {
                if (!warp_wait(&w_full[ws], wph, abort_flag)) { give_up(p.status, abort_flag, 0x152); ok = false; }
                else take();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_arrive_release();                 // nobody leaves while the other CTA may still reach its memories
    cluster_wait_acquire();
    if (warp == 2) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, TMEM_COLS);
    }
}

bool umma_persistent_supports(int64_t M, int64_t K, int64_t N, int r) {
    // every k-block of a tile must exist in full (a whole number of 128-weight blocks), and the tile loop pays off with
    // more tiles than SMs
    return M > 64 && K % 128 == 0 && r <= kLowrankPad && N > 0;
}

template <int NP>
static int launch_persistent(const GemmArgs* a, int n, cudaStream_t stream) {
    using namespace persist;
    const int M = (int)a[0].M, K = (int)a[0].K;
    PersistMaps<NP> maps;
    PersistParams<NP> p{};
    p.M = M; p.K = K; p.tok_tiles = (M + kTok - 1) / kTok; p.lowrank = a[0].r > 0; p.status = a[0].status;
    for (int i = 0; i < n; ++i) {
        const GemmArgs& g = a[i];
        const int N = (int)g.N;
        {
            const uint64_t dims[2] = {(uint64_t)K / 32, (uint64_t)N};
            const uint64_t strides[1] = {(uint64_t)K / 8};
            const uint32_t box[2] = {32, kRows};
            int st = make_map(&maps.w[i], CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, g.packed, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
            if (st != BWLA_OK) return st;
        }
        {
            const uint64_t dims[2] = {(uint64_t)K, (uint64_t)M};
            const uint64_t strides[1] = {(uint64_t)K};
            const uint32_t box[2] = {kBlockK, kHalfTok};
            int st = make_map(&maps.b[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, g.codes, dims, strides, box,
                              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
            if (st != BWLA_OK) return st;
        }
        if (g.r > 0) {
            const uint64_t dims[3] = {(uint64_t)kLowrankPad, (uint64_t)M, 3};
            const uint64_t strides[2] = {(uint64_t)kLowrankPad * 2, (uint64_t)M * kLowrankPad * 2};
            const uint32_t box[3] = {(uint32_t)kLowrankPad, kHalfTok, 1};
            int st = make_map(&maps.t[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, g.Thl, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
            if (st != BWLA_OK) return st;
        } else {
            maps.t[i] = maps.b[i];   // never dereferenced
        }
        PersistProblem& pr = p.prob[i];
        pr.N = N; pr.row_tiles = (N + 2 * kRows - 1) / (2 * kRows); pr.r = g.r;
        pr.scales = g.scales; pr.qsum = g.qsum; pr.zp = g.zp; pr.alpha = g.alpha; pr.mu = g.mu; pr.rowsum = g.rowsum;
        pr.U = (const __nv_bfloat16*)g.U; pr.out = (__nv_bfloat16*)g.out; pr.ldo = g.ldo; pr.acc_debug = g.acc_debug;
        pr.fast = !g.zp && !g.mu && !g.acc_debug && g.out && (int64_t)K << 7 < (int64_t)1 << 22;      // (whatever the codes a caller hands over)
        p.tile_begin[i + 1] = p.tile_begin[i] + pr.row_tiles * p.tok_tiles;
    }
    for (int i = n; i < NP; ++i) { maps.w[i] = maps.w[0]; maps.b[i] = maps.b[0]; maps.t[i] = maps.t[0]; p.tile_begin[i + 1] = p.tile_begin[n]; }

    static thread_local int configured = -1;
    int dev = 0;
    BWLA_CUDA_TRY(cudaGetDevice(&dev));
    if (configured != dev) {
        BWLA_CUDA_TRY(cudaFuncSetAttribute(umma_w1a_persistent_kernel<NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, total));
        configured = dev;
    }
    const int pairs = resident_clusters((const void*)umma_w1a_persistent_kernel<NP>, 2, kThreads, total);
    if (pairs < 1) return cuda_fail(cudaErrorInvalidConfiguration);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2u * (unsigned)std::min(p.tile_begin[n], pairs), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = total;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = launch_overlap_allowed();
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = 2; attrs[1].val.clusterDim.y = 1; attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = 2;
    ProfScope prof(kProfContraction, stream);
    cudaError_t e = cudaLaunchKernelEx(&cfg, umma_w1a_persistent_kernel<NP>, maps, p);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}

int launch_gemm_umma_persistent(const GemmArgs* a, int n, cudaStream_t stream) {
    if (n < 1 || n > kRotMaxProblems) return BWLA_ERR_INVALID_ARG;
    return n == 1 ? launch_persistent<1>(a, n, stream) : launch_persistent<kRotMaxProblems>(a, n, stream);
}

}  // namespace bwla
