// The weight-only operating point (gemm_a16.cu has the definition) for K a multiple of 128: the contraction of bf16 activations with
// signs expanded to +-1 in tensor memory, in persistent CTAs, built like gemm_umma_persist.cu.
//
//   out[t][n] = bf16( alpha[n] * sum_k s[n][k] * yhat[t][k] + U[n,:] . T[t,:] + mu[n] * sum_k yhat[t][k] )
//
// Tile: 128 weight rows (lanes) x 128 tokens (columns).  A stage is 64 values of k: 128 tokens of yhat in shared memory (one 128-byte
// swizzle atom) and the signs of 128 rows, two to a word, in 32 columns of tensor memory.  With both operands in shared memory
// (gemm_a16.cu) the MMAs alone read it at its full rate, beside the stores of the expanded signs, and four warps expanded them: 900
// cycles per 64 values of k instead of the MMAs' 256 (1024 x 4096 x 4096: 63 us, here 50; a stage takes 0.24 us, 0.18 at the
// measured cuBLAS rate).
//
// yhat lies in the interleaved order (inside each group of 32: position 2 (k % 16) + (k % 32) / 16), so that a word of two bf16 takes
// bits j and j + 16 of a sign word: a shift and one three-input logic operation.
//
// The tensor core truncates when it adds to its accumulator, so it only ever holds 512 values of k (as in gemm_a16.cu): the epilogue
// warps add it into running sums in registers, with rounded additions, while the next 512 go to the second accumulator.
//
// Warps 0..3: sign words, yhat and T, MMA issue, per-token sums.  4..11: epilogue, two per lane quarter, 64 tokens each; their running
// sums take registers that the other warps give away.  12..27: expansion, four per lane quarter, every fourth stage each.
#include <cuda_bf16.h>

#include <algorithm>

#include "bwla_common.cuh"
#include "tensor_map.cuh"
#include "umma_ptx.cuh"
#include "umma_wait.cuh"

namespace bwla {

namespace a16p {
constexpr int kRows = 128;                // output rows per tile
constexpr int kTok = 128;                 // tokens per tile
constexpr int kUnitK = 1024;              // weights per row in one sign-word stage
constexpr int kBlockK = 64;               // K per stage
constexpr int kFlush = 8;                 // stages per accumulator
constexpr int WS = 3, AS = 4, EW = 4;
static_assert(AS % EW == 0, "an operand stage must keep one owner among the expander parts");
constexpr int kEpiFirst = 128, kExpFirst = 384;
constexpr int kThreads = kExpFirst + 128 * EW;       // 896
// registers: 72 a thread at launch (896 x 72 = 64512); 128 x 56 + 256 x 112 + 512 x 56 = 64512 after the split
constexpr int kRegsControl = 56, kRegsEpilogue = 112, kRegsExpand = 56;
constexpr int w_bytes = kRows * 128, b_bytes = kTok * 128;
constexpr int u_off = WS * w_bytes + AS * b_bytes;
constexpr int t_off = u_off + kRows * 128;
constexpr int bars_off = t_off + 3 * b_bytes;
constexpr int n_bars = 2 * WS + 2 * AS + 14;
constexpr int misc_off = bars_off + n_bars * 8;
constexpr int tok_off = (misc_off + 31) / 16 * 16;   // [2][sums of the token's values][kTok]
constexpr int used = tok_off + 2 * 4 * kTok;
constexpr int total = used + 1024;
// tensor memory: two accumulators (512 values of k each, in turn), the low-rank accumulator, the operand ring
constexpr int D_COL = 0, LR_COL = 2 * kTok, A_COL = 3 * kTok, TMEM_COLS = 512;
static_assert(A_COL + 32 * AS <= TMEM_COLS, "tensor memory");
static_assert(total <= 232448, "shared memory");
}  // namespace a16p

struct A16PersistParams {
    int M, N, K;
    int row_tiles, tok_tiles;
    int r;
    const float* alpha; const float* mu; const float* ysum;
    const __nv_bfloat16* U;
    __nv_bfloat16* out; int64_t ldo;
    uint32_t* status;
};

namespace {
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ void tmem_st_32x16(uint32_t taddr, const uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
__device__ __forceinline__ uint2 lds_words(const uint8_t* p) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(smem_u32(p)) : "memory");
    return v;
}
}  // namespace

__global__ void __launch_bounds__(a16p::kThreads, 1)
a16_persistent_kernel(const __grid_constant__ CUtensorMap w_map, const __grid_constant__ CUtensorMap b_map,
                           const __grid_constant__ CUtensorMap t_map, A16PersistParams p) {
    using namespace a16p;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* wbuf = smem;
    uint8_t* bbuf = smem + WS * w_bytes;
    uint8_t* ubuf = smem + u_off;
    uint8_t* tbuf = smem + t_off;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + bars_off);
    uint64_t* w_full = bars;                 // [WS]
    uint64_t* w_empty = w_full + WS;
    uint64_t* s_full = w_empty + WS;         // [AS] yhat landed and signs expanded
    uint64_t* s_empty = s_full + AS;         // [AS] the MMAs that read both have completed
    uint64_t* d_full = s_empty + AS;         // [2] 512 values of k are summed
    uint64_t* acc_free = d_full + 2;         // [2] the epilogue has read them
    uint64_t* lr_full = acc_free + 2;        // the tile's low-rank MMAs have completed
    uint64_t* lr_free = lr_full + 1;
    uint64_t* u_full = lr_free + 1;         // the tile's rows of U are staged
    uint64_t* u_empty = u_full + 1;          // the low-rank MMAs have read them
    uint64_t* t_full = u_empty + 1;
    uint64_t* t_empty = t_full + 1;
    uint64_t* tok_full = t_empty + 1;        // [2] per-token sums staged (by tile parity)
    uint64_t* epi_done = tok_full + 2;       // [2] the epilogue is through with them
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + misc_off);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + misc_off + 4);
    auto tok_sum = [&](int buf) { return reinterpret_cast<float*>(smem + tok_off + buf * 4 * kTok); };

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tiles = p.row_tiles * p.tok_tiles;
    const int my_tiles = (int)blockIdx.x < tiles ? (tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x : 0;
    const int units = (p.K + kUnitK - 1) / kUnitK;
    const int kblocks = p.K / kBlockK, groups = (kblocks + kFlush - 1) / kFlush;
    // CTAs that work on the same token tile read the same values: each starts at a unit of its own and goes round, so that they do not
    // all ask the same slices of the L2 at the same time.
    const int u0 = (int)(((int64_t)blockIdx.x * units) / gridDim.x);
    auto unit_at = [&](int j) { const int u = u0 + j; return u < units ? u : u - units; };
    const bool lowrank = p.r > 0;
    // tile i of this CTA: row tiles fastest, so that the CTAs working at the same time share a token tile of yhat in the L2
    auto tile_n0 = [&](int i) { return (((int)blockIdx.x + i * (int)gridDim.x) % p.row_tiles) * kRows; };
    auto tile_t0 = [&](int i) { return (((int)blockIdx.x + i * (int)gridDim.x) / p.row_tiles) * kTok; };

    if (threadIdx.x == 0) {
        *abort_flag = 0;
        for (int i = 0; i < WS; ++i) { mbar_init(&w_full[i], 1); mbar_init(&w_empty[i], 4 * EW); }
        for (int i = 0; i < AS; ++i) { mbar_init(&s_full[i], 5); mbar_init(&s_empty[i], 1); }      // four expander warps and the copy
        for (int i = 0; i < 2; ++i) { mbar_init(&d_full[i], 1); mbar_init(&acc_free[i], 8); }
        mbar_init(lr_full, 1); mbar_init(lr_free, 8);
        mbar_init(u_full, 8); mbar_init(u_empty, 1);
        mbar_init(t_full, 1); mbar_init(t_empty, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(&tok_full[i], 1); mbar_init(&epi_done[i], 8); }
        fence_barrier_init();
        fence_proxy_async();
    }
    if (warp == 2) {
        tmem_alloc(tmem_slot, TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    griddep_launch_dependents();

    if (warp < 4) {
    set_regs_dec<kRegsControl>();
    if (warp == 0) {
        // ---------------- packed sign words (independent of the preceding kernel) ----------------
        if (elect_one()) {
            tma_prefetch_desc(&w_map);
            // one token tile: every word is read once; more: once per token tile, so they may stay
            const uint64_t stream_once = l2_policy_evict_first();
            const bool once = p.tok_tiles == 1;
            int ws = 0; uint32_t wph = 0;
            for (int i = 0; i < my_tiles && !*abort_flag; ++i) {
                const int n0 = tile_n0(i);
                for (int u = 0; u < units && !*abort_flag; ++u) {
                    if (!mbar_test_wait(&w_empty[ws], wph ^ 1)) {
                        griddep_wait();
                        if (!wait_or_abort(&w_empty[ws], wph ^ 1, abort_flag)) { give_up(p.status, abort_flag, 0x410); break; }
                    }
                    mbar_expect_tx(&w_full[ws], w_bytes);
                    if (once) tma_load_2d_hint(wbuf + ws * w_bytes, &w_map, unit_at(u) * (kUnitK / 32), n0, &w_full[ws], stream_once);
                    else tma_load_2d(wbuf + ws * w_bytes, &w_map, unit_at(u) * (kUnitK / 32), n0, &w_full[ws]);
                    if (++ws == WS) { ws = 0; wph ^= 1; }
                }
            }
            if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);
        }
    } else if (warp == 1) {
        // ---------------- yhat and T ----------------
        griddep_wait();
        if (lane == 0) {
            tma_prefetch_desc(&b_map);
            if (lowrank) tma_prefetch_desc(&t_map);
            if (p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0) *abort_flag = 1;   // the call already failed
        }
        __syncwarp();
        if (lane == 0) {
            int bs = 0; uint32_t bph = 0;
            bool ok = true;
            for (int i = 0; i < my_tiles && ok && !*abort_flag; ++i) {
                const int t0 = tile_t0(i);
                int kb = u0 * (kUnitK / kBlockK);
                for (int c = 0; c < kblocks; ++c) {
                    if (!wait_or_abort(&s_empty[bs], bph ^ 1, abort_flag)) { give_up(p.status, abort_flag, 0x421); ok = false; break; }
                    mbar_expect_tx(&s_full[bs], b_bytes);
                    tma_load_2d(bbuf + bs * b_bytes, &b_map, kb * kBlockK, t0, &s_full[bs]);
                    if (++bs == AS) { bs = 0; bph ^= 1; }
                    if (++kb == kblocks) kb = 0;
                }
                // T is first needed when the K loop is over; the previous tile's low-rank MMAs have long read theirs
                if (ok && lowrank) {
                    if (i >= 1 && !wait_or_abort(t_empty, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x422); ok = false; }
                    if (ok) {
                        mbar_expect_tx(t_full, 3 * b_bytes);
                        for (int h = 0; h < 3; ++h) tma_load_3d(tbuf + h * b_bytes, &t_map, 0, t0, h, t_full);
                    }
                }
            }
            if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);
        }
    } else if (warp == 3) {
        // ---------------- per-token sums ----------------
        griddep_wait();
        for (int i = 0; i < my_tiles && !*abort_flag; ++i) {
            const int t0 = tile_t0(i), buf = i & 1;
            if (i >= 2 && !warp_wait(&epi_done[buf], (uint32_t)(((i >> 1) - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x420); break; }
            for (int j = lane; j < kTok; j += 32) tok_sum(buf)[j] = (p.ysum && t0 + j < p.M) ? p.ysum[t0 + j] : 0.f;
            __syncwarp();
            if (lane == 0) mbar_arrive(&tok_full[buf]);
        }
    } else if (warp == 2) {
        // ---------------- MMA issue ----------------
        if (elect_one()) {
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTok >> 3) << 17) | ((128u >> 4) << 24);
            const uint32_t a_base = tmem_base + A_COL;
            const uint64_t desc_hi = smem_desc_sw128(0u, 0u);
            const uint32_t b_lo0 = (smem_u32(bbuf) & 0x3FFFFu) >> 4;
            int as = 0; uint32_t aph = 0;
            bool ok = true;
            int f = 0;                                // running number of the accumulator fills
            griddep_wait();                           // everything this thread waits for follows the preceding kernel
            for (int i = 0; i < my_tiles && ok; ++i) {
                for (int kb = 0; kb < kblocks && ok; ++f) {
                    if (f >= 2 && !wait_or_abort(&acc_free[f & 1], (uint32_t)(((f >> 1) - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x430); ok = false; break; }
                    tc_fence_after();
                    const uint32_t d_addr = tmem_base + D_COL + (uint32_t)(f & 1) * kTok;
                    uint32_t acc = 0;
                    for (int g = 0; g < kFlush && kb < kblocks; ++g, ++kb) {
                        if (!wait_or_abort(&s_full[as], aph, abort_flag)) { give_up(p.status, abort_flag, 0x432); ok = false; break; }
                        tc_fence_after();
                        const uint64_t desc = desc_hi | (uint64_t)(b_lo0 + (uint32_t)as * (b_bytes >> 4));
                        const uint32_t a_addr = a_base + 32 * as;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            mma_f16_ts(d_addr, a_addr + 8 * j, desc + 2 * j, idesc, acc);
                            acc = 1u;
                        }
                        tc_commit(&s_empty[as]);
                        if (++as == AS) { as = 0; aph ^= 1u; }
                    }
                    if (ok) tc_commit(&d_full[f & 1]);
                }
                if (ok && lowrank && i >= 1 && !wait_or_abort(lr_free, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x431); ok = false; }
                if (ok && lowrank) {
                    if (!wait_or_abort(u_full, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x433); ok = false; }
                    if (ok && !wait_or_abort(t_full, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x434); ok = false; }
                    if (ok) {
                        tc_fence_after();
                        const uint32_t u_addr = smem_u32(ubuf);
#pragma unroll 1
                        for (int h = 0; h < 3; ++h) {
                            const uint32_t t_addr = smem_u32(tbuf + h * b_bytes);
#pragma unroll
                            for (int j = 0; j < 4; ++j)      // (zeros beyond r)
                                if (16 * j < p.r) mma_f16_ss(tmem_base + LR_COL, smem_desc_sw128(u_addr, 32 * j), smem_desc_sw128(t_addr, 32 * j),
                                           idesc, (h | j) ? 1u : 0u);
                        }
                        tc_commit(u_empty);
                        tc_commit(t_empty);
                        tc_commit(lr_full);
                    }
                }
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
        int f = 0;
        for (int i = 0; i < my_tiles && ok; ++i) {
            const int n0 = tile_n0(i), t0 = tile_t0(i), buf = i & 1;
            const int n = n0 + e;
            const bool valid_row = n < p.N;
            const float alpha_n = valid_row ? __ldg(p.alpha + n) : 0.f;
            const float mu_n = (p.mu && valid_row) ? __ldg(p.mu + n) : 0.f;
            if (lowrank) {
                // this tile's rows of U: 128 rows x 8 chunks of 16 bytes, 128B-swizzled K-major, zero beyond N and r
                if (ok && i >= 1 && !warp_wait(u_empty, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x440); ok = false; }
                if (ok) {
                    const bool vec = (p.r % 8 == 0) && ((reinterpret_cast<uintptr_t>(p.U) & 15) == 0);
#pragma unroll
                    for (int it = 0; it < 4; ++it) {
                        const int idx = it * 256 + half * 128 + e;
                        const int ur = idx >> 3, ch = idx & 7;
                        uint4 v = make_uint4(0u, 0u, 0u, 0u);
                        const int un = n0 + ur;
                        if (un < p.N && ch * 8 < p.r) {
                            const __nv_bfloat16* src = p.U + (int64_t)un * p.r + ch * 8;
                            if (vec) {
                                v = __ldg(reinterpret_cast<const uint4*>(src));
                            } else {
                                uint32_t w[4] = {0u, 0u, 0u, 0u};
                                for (int c = 0; c < 8 && ch * 8 + c < p.r; ++c)
                                    w[c >> 1] |= (uint32_t)__bfloat16_as_ushort(src[c]) << (16 * (c & 1));
                                v = make_uint4(w[0], w[1], w[2], w[3]);
                            }
                        }
                        *reinterpret_cast<uint4*>(ubuf + ur * 128 + ((ch ^ (ur & 7)) << 4)) = v;
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(u_full);
                }
            }
            float run[64];
#pragma unroll
            for (int c = 0; c < 64; ++c) run[c] = 0.f;
            for (int g = 0; g < groups && ok; ++g, ++f) {
                if (!warp_wait(&d_full[f & 1], (uint32_t)((f >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x442); ok = false; break; }
                tc_fence_after();
                const uint32_t d_addr = tmem_base + lane_addr + D_COL + (uint32_t)(f & 1) * kTok + 64 * half;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t v[16];
                    tmem_ld_32x16(d_addr + 16 * c, v);
                    tc_wait_ld();
                    if (c == 3) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_free[f & 1]);
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) run[16 * c + j] += __uint_as_float(v[j]);
                }
            }
            if (i == 0) griddep_wait();                       // nothing is stored before the preceding kernel has completed
            if (ok && !warp_wait(&tok_full[buf], (uint32_t)((i >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x441); ok = false; }
            if (ok && lowrank && !warp_wait(lr_full, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x443); ok = false; }
            if (ok) {
                tc_fence_after();
                const float4* ys_s = reinterpret_cast<const float4*>(tok_sum(buf));
                // (stores: lanes with neighbouring rows swap halves, as in gemm_umma_persist.cu)
                const int odd = lane & 1;
                const uint32_t sel = odd ? 0x3276u : 0x5410u;
                const int n_pair = n & ~1;
                const bool pair_ok = ((reinterpret_cast<uintptr_t>(p.out) & 3) == 0) && (p.ldo & 1) == 0 && n_pair + 1 < p.N;
                const bool whole = __all_sync(0xFFFFFFFFu, pair_ok) && t0 + kTok <= p.M;
                __nv_bfloat16* at = p.out + (int64_t)(t0 + 64 * half + odd) * p.ldo + n_pair;
                const int64_t step = 2 * p.ldo;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t l[16];
                    if (lowrank) {
                        tmem_ld_32x16(tmem_base + lane_addr + LR_COL + 64 * half + 16 * c, l);
                        tc_wait_ld();
                        if (c == 3) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(lr_free);
                        }
                    }
                    const int tok0 = 64 * half + 16 * c;
                    if (t0 + tok0 >= p.M) continue;              // warp-uniform; nothing of this chunk is stored
#pragma unroll
                    for (int j = 0; j < 16; j += 4) {
                        const float4 ys = ys_s[(tok0 + j) >> 2];
                        const float yss[4] = {ys.x, ys.y, ys.z, ys.w};
                        float y[4];
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            y[h] = fmaf(mu_n, yss[h], fmaf(alpha_n, run[16 * c + j + h], lowrank ? __uint_as_float(l[j + h]) : 0.f));
#pragma unroll
                        for (int h = 0; h < 4; h += 2) {
                            const uint32_t word = pack_bf16x2(y[h], y[h + 1]);      // two tokens of this lane's row
                            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, word, 1);
                            const int t = t0 + tok0 + j + h;
                            if (whole) {
                                *reinterpret_cast<uint32_t*>(at) = __byte_perm(word, other, sel);
                                at += step;
                            } else if (pair_ok) {
                                if (t + odd < p.M) *reinterpret_cast<uint32_t*>(p.out + (int64_t)(t + odd) * p.ldo + n_pair) = __byte_perm(word, other, sel);
                            } else if (valid_row) {
                                if (t < p.M) p.out[(int64_t)t * p.ldo + n] = __ushort_as_bfloat16((unsigned short)word);
                                if (t + 1 < p.M) p.out[(int64_t)(t + 1) * p.ldo + n] = __ushort_as_bfloat16((unsigned short)(word >> 16));
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
        set_regs_dec<kRegsExpand>();
        // ---------------- expansion of sign bits into the operand ring (tile boundaries do not matter here) ----------------
        const int q = warp & 3;
        const int part = (warp - 12) >> 2;             // which of the EW warps of the lane quarter
        const int row = q * 32 + lane;
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        // A warp's words of a unit go to registers, a unit ahead, and the stage is let go at once (see gemm_umma_persist.cu).
        // Block g of this CTA (a running count over its tiles) belongs to part g % EW and to stage g % AS.  AS is a multiple of
        // EW, so a stage always has the same owner and the owner is never more than one phase ahead of the stage's consumer: a
        // parity wait cannot tell a phase from the one two before it.  (The last unit of a row may hold fewer than sixteen
        // blocks, which is why neither follows from the position inside the unit.)
        constexpr int PER = kUnitK / kBlockK / EW;
        int ws = 0; uint32_t wph = 0;
        const int total = my_tiles * units;
        int c = 0, u_nxt = 0;                         // next unit to take: running number, position in its row
        int base_nxt = 0;                             // blocks of this CTA before it
        uint2 nxt[PER];
        int ns_nxt = 0, first_nxt = 0, g_nxt = 0;
        bool ok = true;
        auto take = [&]() {                           // (the unit's stage is full)
            ns_nxt = min(kUnitK / kBlockK, (p.K - unit_at(u_nxt) * kUnitK) / kBlockK);
            first_nxt = (part + EW - base_nxt % EW) % EW;
            g_nxt = base_nxt + first_nxt;
            const uint8_t* wrow = wbuf + ws * w_bytes + row * 128;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int blk = first_nxt + EW * q;                   // 8 bytes of the row's 128
                nxt[q] = lds_words(wrow + (((blk >> 1) ^ (row & 7)) << 4) + 8 * (blk & 1));
            }
            // (behind the loads' data: see release_stage)
            uint32_t seen = 0u;
#pragma unroll
            for (int q = 0; q < PER; ++q) seen ^= nxt[q].x ^ nxt[q].y;
            release_stage(&w_empty[ws], seen);
            if (++ws == WS) { ws = 0; wph ^= 1u; }
            base_nxt += ns_nxt;
            if (++u_nxt == units) u_nxt = 0;
            ++c;
        };
        if (total > 0) {
            if (!warp_wait(&w_full[ws], wph, abort_flag)) { give_up(p.status, abort_flag, 0x450); ok = false; }
            else take();
        }
        for (int i = 0; i < total && ok; ++i) {
            uint2 cur[PER];
#pragma unroll
            for (int q = 0; q < PER; ++q) cur[q] = nxt[q];
            const int ns = ns_nxt, first = first_nxt, g = g_nxt;
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                if (c == i + 1 && c < total && __all_sync(0xFFFFFFFFu, mbar_test_wait(&w_full[ws], wph))) take();
                if (first + EW * q < ns && ok) {
                    const int as = (g + EW * q) % AS;
                    const uint32_t aph = (uint32_t)(((g + EW * q) / AS) & 1);
                    if (!__all_sync(0xFFFFFFFFu, mbar_test_wait(&s_empty[as], aph ^ 1u))) {
                        griddep_wait();
                        if (!warp_wait(&s_empty[as], aph ^ 1u, abort_flag)) { give_up(p.status, abort_flag, 0x451); ok = false; }
                    }
                    if (ok) {
                        tc_fence_after();
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const uint32_t w = ~(k == 0 ? cur[q].x : cur[q].y);       // a set bit now means -1
                            uint32_t v[16];
#pragma unroll
                            for (int j = 0; j < 16; ++j) v[j] = ((w << (15 - j)) & 0x80008000u) | 0x3F803F80u;
                            tmem_st_32x16(tmem_base + lane_addr + A_COL + 32 * as + 16 * k, v);
                        }
                        tc_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&s_full[as]);
                    }
                }
            }
            if (c == i + 1 && c < total && ok) {
                if (!warp_wait(&w_full[ws], wph, abort_flag)) { give_up(p.status, abort_flag, 0x452); ok = false; }
                else take();
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, TMEM_COLS);
    }
}

bool a16_persistent_supports(int64_t K) { return K % 128 == 0; }       // (16-byte strides of the sign words' rows)

int launch_a16_persistent(const void* yhat, const float* ysum, int64_t M64, int64_t K64, int64_t N64, const uint32_t* packed,
                          const float* alpha, const float* mu, const void* U, int r, const void* Thl, void* out, int64_t ldo,
                          uint32_t* status, cudaStream_t stream) {
    using namespace a16p;
    const int M = (int)M64, N = (int)N64, K = (int)K64;
    const int sms = sm_count();
    if (sms <= 0) return BWLA_ERR_CUDA;
    CUtensorMap wm, bm, tm;
    {
        const uint64_t dims[2] = {(uint64_t)K / 32, (uint64_t)N};
        const uint64_t strides[1] = {(uint64_t)K / 8};
        const uint32_t box[2] = {32, kRows};
        int st = make_map(&wm, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, packed, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
        if (st != BWLA_OK) return st;
    }
    {
        const uint64_t dims[2] = {(uint64_t)K, (uint64_t)M};
        const uint64_t strides[1] = {(uint64_t)K * 2};
        const uint32_t box[2] = {kBlockK, kTok};
        int st = make_map(&bm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, yhat, dims, strides, box,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
        if (st != BWLA_OK) return st;
    }
    if (r > 0) {
        const uint64_t dims[3] = {(uint64_t)kLowrankPad, (uint64_t)M, 3};
        const uint64_t strides[2] = {(uint64_t)kLowrankPad * 2, (uint64_t)M * kLowrankPad * 2};
        const uint32_t box[3] = {(uint32_t)kLowrankPad, kTok, 1};
        int st = make_map(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, Thl, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
        if (st != BWLA_OK) return st;
    } else {
        tm = bm;   // never dereferenced
    }
    A16PersistParams p{};
    p.M = M; p.N = N; p.K = K; p.row_tiles = (N + kRows - 1) / kRows; p.tok_tiles = (M + kTok - 1) / kTok; p.r = r;
    p.alpha = alpha; p.mu = mu; p.ysum = ysum; p.U = (const __nv_bfloat16*)U; p.out = (__nv_bfloat16*)out; p.ldo = ldo; p.status = status;
    const int tiles = p.row_tiles * p.tok_tiles;

    static thread_local int configured = -1;
    int dev = 0;
    BWLA_CUDA_TRY(cudaGetDevice(&dev));
    if (configured != dev) {
        BWLA_CUDA_TRY(cudaFuncSetAttribute(a16_persistent_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, total));
        configured = dev;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)std::min(tiles, sms), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = total;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[1];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = launch_overlap_allowed();
    cfg.attrs = attrs;
    cfg.numAttrs = 1;
    ProfScope prof(kProfContraction, stream);
    cudaError_t e = cudaLaunchKernelEx(&cfg, a16_persistent_kernel, wm, bm, tm, p);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}

}  // namespace bwla
