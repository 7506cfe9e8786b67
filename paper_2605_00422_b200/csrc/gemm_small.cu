// The binary-weight contraction for a decode batch (up to 64 tokens) on warp-level int8 MMAs, every linear of a group in one
// launch.
//
//   tot[n][t] = sum_k bit(n,k) * q[t][k],   acc = 2 tot - sum_k q[t][k] - zp[t] * rowsum[n]            (sign = 2 bit - 1)
//   out[t][n] = bf16(alpha[n] * s_t * acc + U[n,:] . T[t,:] [+ mu[n] * s_t * sum_k (q[t][k] - zp[t])])  (Eq. 4; Sec. 3.2)
//
// Why not tcgen05 here: a decode contraction is a few microseconds of latencies, and one tcgen05.mma costs 51 cycles however
// few its tokens (80 weights per cycle and SM at any batch).  mma.sync m16n8k32 takes 2 cycles per SM for 512 weights x 8
// tokens (256 weights per cycle at 8 tokens, 128 at 16), and the sign bits become its A operand in registers, with no trip
// through tensor memory and no expander / issuer hand-over.
//
// Operand order.  A step is 128 values of k: lane t of a quad holds the sign word of the t-th 32 of them.  The interleaved code
// layout puts k = j + 8 i of every 32 at byte 4 j + i, so byte i of (word >> j) & 0x01010101 meets code word j; an MMA takes
// code words q and q + 4 of the four lanes.  With few tokens, where these instructions are the bound, 2 (or 4) neighbouring bit
// positions are left where they are and have accumulators of their own (masks 0x01.., 0x02.., ... of a word shifted by
// multiples of 2 (4) only), added with one shift each at the end.
//
// Work split.  CTA = RW row groups of 32 rows x KW K slices (16 warps; from 33 tokens on also x 2 token halves), one CTA per
// SM; it takes tiles of 32 RW rows in turn.  One thread streams the sign words by TMA (boxes of 32 RW rows x 1024 k, 128-byte
// swizzle) into a ring as deep as shared memory allows, starting before the preceding kernel has finished (no warp of its own:
// 16 warps may have 128 registers a thread, 17 only 96); the CTA's codes and T lie in shared memory for all its tiles (rows of
// 128 bytes, swizzled the same way: every read is free of bank conflicts).  K is split over a cluster of S CTAs where the codes
// would not fit or rows are few.  Partial sums meet in shared memory (of the CTA, then of the cluster), and the warps of a
// group share out the epilogue, which also evaluates U T (bf16 MMAs, three terms of T).
//
// PL = 3 is the weight-only operating point: an activation is a 23-bit fixed-point number of a power-of-two scale, kept as
// three signed base-256 digits (rot_mma.cu); the digits are contracted like three tokens' codes, exactly, and put together in
// the epilogue.
// Every wait is bounded (umma_wait.cuh).
#include <cuda_bf16.h>

#include <algorithm>

#include "bwla_common.cuh"
#include "rot_mma.cuh"
#include "tensor_map.cuh"
#include "umma_ptx.cuh"
#include "umma_wait.cuh"

namespace bwla {

using namespace ptx;

namespace small_ {
constexpr int kWarps = 16, kThreads = 32 * kWarps;
constexpr int kUnit = 1024, kSteps = 8;                       // k per ring stage; steps of 128 k in it
constexpr int kMaxStages = 12;
constexpr int kSmemMax = 232448 - 1024 - 256;                 // (the base is aligned to 1024 bytes; barriers are static)
// Warps a row group's tokens are dealt to: the accumulators of 64 tokens (12 tiles of digits) do not fit one warp's registers
// (each then expands the sign bits for itself, which its MMAs cover).
__host__ __device__ constexpr int token_warps(int NT) { return NT >= 8 ? 2 : 1; }
}  // namespace small_

struct SmallProblem {
    const int8_t* codes;                  // [PL][M][K]
    const float* scales; const int32_t* qsum; const int32_t* zp; const int32_t* rowsum;
    const float* alpha; const float* mu;
    const __nv_bfloat16* U; const __nv_bfloat16* Thl;
    __nv_bfloat16* out; int64_t ldo; int32_t* acc_debug;
    int N, r, tiles;
    int cluster_begin, clusters;          // clusters [cluster_begin, cluster_begin + clusters) of the launch
};
struct SmallParams {
    SmallProblem prob[kRotMaxProblems];
    int n_problems, M, K, units, S;
    int stages;                           // of the sign-word ring
    int flush;                            // rounds between cluster-wide reductions (S > 1)
    int ring_off, t_off, tok_off, red_off, csum_off;
    uint32_t* status;
};
struct SmallMaps { CUtensorMap w[kRotMaxProblems]; };

__device__ __forceinline__ void imma_16832(int32_t (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, int32_t x, int32_t y, int32_t z, int32_t w) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ void prefetch_l2_bulk(const void* p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// NTP: token tiles of 8; PL: digit planes per token; KW: warps that share a row group and split K; SPLIT: clusters split K
template <int NTP, int PL, int KW, bool SPLIT>
__global__ void __launch_bounds__(small_::kThreads, 1) gemm_small_kernel(const __grid_constant__ SmallMaps maps, const __grid_constant__ SmallParams p) {
    using namespace small_;
    constexpr int NT = NTP * PL, TW = token_warps(NT), NTPW = NTP / TW, NTW = NT / TW;        // ... W: of one warp
    constexpr int RW = kWarps / (KW * TW), TOK = 8 * NT, SETS = NT == 1 ? 4 : NT <= 3 ? 2 : 1;
    constexpr int CH = PL == 3 || NTPW < 2 ? 1 : 2, FR = 2 * CH;                              // token tiles, fragments reduced at a time
    constexpr int kStageBytes = RW * 32 * 128;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    __shared__ uint64_t full[kMaxStages], empty[kMaxStages];
    __shared__ int abort_word;
    volatile int* abort_flag = &abort_word;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int cl_all = (int)blockIdx.x / p.S, rank = SPLIT ? (int)blockIdx.x - cl_all * p.S : 0;
    int pi = 0;
    while (pi + 1 < p.n_problems && cl_all >= p.prob[pi + 1].cluster_begin) ++pi;
    const SmallProblem& pr = p.prob[pi];
    const int cl = cl_all - pr.cluster_begin, clusters = pr.clusters;
    const int ub = (int)((int64_t)p.units * rank / p.S), un = (int)((int64_t)p.units * (rank + 1) / p.S) - ub;   // this CTA's units
    const int rounds = (pr.tiles - cl + clusters - 1) / clusters;      // tiles cl, cl + clusters, ... (the same for a whole cluster)

    if (tid == 0) {
        abort_word = 0;
        for (int i = 0; i < p.stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], kWarps); }
        fence_barrier_init();
        fence_proxy_async();
    }
    __syncthreads();
    griddep_launch_dependents();

    // ---- sign words (constants of the layer): the ring is filled before the preceding kernel has finished, and refilled one
    //      stage behind the consumption, when every warp has let go of the stage before
    const int total = rounds * un;
    auto request = [&](int c) {                       // stage number c of this CTA's sequence (thread 0)
        const int i = c / un, u = c - i * un, st = c % p.stages;
        mbar_expect_tx(&full[st], kStageBytes);
        tma_load_2d_hint(smem + p.ring_off + st * kStageBytes, &maps.w[pi], (ub + u) * (kUnit / 32), (cl + i * clusters) * (32 * RW), &full[st],
                         l2_policy_evict_first());
    };
    if (tid == 0) {
        tma_prefetch_desc(&maps.w[pi]);
        for (int c = 0; c < min(p.stages, total); ++c) request(c);
    }
    // the rows of U the epilogues will want come from HBM too: into the L2 before they are needed
    if (pr.r > 0 && tid >= 32 && tid < 32 + rounds) {
        const int n0 = (cl + (tid - 32) * clusters) * (32 * RW);
        const uintptr_t lo = reinterpret_cast<uintptr_t>(pr.U + (int64_t)n0 * pr.r);
        const uintptr_t hi = reinterpret_cast<uintptr_t>(pr.U + (int64_t)min(n0 + 32 * RW, pr.N) * pr.r);
        const uintptr_t a0 = (lo + 15) & ~(uintptr_t)15;
        if (hi >= a0 + 16) prefetch_l2_bulk(reinterpret_cast<const void*>(a0), (uint32_t)((hi - a0) & ~(uintptr_t)15));
    }
    __syncwarp();
    griddep_wait();
    if (lane == 0 && p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0) *abort_flag = 1;      // the call already failed
    // ---- codes (128-byte rows: step of 128 k, token), T (128-byte rows: term, token) and the per-token scalars; the 16-byte
    //      pieces of a row are permuted by the token's low bits
    const int pieces = min(un * (kUnit / 16), (p.K >> 4) - ub * (kUnit / 16));
    for (int t = warp; t < PL * p.M; t += kWarps) {
        const int plane = PL > 1 ? t / p.M : 0, row = plane * (8 * NTP) + (t - plane * p.M);
        const int8_t* src = pr.codes + (int64_t)t * p.K + (int64_t)ub * kUnit;
        const uint32_t dst = smem_u32(smem) + row * 128;
        for (int c = lane; c < pieces; c += 32)
            cp_async16(dst + (uint32_t)((c >> 3) * (TOK * 128) + (((c & 7) ^ (row & 7)) << 4)), src + 16 * c);
    }
    if (pr.r > 0)
        for (int i = tid; i < 3 * p.M * 8; i += kThreads) {
            const int row = i >> 3, c = i & 7, h = row / p.M, t = row - h * p.M;
            cp_async16(smem_u32(smem) + (uint32_t)(p.t_off + (h * 8 * NTP + t) * 128 + ((c ^ (t & 7)) << 4)), pr.Thl + (int64_t)row * kLowrankPad + 8 * c);
        }
    float* sc_s = reinterpret_cast<float*>(smem + p.tok_off);
    int32_t *qs_s = reinterpret_cast<int32_t*>(sc_s) + TOK, *zp_s = qs_s + TOK;
    if (tid < TOK) {
        float sc = 0.f; int32_t qs = 0, zp = 0;
        const int plane = tid / (8 * NTP), t = tid - plane * (8 * NTP);
        if (t < p.M) {
            sc = pr.scales[t];
            const int4* parts = reinterpret_cast<const int4*>(pr.qsum + ((size_t)plane * p.M + t) * kQsumParts);
            const int4 a = parts[0], b = parts[1];
            qs = a.x + a.y + a.z + a.w + b.x + b.y + b.z + b.w;
            if (pr.zp) zp = pr.zp[t];
        }
        sc_s[tid] = sc; qs_s[tid] = qs; zp_s[tid] = zp;
    }
    cp_async_wait_all();
    __syncthreads();

    const int grp = warp / KW, kw = warp - grp * KW, rw = grp / TW, tw = grp - rw * TW;
    // this lane's code pieces of a step: token gq, pieces 2 tq and 2 tq + 1; its sign words: rows gq + 8 j, piece = the step
    const int b_lo = ((2 * tq) ^ gq) << 4, b_hi = ((2 * tq + 1) ^ gq) << 4;
    const uint8_t* w_base = smem + p.ring_off + (rw * 32 + gq) * 128 + 4 * tq;
    constexpr int SPW = kSteps / KW;                  // steps of a stage per warp
    const uint32_t red = smem_u32(smem) + p.red_off + (uint32_t)(grp * KW * FR * PL * 512 + lane * 16);
    const uint32_t csum = SPLIT ? smem_u32(smem) + p.csum_off + lane * 16 : 0u;

    // one fragment (16 rows x 8 tokens) of a finished tile
    auto epilogue = [&](int tile, int rg, int mt, int nt, const int32_t (&v)[PL][4]) {
        const int n_lo = (tile * RW + rg) * 32 + 16 * mt + gq, n_hi = n_lo + 8;
        const bool ok_lo = n_lo < pr.N, ok_hi = n_hi < pr.N;
        float lr[4] = {0.f, 0.f, 0.f, 0.f};
        if (pr.r > 0) {
            // U T with the 64 columns dealt to the quad's lanes, 16 each (a sum does not care in which order)
            uint32_t ul[8], uh[8];
            const __nv_bfloat16* u_lo = pr.U + (int64_t)(ok_lo ? n_lo : 0) * pr.r + 16 * tq;
            const __nv_bfloat16* u_hi = pr.U + (int64_t)(ok_hi ? n_hi : 0) * pr.r + 16 * tq;
            if ((pr.r & 7) == 0 && (reinterpret_cast<uintptr_t>(pr.U) & 15) == 0) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool in = 16 * tq + 8 * h < pr.r;
                    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
                    const uint4 a = in ? __ldg(reinterpret_cast<const uint4*>(u_lo) + h) : z, b = in ? __ldg(reinterpret_cast<const uint4*>(u_hi) + h) : z;
                    ul[4 * h] = a.x; ul[4 * h + 1] = a.y; ul[4 * h + 2] = a.z; ul[4 * h + 3] = a.w;
                    uh[4 * h] = b.x; uh[4 * h + 1] = b.y; uh[4 * h + 2] = b.z; uh[4 * h + 3] = b.w;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int c0 = 16 * tq + 2 * c;
                    const uint32_t a0 = c0 < pr.r ? __bfloat16_as_ushort(u_lo[2 * c]) : 0u, a1 = c0 + 1 < pr.r ? __bfloat16_as_ushort(u_lo[2 * c + 1]) : 0u;
                    const uint32_t b0 = c0 < pr.r ? __bfloat16_as_ushort(u_hi[2 * c]) : 0u, b1 = c0 + 1 < pr.r ? __bfloat16_as_ushort(u_hi[2 * c + 1]) : 0u;
                    ul[c] = a0 | (a1 << 16); uh[c] = b0 | (b1 << 16);
                }
            }
            const uint32_t tb = smem_u32(smem) + p.t_off + (8 * nt + gq) * 128;
#pragma unroll
            for (int h = 2; h >= 0; --h) {             // small terms first
                const uint4 x = lds128(tb + h * (8 * NTP * 128) + (((2 * tq) ^ gq) << 4)), y = lds128(tb + h * (8 * NTP * 128) + (((2 * tq + 1) ^ gq) << 4));
                const uint32_t t8[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t ua[4] = {ul[2 * kk], uh[2 * kk], ul[2 * kk + 1], uh[2 * kk + 1]};
                    mma_16816<false>(lr, ua, t8[2 * kk], t8[2 * kk + 1], lr);
                }
            }
        }
        const float al[2] = {ok_lo ? __ldg(pr.alpha + n_lo) : 0.f, ok_hi ? __ldg(pr.alpha + n_hi) : 0.f};
        const float mu[2] = {pr.mu && ok_lo ? __ldg(pr.mu + n_lo) : 0.f, pr.mu && ok_hi ? __ldg(pr.mu + n_hi) : 0.f};
        const int32_t rs[2] = {pr.zp && ok_lo ? __ldg(pr.rowsum + n_lo) : 0, pr.zp && ok_hi ? __ldg(pr.rowsum + n_hi) : 0};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 8 * nt + 2 * tq + (i & 1), h = i >> 1, n = h ? n_hi : n_lo;
            const float sc = sc_s[t];
            float accf, qsf;
            if constexpr (PL == 1) {
                const int32_t qs = qs_s[t], zp = zp_s[t], acc = 2 * v[0][i] - qs - zp * rs[h];
                if (pr.acc_debug && t < p.M && (h ? ok_hi : ok_lo)) pr.acc_debug[(int64_t)t * pr.N + n] = acc;
                accf = (float)acc; qsf = (float)(qs - p.K * zp);
            } else {
                // the low two digits' sums together are still exact in int32 (|sum of a digit| <= 128 K)
                const int32_t q0 = qs_s[t], q1 = qs_s[t + 8 * NTP], q2 = qs_s[t + 16 * NTP];
                accf = fmaf((float)(2 * v[PL - 1][i] - q2), 65536.f, (float)(256 * (2 * v[PL / 2][i] - q1) + (2 * v[0][i] - q0)));
                qsf = fmaf((float)q2, 65536.f, (float)(256 * q1 + q0));
            }
            if (t < p.M && (h ? ok_hi : ok_lo) && pr.out) {
                const float y = fmaf(__fmul_rn(mu[h], sc), qsf, __fmul_rn(__fmul_rn(al[h], sc), accf) + lr[i]);
                pr.out[(int64_t)t * pr.ldo + n] = __float2bfloat16_rn(y);
            }
        }
    };

    int st = 0; uint32_t ph = 0;
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i < rounds; ++i) {
        const int tile = cl + i * clusters;
        int32_t acc[SETS][2][NTW][4];
#pragma unroll
        for (int s = 0; s < SETS; ++s)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int nt = 0; nt < NTW; ++nt)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[s][mt][nt][e] = 0;
#pragma unroll 1
        for (int u = 0; u < un; ++u) {
            if (ok && !warp_wait(&full[st], ph, abort_flag)) { give_up(p.status, abort_flag, 0x420); ok = false; }
            const uint8_t* w_stage = w_base + st * kStageBytes;
            uint32_t w[SPW][4];
#pragma unroll
            for (int x = 0; x < SPW; ++x)
#pragma unroll
                for (int j = 0; j < 4; ++j) w[x][j] = *reinterpret_cast<const uint32_t*>(w_stage + j * 1024 + (((kw * SPW + x) ^ gq) << 4));
            // column tile j of this warp: plane j / NTPW, token tile tw * NTPW + j % NTPW
            const uint8_t* b_unit = smem + (8 * NTPW * tw + gq) * 128 + (u * kSteps + kw * SPW) * (TOK * 128);
#pragma unroll
            for (int x = 0; x < SPW; ++x) {
                uint32_t a[2][4][4];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const uint32_t lo = w[x][2 * mt], hi = w[x][2 * mt + 1];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int sh = q & ~(SETS - 1);
                        const uint32_t m = 0x01010101u << (q & (SETS - 1));
                        a[mt][q][0] = (lo >> sh) & m; a[mt][q][1] = (hi >> sh) & m;
                        a[mt][q][2] = (lo >> (sh + 4)) & m; a[mt][q][3] = (hi >> (sh + 4)) & m;
                    }
                }
#pragma unroll
                for (int nt = 0; nt < NTW; ++nt) {
                    const uint8_t* at = b_unit + (x * TOK + 8 * ((nt / NTPW) * NTP + nt % NTPW)) * 128;
                    const uint4 c0 = *reinterpret_cast<const uint4*>(at + b_lo), c1 = *reinterpret_cast<const uint4*>(at + b_hi);
                    const uint32_t bl[4] = {c0.x, c0.y, c0.z, c0.w}, bh[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
                            imma_16832(acc[q & (SETS - 1)][mt][nt], a[mt][q][0], a[mt][q][1], a[mt][q][2], a[mt][q][3], bl[q], bh[q]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[st]);
            if (tid == 0) {
                const int c = i * un + u - 1;         // the stage before this one
                if (c >= 0 && c + p.stages < total && !*abort_flag) {
                    if (wait_or_abort(&empty[st > 0 ? st - 1 : p.stages - 1], st > 0 ? ph : ph ^ 1u, abort_flag)) request(c + p.stages);
                    else give_up(p.status, abort_flag, 0x410);
                }
            }
            if (++st == p.stages) { st = 0; ph ^= 1u; }
        }
        // ---- the KW slices of the tile meet, CH token tiles at a time
#pragma unroll
        for (int c0 = 0; c0 < NTPW; c0 += CH) {
#pragma unroll
            for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                for (int c = 0; c < CH; ++c)
#pragma unroll
                    for (int pl = 0; pl < PL; ++pl) {
                        int32_t v[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            v[e] = acc[0][mt][pl * NTPW + c0 + c][e];
#pragma unroll
                            for (int z = 1; z < SETS; ++z) v[e] += acc[z][mt][pl * NTPW + c0 + c][e] >> z;
                        }
                        sts128(red + (uint32_t)(((kw * FR + mt * CH + c) * PL + pl) * 512), v[0], v[1], v[2], v[3]);
                    }
            named_barrier(1 + grp, 32 * KW);
#pragma unroll 1
            for (int f = kw; f < FR; f += KW) {
                int32_t v[PL][4];
#pragma unroll
                for (int pl = 0; pl < PL; ++pl) {
                    v[pl][0] = v[pl][1] = v[pl][2] = v[pl][3] = 0;
#pragma unroll
                    for (int k = 0; k < KW; ++k) {
                        const uint4 q = lds128(red + (uint32_t)(((k * FR + f) * PL + pl) * 512));
                        v[pl][0] += (int32_t)q.x; v[pl][1] += (int32_t)q.y; v[pl][2] += (int32_t)q.z; v[pl][3] += (int32_t)q.w;
                    }
                }
                const int mt = f / CH, nt = NTPW * tw + c0 + f - mt * CH;
                if (!SPLIT) {
                    if (!*abort_flag) epilogue(tile, rw, mt, nt, v);
                } else {
#pragma unroll
                    for (int pl = 0; pl < PL; ++pl)
                        sts128(csum + (uint32_t)(((((i % p.flush) * RW + rw) * 2 * NTP + 2 * nt + mt) * PL + pl) * 512), v[pl][0], v[pl][1], v[pl][2], v[pl][3]);
                }
            }
            named_barrier(1 + grp, 32 * KW);          // (the buffer may be written again)
        }
        if (SPLIT && ((i + 1) % p.flush == 0 || i + 1 == rounds)) {
            // ---- the cluster's partial sums: every CTA takes its share of the fragments of the last rounds
            cluster_arrive_release(); cluster_wait_acquire();
            const int first = i / p.flush * p.flush, items = (i + 1 - first) * RW * 2 * NTP;
#pragma unroll 1
            for (int it = rank + p.S * warp; it < items && !*abort_flag; it += p.S * kWarps) {
                const int rel = it / (2 * NTP), f = it - rel * 2 * NTP;
                int32_t v[PL][4];
#pragma unroll
                for (int pl = 0; pl < PL; ++pl) {
                    const uint32_t at = csum + (uint32_t)((it * PL + pl) * 512);
                    uint4 q[8];
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (s < p.S) q[s] = ld_shared_cluster_v4(map_shared_rank(at, (uint32_t)s));
                    v[pl][0] = v[pl][1] = v[pl][2] = v[pl][3] = 0;
#pragma unroll
                    for (int s = 0; s < 8; ++s)
                        if (s < p.S) { v[pl][0] += (int32_t)q[s].x; v[pl][1] += (int32_t)q[s].y; v[pl][2] += (int32_t)q[s].z; v[pl][3] += (int32_t)q[s].w; }
                }
                epilogue(cl + (first + rel / RW) * clusters, rel % RW, f & 1, f >> 1, v);
            }
            cluster_arrive_release(); cluster_wait_acquire();       // everybody has read: the buffers may be written again
        }
    }
    if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);   // let copies in flight land
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
struct SmallPlan { int S, KW, stages, flush, ring_off, t_off, tok_off, red_off, csum_off, smem; int clusters[kRotMaxProblems]; };

static int token_tiles(int64_t M) { return M <= 8 ? 1 : M <= 16 ? 2 : M <= 32 ? 4 : 8; }
static int tile_rows(int NT, int KW) { return 32 * (small_::kWarps / (KW * small_::token_warps(NT))); }

// Shared memory for S CTAs per cluster and KW K slices; false when it does not fit.
static bool small_layout(int NTP, int PL, int units, int S, int KW, bool lowrank, int rounds, int most_stages, SmallPlan* out) {
    using namespace small_;
    const int NT = NTP * PL, tok = 8 * NT, ch = PL == 3 || NTP / token_warps(NT) < 2 ? 1 : 2, rows = tile_rows(NT, KW);
    SmallPlan pl{};
    pl.S = S; pl.KW = KW;
    int off = ((units + S - 1) / S) * kSteps * tok * 128;
    pl.t_off = off; off += lowrank ? 3 * 8 * NTP * 128 : 0;
    pl.red_off = off; off += kWarps * 2 * ch * PL * 512;
    pl.csum_off = off;
    pl.flush = 1;
    const int stage = rows * 128, per_round = rows / 32 * 2 * NT * 512, tok_bytes = (12 * tok + 1023) / 1024 * 1024;
    if (S > 1) {
        pl.flush = std::max(1, std::min(rounds, (kSmemMax - off - tok_bytes - 4 * stage) / per_round));
        off += pl.flush * per_round;
    }
    pl.tok_off = off; off += tok_bytes;
    pl.ring_off = off = (off + 1023) / 1024 * 1024;
    pl.stages = std::min(std::min(kMaxStages, most_stages), (kSmemMax - off) / stage);
    if (pl.stages < std::min(2, most_stages)) return false;
    pl.smem = off + pl.stages * stage + 1024;
    *out = pl;
    return true;
}

// How many clusters of S such CTAs the device holds at once.  (Clusters are placed inside a GPC, so this is less than SMs / S:
// asked once per size and thread.)
static int resident_small_clusters(int S) {
    static thread_local int known[9], known_dev = -1;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    if (known_dev != dev) { for (int& k : known) k = -1; known_dev = dev; }
    if (known[S] < 0) {
        auto kernel = gemm_small_kernel<2, 1, 4, true>;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(S * sm_count()), 1, 1);
        cfg.blockDim = dim3(small_::kThreads, 1, 1);
        cfg.dynamicSmemBytes = small_::kSmemMax + 1024;
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = (unsigned)S; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a; cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, small_::kSmemMax + 1024) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        known[S] = n;
    }
    return known[S];
}

// Picks S and KW by an estimate of cycles: rounds x (stages per tile x MMA or ALU cycles of the 16 warps, plus the reduction
// and epilogue of a round), plus filling the CTA's codes from the L2, plus the cluster barriers.
static bool small_plan_search(int NTP, int PL, int units, const int64_t* N, int n, bool lowrank, int sms, SmallPlan* best) {
    using namespace small_;
    const int NT = NTP * PL;
    double best_cost = 0.0;
    bool found = false;
    for (int KW = 4; KW <= 8; KW *= 2)
        for (int S = 1; S <= 8 && S <= units; ++S) {
            const int rows = tile_rows(NT, KW);
            const int per_cta = (units + S - 1) / S;
            if (per_cta * kSteps * 8 * NT * 128 > kSmemMax) continue;
            const int total = S == 1 ? sms : resident_small_clusters(S);      // clusters the device holds
            if (total < n) break;
            int tiles[kRotMaxProblems], cl[kRotMaxProblems], used = 0, rounds = 1;
            int64_t all = 0;
            for (int i = 0; i < n; ++i) { tiles[i] = (int)((N[i] + rows - 1) / rows); all += tiles[i]; }
            // clusters per problem, by row tiles: at least one each, never more than tiles
            for (int i = 0; i < n; ++i) {
                cl[i] = (int)std::max<int64_t>(1, std::min<int64_t>(tiles[i], (int64_t)total * tiles[i] / all));
                used += cl[i];
            }
            while (used > total) {                                    // (only through the minimum of one each)
                int big = 0;
                for (int i = 1; i < n; ++i) if (cl[i] > cl[big]) big = i;
                --cl[big]; --used;
            }
            while (used < total) {                                    // what is left goes to whoever has most rounds
                int worst = -1, wr = 1;
                for (int i = 0; i < n; ++i) {
                    const int r = (tiles[i] + cl[i] - 1) / cl[i];
                    if (r > wr) { wr = r; worst = i; }
                }
                if (worst < 0) break;
                ++cl[worst]; ++used;
            }
            for (int i = 0; i < n; ++i) rounds = std::max(rounds, (tiles[i] + cl[i] - 1) / cl[i]);
            SmallPlan pl;
            if (!small_layout(NTP, PL, units, S, KW, lowrank, rounds, rounds * per_cta, &pl)) continue;
            // a stage is kSteps steps of the row groups: 4 x 2 x NT MMAs of 2 cycles, or about 60 ALU instructions of half a cycle
            const double stage_cycles = kSteps * (rows / 32) * (NT == 1 ? 32.0 : 16.0 * NT + 6.0);
            const double cost = rounds * (per_cta * stage_cycles + 900.0) + per_cta * kSteps * 8.0 * NT * 128.0 / 40.0 +
                                (S > 1 ? 2500.0 * ((rounds + pl.flush - 1) / pl.flush) : 0.0);
            if (!found || cost < best_cost) {
                best_cost = cost; *best = pl; found = true;
                for (int i = 0; i < n; ++i) best->clusters[i] = cl[i];
            }
        }
    return found;
}

// The plans of the shapes a thread has called lately: a decode loop asks for the same few on every step.
static bool small_plan(const GemmArgs* a, int n, int planes, SmallPlan* out) {
    using namespace small_;
    struct Key { int dev, NTP, PL, units, n, lowrank; int64_t N[kRotMaxProblems]; };
    struct Known { Key k; bool ok; SmallPlan plan; };
    static thread_local Known known[16];
    static thread_local int used = 0;
    const int64_t M = a[0].M, K = a[0].K;
    if (n < 1 || n > kRotMaxProblems || M < 1 || M > (planes == 3 ? 32 : 64) || K % 128 != 0 || (planes == 3 && K > 25600)) return false;
    Key k{};
    for (int i = 0; i < n; ++i) {
        if (a[i].N < 1 || a[i].N > ((int64_t)1 << 30) || a[i].r > kLowrankPad || M * a[i].N >= (int64_t)1 << 31) return false;
        k.N[i] = a[i].N;
        if (a[i].r > 0) k.lowrank = 1;
    }
    if (cudaGetDevice(&k.dev) != cudaSuccess) { cudaGetLastError(); return false; }
    k.NTP = token_tiles(M); k.PL = planes; k.units = (int)((K + kUnit - 1) / kUnit); k.n = n;
    auto same = [&](const Key& o) {
        return o.dev == k.dev && o.NTP == k.NTP && o.PL == k.PL && o.units == k.units && o.n == k.n && o.lowrank == k.lowrank &&
               std::equal(k.N, k.N + kRotMaxProblems, o.N);
    };
    for (int i = 0; i < 16 && i < used; ++i)
        if (same(known[i].k)) { *out = known[i].plan; return known[i].ok; }
    const int sms = sm_count();
    Known& slot = known[used % 16];
    slot.k = k;
    slot.ok = sms > 0 && encode_tiled_fn() && small_plan_search(k.NTP, k.PL, k.units, k.N, n, k.lowrank != 0, sms, &slot.plan);
    ++used;
    *out = slot.plan;
    return slot.ok;
}

bool gemm_small_fits(const GemmArgs* a, int n, int planes) {
    SmallPlan pl;
    return small_plan(a, n, planes, &pl);
}

template <int NTP, int PL, int KW, bool SPLIT>
static int launch_small_t(const SmallMaps& maps, const SmallParams& p, int grid, int smem, cudaStream_t stream) {
    auto kernel = gemm_small_kernel<NTP, PL, KW, SPLIT>;
    static thread_local int configured = -1;
    int dev = 0;
    BWLA_CUDA_TRY(cudaGetDevice(&dev));
    if (configured != dev) {
        BWLA_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, small_::kSmemMax + 1024));
        configured = dev;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(small_::kThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = launch_overlap_allowed();
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = (unsigned)p.S; attrs[1].val.clusterDim.y = 1; attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = SPLIT ? 2 : 1;
    ProfScope prof(kProfContraction, stream);
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, maps, p);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}
template <int NTP, int PL>
static int launch_small_nt(const SmallMaps& maps, const SmallParams& p, int KW, int grid, int smem, cudaStream_t stream) {
    if (KW == 4) return p.S > 1 ? launch_small_t<NTP, PL, 4, true>(maps, p, grid, smem, stream) : launch_small_t<NTP, PL, 4, false>(maps, p, grid, smem, stream);
    return p.S > 1 ? launch_small_t<NTP, PL, 8, true>(maps, p, grid, smem, stream) : launch_small_t<NTP, PL, 8, false>(maps, p, grid, smem, stream);
}

// All problems have the same M, K and bits; a[i].codes: int8 [planes][M][K] in the interleaved order; a[i].Thl: bf16 [3][M][64].
// *taken is false where the shapes do not fit (nothing has been launched then).
int launch_gemm_small(const GemmArgs* a, int n, int planes, bool* taken, cudaStream_t stream) {
    SmallPlan pl;
    *taken = small_plan(a, n, planes, &pl);
    if (!*taken) return BWLA_OK;
    const int M = (int)a[0].M, K = (int)a[0].K, NTP = token_tiles(M);
    SmallParams p{};
    SmallMaps maps;
    p.n_problems = n; p.M = M; p.K = K; p.units = (K + small_::kUnit - 1) / small_::kUnit; p.S = pl.S; p.stages = pl.stages; p.flush = pl.flush;
    p.ring_off = pl.ring_off; p.t_off = pl.t_off; p.tok_off = pl.tok_off; p.red_off = pl.red_off; p.csum_off = pl.csum_off;
    p.status = a[0].status;
    const int rows = tile_rows(NTP * planes, pl.KW);
    int begin = 0;
    for (int i = 0; i < n; ++i) {
        SmallProblem& q = p.prob[i];
        q.codes = a[i].codes; q.scales = a[i].scales; q.qsum = a[i].qsum; q.zp = a[i].zp; q.rowsum = a[i].rowsum;
        q.alpha = a[i].alpha; q.mu = a[i].mu; q.U = (const __nv_bfloat16*)a[i].U; q.Thl = (const __nv_bfloat16*)a[i].Thl;
        q.out = (__nv_bfloat16*)a[i].out; q.ldo = a[i].ldo; q.acc_debug = a[i].acc_debug;
        q.N = (int)a[i].N; q.r = a[i].r; q.tiles = ((int)a[i].N + rows - 1) / rows; q.cluster_begin = begin; q.clusters = pl.clusters[i];
        begin += pl.clusters[i];
        const uint64_t dims[2] = {(uint64_t)K / 32, (uint64_t)a[i].N};
        const uint64_t strides[1] = {(uint64_t)K / 8};
        const uint32_t box[2] = {32, (uint32_t)rows};
        int st = make_map(&maps.w[i], CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, a[i].packed, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B);
        if (st != BWLA_OK) return st;
    }
    for (int i = n; i < kRotMaxProblems; ++i) maps.w[i] = maps.w[0];
    const int grid = begin * pl.S;
    if (planes == 3) {
        switch (NTP) {
            case 1: return launch_small_nt<1, 3>(maps, p, pl.KW, grid, pl.smem, stream);
            case 2: return launch_small_nt<2, 3>(maps, p, pl.KW, grid, pl.smem, stream);
            default: return launch_small_nt<4, 3>(maps, p, pl.KW, grid, pl.smem, stream);
        }
    }
    switch (NTP) {
        case 1: return launch_small_nt<1, 1>(maps, p, pl.KW, grid, pl.smem, stream);
        case 2: return launch_small_nt<2, 1>(maps, p, pl.KW, grid, pl.smem, stream);
        case 4: return launch_small_nt<4, 1>(maps, p, pl.KW, grid, pl.smem, stream);
        default: return launch_small_nt<8, 1>(maps, p, pl.KW, grid, pl.smem, stream);
    }
}

}  // namespace bwla
