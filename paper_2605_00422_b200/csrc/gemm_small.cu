// The binary-weight contraction for a decode batch (up to 16 tokens, 4 as digits) on warp-level int8 MMAs, every linear of a group in
// one launch.
//
//   tot[n][t] = sum_k bit(n,k) * q[t][k],   acc = 2 tot - sum_k q[t][k] - zp[t] * rowsum[n]            (sign = 2 bit - 1)
//   out[t][n] = bf16(alpha[n] * s_t * acc + U[n,:] . T[t,:] [+ mu[n] * s_t * sum_k (q[t][k] - zp[t])])  (Eq. 4; Sec. 3.2)
//
// Why not tcgen05 here: a decode contraction is a few microseconds of latencies, and one tcgen05.mma costs 51 cycles however
// few its tokens (80 weights per cycle and SM at any batch).  mma.sync m16n8k32 takes 2 cycles per SM for 512 weights x 8
// tokens (256 weights per cycle at 8 tokens, 128 at 16), and the sign bits become its A operand in registers, with no trip
// through tensor memory and no expander / issuer hand-over.
//
// Operand order.  An item is 32 rows x 512 values of k: lane t of a quad holds the four sign words of the t-th 128 of them, for
// rows gq + 8 j.  The interleaved code layout puts k = j + 8 i of every 32 at byte 4 j + i, so byte i of (word >> j) & 0x01010101
// meets code word j; an MMA takes code words q and q + 4 of the four lanes' words.  With few tokens, where these instructions
// are the bound, 2 (or 4) neighbouring bit positions are left where they are and have accumulators of their own (masks 0x01..,
// 0x02.., ... of a word shifted by multiples of 2 (4) only), added with one shift each at the end.
//
// Work split.  A CTA (16 warps, one CTA per SM) owns a run of 32-row groups; the items of a run go to the warps in equal
// contiguous shares, with no barrier until all are done: a warp loads its sign words straight into registers, one item ahead,
// and adds its sums to the CTA's in shared memory when it leaves a group.  (Tiles of 128 rows whose K was shared by four
// warps, behind a TMA ring, spent half of their time at barriers and in the epilogue of every tile.)  The rows' sign words,
// scales and rows of U are asked into the L2 before the preceding kernel has finished; the CTA's codes and T lie in shared
// memory (rows of 128 bytes, permuted so that every read is free of bank conflicts).  K is split over a cluster of S CTAs
// where the codes would not fit or rows are few.  The epilogue, once per run, also evaluates U T (bf16 MMAs, three terms of T).
//
// PL = 3 is the weight-only operating point for up to 4 tokens whose codes fit one CTA (more: gemm_umma.cu): an activation is a
// 23-bit fixed-point number of a power-of-two scale, kept as
// three signed base-256 digits (rot_mma.cu); the digits are contracted like three tokens' codes, exactly, and put together in
// the epilogue.
#include <cuda_bf16.h>

#include <algorithm>

#include "bwla_common.cuh"
#include "rot_mma.cuh"
#include "umma_ptx.cuh"

namespace bwla {

using namespace ptx;

namespace small_ {
constexpr int kWarps = 16, kThreads = 32 * kWarps;
constexpr int kUnit = 512, kSteps = 4;                        // k per item; code rows of 128 k in it
constexpr int kSmemMax = 232448 - 256;
}  // namespace small_

struct SmallProblem {
    const uint32_t* packed; const int8_t* codes;              // codes [PL][M][K]
    const float* scales; const int32_t* qsum; const int32_t* zp; const int32_t* rowsum;
    const float* alpha; const float* mu;
    const __nv_bfloat16* U; const __nv_bfloat16* Thl;
    __nv_bfloat16* out; int64_t ldo; int32_t* acc_debug;
    int N, r, groups;                     // 32-row groups
    int cluster_begin, clusters;          // clusters [cluster_begin, cluster_begin + clusters) of the launch
};
struct SmallParams {
    SmallProblem prob[kRotMaxProblems];
    int n_problems, M, K, units, S;
    int run;                              // groups whose sums fit shared memory at a time
    int t_off, tok_off, acc_off;
    uint32_t* status;
};

__device__ __forceinline__ void imma_16832(int32_t (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void red_shared_add(uint32_t addr, int32_t v) { asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ int32_t ld_cluster_s32(uint32_t addr) {
    int32_t v;
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// sign words: read once, straight to registers
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// NTP: token tiles of 8; PL: digit planes per token; SPLIT: clusters split K
template <int NTP, int PL, bool SPLIT>
__global__ void __launch_bounds__(small_::kThreads, 1) gemm_small_kernel(const __grid_constant__ SmallParams p) {
    using namespace small_;
    constexpr int NT = NTP * PL;
    constexpr bool AHEAD = NT == 1;                   // (registers: beyond that the rows of a fragment are fetched when its turn comes)
    constexpr int TOK = 8 * NT, SETS = NT == 1 ? 4 : NT <= 3 ? 2 : 1;
    extern __shared__ __align__(16) uint8_t smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
    const int cl_all = (int)blockIdx.x / p.S, rank = SPLIT ? (int)blockIdx.x - cl_all * p.S : 0;
    int pi = 0;
    while (pi + 1 < p.n_problems && cl_all >= p.prob[pi + 1].cluster_begin) ++pi;
    const SmallProblem& pr = p.prob[pi];
    const int cl = cl_all - pr.cluster_begin;
    const int ub = (int)((int64_t)p.units * rank / p.S), un = (int)((int64_t)p.units * (rank + 1) / p.S) - ub;   // this CTA's units
    const int g_lo = (int)((int64_t)pr.groups * cl / pr.clusters), g_hi = (int)((int64_t)pr.groups * (cl + 1) / pr.clusters);
    const int row_bytes = p.K >> 3;

    griddep_launch_dependents();
    // ---- constants of the layer, before the preceding kernel has finished: this CTA's share of the sign words, and its rows' scales
    //      and rows of U, into the L2
    {
        const int rows = min((g_hi - g_lo) * 32, pr.N - g_lo * 32);
        const uint8_t* w = reinterpret_cast<const uint8_t*>(pr.packed) + (int64_t)g_lo * 32 * row_bytes + ub * (kUnit / 8);
        const uint32_t bytes = (uint32_t)min(un * (kUnit / 8), row_bytes - ub * (kUnit / 8));
        for (int i = tid; i < rows; i += kThreads) prefetch_l2_bulk(w + (int64_t)i * row_bytes, bytes);
        for (int i = tid; i < (rows + 31) / 32; i += kThreads) {
            const int n0 = (g_lo + i) * 32;
            prefetch_l2_line(pr.alpha + n0);
            if (pr.mu) prefetch_l2_line(pr.mu + n0);
            if (pr.zp) prefetch_l2_line(pr.rowsum + n0);
        }
        // (line by line: bulk prefetches of U behind those of the sign words were seen to arrive late)
        if (pr.r > 0) {
            const uint8_t* u = reinterpret_cast<const uint8_t*>(pr.U) + (int64_t)g_lo * 32 * pr.r * 2;
            for (int i = 128 * tid; i < rows * pr.r * 2; i += 128 * kThreads) prefetch_l2_line(u + i);
        }
    }
    // this warp's items of a run of `n` groups from `g`: [lo, hi) in the order (group, unit)
    int g = g_lo, n = min(p.run, g_hi - g_lo), it, it_end;
    auto share = [&]() {
        const int all = n * un;
        it = all * warp / kWarps; it_end = all * (warp + 1) / kWarps;
    };
    share();
    auto load_w = [&](uint4 (&w)[4], int item) {
        const int sub = item / un, u = item - sub * un;
        const int n0 = (g + sub) * 32 + gq, k16 = (ub + u) * (kUnit / 128) + tq;            // 16-byte pieces of a row
        const uint8_t* at = reinterpret_cast<const uint8_t*>(pr.packed) + 16 * k16;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            w[j] = 128 * k16 < p.K ? ldg_stream(at + (int64_t)min(n0 + 8 * j, pr.N - 1) * row_bytes) : make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 wn[4];
    if (it < it_end) load_w(wn, it);
    int32_t* const accs = reinterpret_cast<int32_t*>(smem + p.acc_off);      // [group of the run][row half][column tile][4][32 lanes]
    for (int i = tid; i < p.run * 2 * NT * 32; i += kThreads) reinterpret_cast<uint4*>(accs)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (warp == 0) {
        if (lane == 0 && p.status) touch(p.status);
        if (lane == 1) touch(pr.codes);
        if (lane == 2 && pr.r > 0) touch(pr.U + (int64_t)g_lo * 32 * pr.r);
        if (lane == 3) touch(pr.alpha + g_lo * 32);
        if (lane == 4 && pr.out) touch(pr.out + g_lo * 32);
        if (lane == 5 && pr.r > 0) touch(pr.Thl);
    }
    griddep_wait();
    // ---- codes (128-byte rows: 128 k, token), T (128-byte rows: term, token) and the per-token scalars; the 16-byte pieces of a
    //      row are permuted by the token's low bits (and, for the codes, the row's place among the four of an item)
    const int pieces = min(un * (kUnit / 16), (p.K >> 4) - ub * (kUnit / 16));
    for (int t = warp; t < PL * p.M; t += kWarps) {
        const int plane = PL > 1 ? t / p.M : 0, row = plane * (8 * NTP) + (t - plane * p.M);
        const int8_t* src = pr.codes + (int64_t)t * p.K + (int64_t)ub * kUnit;
        const uint32_t dst = smem_u32(smem) + row * 128;
        for (int c = lane; c < pieces; c += 32)
            cp_async16(dst + (uint32_t)((c >> 3) * (TOK * 128) + (((c & 7) ^ (row & 7) ^ (((c >> 3) & 3) << 1)) << 4)), src + 16 * c);
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
    // (behind the copies: the look at the status word is a trip to the L2)
    const bool failed = p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0;       // the call already failed
    cp_async_wait_all();
    __syncthreads();

    // ---- epilogue of one fragment (16 rows x 8 tokens), in two halves: what it needs from global memory is requested a fragment
    //      ahead (an L2 round trip each otherwise: rows of U, then the scales, then the shifts)
    struct Rows { uint32_t ul[8], uh[8]; float al[2], mu[2]; int32_t rs[2]; };
    const bool u_vec = (pr.r & 7) == 0 && (reinterpret_cast<uintptr_t>(pr.U) & 15) == 0;
    auto fetch_rows = [&](Rows& w, int grp, int mt) {
        const int n_lo = grp * 32 + 16 * mt + gq, n_hi = n_lo + 8;
        const bool ok_lo = n_lo < pr.N, ok_hi = n_hi < pr.N;
        w.al[0] = ok_lo ? __ldg(pr.alpha + n_lo) : 0.f; w.al[1] = ok_hi ? __ldg(pr.alpha + n_hi) : 0.f;
        w.mu[0] = pr.mu && ok_lo ? __ldg(pr.mu + n_lo) : 0.f; w.mu[1] = pr.mu && ok_hi ? __ldg(pr.mu + n_hi) : 0.f;
        w.rs[0] = pr.zp && ok_lo ? __ldg(pr.rowsum + n_lo) : 0; w.rs[1] = pr.zp && ok_hi ? __ldg(pr.rowsum + n_hi) : 0;
        if (pr.r > 0) {
            // U T with the 64 columns dealt to the quad's lanes, 16 each (a sum does not care in which order)
            const __nv_bfloat16* u_lo = pr.U + (int64_t)(ok_lo ? n_lo : 0) * pr.r + 16 * tq;
            const __nv_bfloat16* u_hi = pr.U + (int64_t)(ok_hi ? n_hi : 0) * pr.r + 16 * tq;
            if (u_vec) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool in = 16 * tq + 8 * h < pr.r;
                    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
                    const uint4 a = in ? __ldg(reinterpret_cast<const uint4*>(u_lo) + h) : z, b = in ? __ldg(reinterpret_cast<const uint4*>(u_hi) + h) : z;
                    w.ul[4 * h] = a.x; w.ul[4 * h + 1] = a.y; w.ul[4 * h + 2] = a.z; w.ul[4 * h + 3] = a.w;
                    w.uh[4 * h] = b.x; w.uh[4 * h + 1] = b.y; w.uh[4 * h + 2] = b.z; w.uh[4 * h + 3] = b.w;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int c0 = 16 * tq + 2 * c;
                    const uint32_t a0 = c0 < pr.r ? __bfloat16_as_ushort(u_lo[2 * c]) : 0u, a1 = c0 + 1 < pr.r ? __bfloat16_as_ushort(u_lo[2 * c + 1]) : 0u;
                    const uint32_t b0 = c0 < pr.r ? __bfloat16_as_ushort(u_hi[2 * c]) : 0u, b1 = c0 + 1 < pr.r ? __bfloat16_as_ushort(u_hi[2 * c + 1]) : 0u;
                    w.ul[c] = a0 | (a1 << 16); w.uh[c] = b0 | (b1 << 16);
                }
            }
        }
    };
    auto epilogue = [&](const Rows& w, int grp, int mt, int nt, const int32_t (&v)[PL][4]) {
        const int n_lo = grp * 32 + 16 * mt + gq, n_hi = n_lo + 8;
        float lr[3][4];                                // the three terms of T side by side: three short chains instead of a long one
#pragma unroll
        for (int h = 0; h < 3; ++h) lr[h][0] = lr[h][1] = lr[h][2] = lr[h][3] = 0.f;
        if (pr.r > 0) {
            const uint8_t* tb = smem + p.t_off + (8 * nt + gq) * 128;
#pragma unroll
            for (int h = 0; h < 3; ++h) {
                const uint4 x = *reinterpret_cast<const uint4*>(tb + h * (8 * NTP * 128) + (((2 * tq) ^ gq) << 4));
                const uint4 y = *reinterpret_cast<const uint4*>(tb + h * (8 * NTP * 128) + (((2 * tq + 1) ^ gq) << 4));
                const uint32_t t8[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const uint32_t ua[4] = {w.ul[2 * kk], w.uh[2 * kk], w.ul[2 * kk + 1], w.uh[2 * kk + 1]};
                    mma_16816<false>(lr[h], ua, t8[2 * kk], t8[2 * kk + 1], lr[h]);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 8 * nt + 2 * tq + (i & 1), h = i >> 1, n = h ? n_hi : n_lo;
            const bool live = t < p.M && n < pr.N;
            const float sc = sc_s[t];
            float accf, qsf;
            if constexpr (PL == 1) {
                const int32_t qs = qs_s[t], zp = zp_s[t], acc = 2 * v[0][i] - qs - zp * w.rs[h];
                if (pr.acc_debug && live) pr.acc_debug[(int64_t)t * pr.N + n] = acc;
                accf = (float)acc; qsf = (float)(qs - p.K * zp);
            } else {
                // the low two digits' sums together are still exact in int32 (|sum of a digit| <= 128 K)
                const int32_t q0 = qs_s[t], q1 = qs_s[t + 8 * NTP], q2 = qs_s[t + 16 * NTP];
                accf = fmaf((float)(2 * v[PL - 1][i] - q2), 65536.f, (float)(256 * (2 * v[PL / 2][i] - q1) + (2 * v[0][i] - q0)));
                qsf = fmaf((float)q2, 65536.f, (float)(256 * q1 + q0));
            }
            if (live && pr.out) {
                const float low = lr[0][i] + (lr[1][i] + lr[2][i]);
                float y;
                if constexpr (PL == 1) y = fmaf(__fmul_rn(w.mu[h], sc), qsf, __fmul_rn(__fmul_rn(w.al[h], sc), accf) + low);
                else y = fmaf(w.mu[h], __fmul_rn(qsf, sc), __fmul_rn(w.al[h], __fmul_rn(accf, sc)) + low);      // (sc: a power of two, may be subnormal)
                pr.out[(int64_t)t * pr.ldo + n] = __float2bfloat16_rn(y);
            }
        }
    };
    const uint32_t b0 = smem_u32(smem) + (uint32_t)((tq * TOK + gq) * 128), b_swz = (uint32_t)((gq ^ (tq << 1)) << 4);
#pragma unroll 1
    while (g < g_hi) {
        int32_t acc[SETS][2][NT][4];
        int sub = it < it_end ? it / un : 0, u = it - sub * un;
        auto clear = [&]() {
#pragma unroll
            for (int s = 0; s < SETS; ++s)
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[s][mt][nt][e] = 0;
        };
        clear();
#pragma unroll 1
        for (; it < it_end; ++it) {
            uint4 w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = wn[j];
            if (it + 1 < it_end) load_w(wn, it + 1);
            // column tile j of the item: plane j / NTP, token tile j % NTP
            const uint32_t b_item = b0 + (uint32_t)(u * kSteps * TOK * 128);
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                uint32_t a[2][4][4];
#pragma unroll
                for (int mt = 0; mt < 2; ++mt) {
                    const uint4 lo4 = w[2 * mt], hi4 = w[2 * mt + 1];
                    const uint32_t lo = x == 0 ? lo4.x : x == 1 ? lo4.y : x == 2 ? lo4.z : lo4.w;
                    const uint32_t hi = x == 0 ? hi4.x : x == 1 ? hi4.y : x == 2 ? hi4.z : hi4.w;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int sh = q & ~(SETS - 1);
                        const uint32_t m = 0x01010101u << (q & (SETS - 1));
                        a[mt][q][0] = (lo >> sh) & m; a[mt][q][1] = (hi >> sh) & m;
                        a[mt][q][2] = (lo >> (sh + 4)) & m; a[mt][q][3] = (hi >> (sh + 4)) & m;
                    }
                }
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const uint32_t at = b_item + (uint32_t)(8 * nt * 128);
                    const uint4 c0 = lds128(at + ((uint32_t)(32 * x) ^ b_swz)), c1 = lds128(at + ((uint32_t)(32 * x + 16) ^ b_swz));
                    const uint32_t bl[4] = {c0.x, c0.y, c0.z, c0.w}, bh[4] = {c1.x, c1.y, c1.z, c1.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
#pragma unroll
                        for (int mt = 0; mt < 2; ++mt)
                            imma_16832(acc[q & (SETS - 1)][mt][nt], a[mt][q][0], a[mt][q][1], a[mt][q][2], a[mt][q][3], bl[q], bh[q]);
                }
            }
            if (++u == un || it + 1 == it_end) {
                // the group (or the warp's share of it) is done: into the CTA's sums
                const uint32_t at = smem_u32(accs) + (uint32_t)((sub * 2 * NT * 128 + lane) * 4);
#pragma unroll
                for (int mt = 0; mt < 2; ++mt)
#pragma unroll
                    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            int32_t v = acc[0][mt][nt][e];
#pragma unroll
                            for (int z = 1; z < SETS; ++z) v += acc[z][mt][nt][e] >> z;
                            red_shared_add(at + (uint32_t)(((mt * NT + nt) * 4 + e) * 128), v);
                        }
                clear();
                u = 0; ++sub;
            }
        }
        // the next run's first sign words, and what the first fragment of this one needs, are on their way while the warps meet
        const int g_now = g, n_now = n, frags = n_now * 2 * NTP, f_step = (SPLIT ? p.S : 1) * kWarps;
        int f = SPLIT ? rank * kWarps + warp : warp;
        Rows rows;
        if (AHEAD && f < frags) fetch_rows(rows, g_now + f / (2 * NTP), f / NTP & 1);
        g += n; n = min(p.run, g_hi - g);
        if (g < g_hi) {
            share();
            if (it < it_end) load_w(wn, it);
        }
        if (SPLIT) { cluster_arrive_release(); cluster_wait_acquire(); }
        else __syncthreads();
        // ---- epilogue: the fragments of the run, dealt to the warps (of the whole cluster)
#pragma unroll 1
        for (; f < frags && !failed; f += f_step) {
            const int grp = f / (2 * NTP), mt = f / NTP & 1, nt = f % NTP;
            if (!AHEAD) fetch_rows(rows, g_now + grp, mt);
            const Rows now = rows;
            if (AHEAD && f + f_step < frags) fetch_rows(rows, g_now + (f + f_step) / (2 * NTP), (f + f_step) / NTP & 1);
            int32_t v[PL][4];
#pragma unroll
            for (int pl = 0; pl < PL; ++pl) {
                int32_t* at = accs + ((grp * 2 + mt) * NT + pl * NTP + nt) * 128 + lane;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (!SPLIT) {
                        v[pl][e] = at[32 * e];
                        at[32 * e] = 0;
                    } else {
                        const uint32_t a = smem_u32(at + 32 * e);
                        int32_t q[8];
#pragma unroll
                        for (int s = 0; s < 8; ++s)
                            if (s < p.S) q[s] = ld_cluster_s32(map_shared_rank(a, (uint32_t)s));
                        v[pl][e] = 0;
#pragma unroll
                        for (int s = 0; s < 8; ++s)
                            if (s < p.S) v[pl][e] += q[s];
                    }
                }
            }
            epilogue(now, g_now + grp, mt, nt, v);
        }
        if (SPLIT) {
            cluster_arrive_release(); cluster_wait_acquire();       // everybody has read
            if (g < g_hi) {
                for (int i = tid; i < n_now * 2 * NT * 32; i += kThreads) reinterpret_cast<uint4*>(accs)[i] = make_uint4(0u, 0u, 0u, 0u);
                __syncthreads();
            }
        } else if (g < g_hi) {
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
struct SmallPlan { int S, run, t_off, tok_off, acc_off, smem; int clusters[kRotMaxProblems]; };

static int token_tiles(int64_t M) { return M <= 8 ? 1 : 2; }

// How many clusters of S such CTAs the device holds at once.  (Clusters are placed inside a GPC, so this is less than SMs / S:
// asked once per size and thread.)
static int resident_small_clusters(int S) {
    static thread_local int known[9], known_dev = -1;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    if (known_dev != dev) { for (int& k : known) k = -1; known_dev = dev; }
    if (known[S] < 0) {
        auto kernel = gemm_small_kernel<2, 1, true>;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(S * sm_count()), 1, 1);
        cfg.blockDim = dim3(small_::kThreads, 1, 1);
        cfg.dynamicSmemBytes = small_::kSmemMax;
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = (unsigned)S; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a; cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, small_::kSmemMax) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
        known[S] = n;
    }
    return known[S];
}

// Picks S by an estimate of cycles: the items of the longest run chain at the measured rate of the loop (32 and 52 cycles per
// 128 k, row group and scheduler-quarter at 8 and 16 tokens), a round of barriers and epilogue per run, filling the CTA's codes from
// the L2, and the cluster's barriers.
static bool small_plan_search(int NTP, int PL, int units, const int64_t* N, int n, bool lowrank, int sms, int spare, int room, SmallPlan* best) {
    using namespace small_;
    const int NT = NTP * PL, tok = 8 * NT;
    double best_cost = 0.0;
    bool found = false;
    for (int S = 1; S <= 8 && S <= units; ++S) {
        const int per_cta = (units + S - 1) / S;
        SmallPlan pl{};
        pl.S = S;
        int off = per_cta * kSteps * tok * 128;
        pl.t_off = off; off += lowrank ? 3 * 8 * NTP * 128 : 0;
        pl.tok_off = off; off += (12 * tok + 15) / 16 * 16;
        pl.acc_off = off;
        const int group_bytes = 2 * NT * 512;
        const int fit = (kSmemMax - off) / group_bytes;
        if (fit < 1) continue;
        const int total = std::min((sms - spare) / S, S == 1 ? sms : resident_small_clusters(S) - room);      // clusters the device holds
        if (total < n) break;
        int groups[kRotMaxProblems], used = 0, longest = 1;
        int64_t all = 0;
        for (int i = 0; i < n; ++i) { groups[i] = (int)((N[i] + 31) / 32); all += groups[i]; }
        // clusters per problem, by row groups: at least one each, never more than groups
        for (int i = 0; i < n; ++i) {
            pl.clusters[i] = (int)std::max<int64_t>(1, std::min<int64_t>(groups[i], (int64_t)total * groups[i] / all));
            used += pl.clusters[i];
        }
        while (used > total) {                                    // (only through the minimum of one each)
            int big = 0;
            for (int i = 1; i < n; ++i) if (pl.clusters[i] > pl.clusters[big]) big = i;
            --pl.clusters[big]; --used;
        }
        auto chain = [&](int i) { return (groups[i] + pl.clusters[i] - 1) / pl.clusters[i]; };
        while (used < total) {                                    // what is left goes to whoever has the longest chain
            int worst = 0;
            for (int i = 1; i < n; ++i) if (chain(i) > chain(worst)) worst = i;
            if (chain(worst) == 1) break;
            ++pl.clusters[worst]; ++used;
        }
        for (int i = 0; i < n; ++i) longest = std::max(longest, chain(i));
        pl.run = std::min(longest, fit);
        pl.smem = off + pl.run * group_bytes;
        const double step = NT == 1 ? 30.0 : 22.0 * NT + 8.0;     // cycles per SM and code row of an item
        const int runs = (longest + pl.run - 1) / pl.run;
        auto items = [&](int g) { return (double)((g * per_cta + kWarps - 1) / kWarps) * kWarps; };
        const double cost = (runs - 1) * items(pl.run) * kSteps * step + items(longest - (runs - 1) * pl.run) * kSteps * step +
                            runs * (1500.0 + 60.0 * NT * pl.run / S) + per_cta * kSteps * tok * 128 / 40.0 + (S > 1 ? 1500.0 + 1000.0 * runs : 0.0);
        if (!found || cost < best_cost) { best_cost = cost; *best = pl; found = true; }
    }
    return found;
}

// The plans of the shapes a thread has called lately: a decode loop asks for the same few on every step.
static bool small_plan(const GemmArgs* a, int n, int planes, SmallPlan* out) {
    using namespace small_;
    struct Key { int dev, NTP, PL, units, n, lowrank, spare, room; int64_t N[kRotMaxProblems]; };
    struct Known { Key k; bool ok; SmallPlan plan; };
    static thread_local Known known[16];
    static thread_local int used = 0;
    const int64_t M = a[0].M, K = a[0].K;
    if (n < 1 || n > kRotMaxProblems || M < 1 || M > (planes == 3 ? kSmallDigitTokens : kSmallTokens) || K % 128 != 0 || (planes == 3 && K > 25600)) return false;
    Key k{};
    for (int i = 0; i < n; ++i) {
        if (a[i].N < 1 || a[i].N > ((int64_t)1 << 30) || a[i].r > kLowrankPad || M * a[i].N >= (int64_t)1 << 31) return false;
        k.N[i] = a[i].N;
        if (a[i].r > 0) k.lowrank = 1;
    }
    if (cudaGetDevice(&k.dev) != cudaSuccess) { cudaGetLastError(); return false; }
    k.NTP = token_tiles(M); k.PL = planes; k.units = (int)((K + kUnit - 1) / kUnit); k.n = n;
    // With very few tokens the rotation kernels before and after have a handful of CTAs: a few SMs are left to them, so that this
    // kernel starts whole while the one before still runs, and the next one's constants arrive under this one.
    k.spare = M <= 2 ? 8 : 0;
    // Clusters of this kernel that a rotation in clusters leaves no room would start, and fetch their constants, when it has ended: two are left out
    // (one token, 160 x 160 to 1024 and 12288 outputs, raw: 26.5 -> 19.0 us, 42.1 -> 32.2; 108 x 128 to 5120: 23.5 -> 21.5; a rotation in single CTAs needs
    // none, 86 x 128 to 5120: 20.3 us, 21.3 with two left out).
    k.room = k.spare > 0 && planes == 1 && a[0].rot_cluster > 1 ? 2 : 0;
    auto same = [&](const Key& o) {
        return o.dev == k.dev && o.NTP == k.NTP && o.PL == k.PL && o.units == k.units && o.n == k.n && o.lowrank == k.lowrank && o.spare == k.spare && o.room == k.room &&
               std::equal(k.N, k.N + kRotMaxProblems, o.N);
    };
    for (int i = 0; i < 16 && i < used; ++i)
        if (same(known[i].k)) { *out = known[i].plan; return known[i].ok; }
    const int sms = sm_count();
    Known& slot = known[used % 16];
    slot.k = k;
    slot.ok = sms > 0 && small_plan_search(k.NTP, k.PL, k.units, k.N, n, k.lowrank != 0, sms, k.spare, k.room, &slot.plan);
    ++used;
    *out = slot.plan;
    return slot.ok;
}

bool gemm_small_fits(const GemmArgs* a, int n, int planes) {
    SmallPlan pl;
    return small_plan(a, n, planes, &pl) && (planes == 1 || pl.S == 1);
}

int gemm_small_blocks(const GemmArgs& a) {
    SmallPlan pl;
    return small_plan(&a, 1, 1, &pl) ? pl.clusters[0] * pl.S : 0;
}

template <int NTP, int PL, bool SPLIT>
static int launch_small_t(const SmallParams& p, int grid, int smem, cudaStream_t stream) {
    auto kernel = gemm_small_kernel<NTP, PL, SPLIT>;
    static thread_local int configured = -1;
    int dev = 0;
    BWLA_CUDA_TRY(cudaGetDevice(&dev));
    if (configured != dev) {
        BWLA_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, small_::kSmemMax));
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
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, p);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}
template <int NTP, int PL>
static int launch_small_nt(const SmallParams& p, int grid, int smem, cudaStream_t stream) {
    return p.S > 1 ? launch_small_t<NTP, PL, true>(p, grid, smem, stream) : launch_small_t<NTP, PL, false>(p, grid, smem, stream);
}

// All problems have the same M, K and bits; a[i].codes: int8 [planes][M][K] in the interleaved order; a[i].Thl: bf16 [3][M][64].
// *taken is false where the shapes do not fit (nothing has been launched then).
int launch_gemm_small(const GemmArgs* a, int n, int planes, bool* taken, cudaStream_t stream) {
    SmallPlan pl;
    *taken = small_plan(a, n, planes, &pl) && (planes == 1 || pl.S == 1);
    if (!*taken) return BWLA_OK;
    const int M = (int)a[0].M, K = (int)a[0].K, NTP = token_tiles(M);
    SmallParams p{};
    p.n_problems = n; p.M = M; p.K = K; p.units = (K + small_::kUnit - 1) / small_::kUnit; p.S = pl.S; p.run = pl.run;
    p.t_off = pl.t_off; p.tok_off = pl.tok_off; p.acc_off = pl.acc_off;
    p.status = a[0].status;
    int begin = 0;
    for (int i = 0; i < n; ++i) {
        SmallProblem& q = p.prob[i];
        q.packed = a[i].packed; q.codes = a[i].codes; q.scales = a[i].scales; q.qsum = a[i].qsum; q.zp = a[i].zp; q.rowsum = a[i].rowsum;
        q.alpha = a[i].alpha; q.mu = a[i].mu; q.U = (const __nv_bfloat16*)a[i].U; q.Thl = (const __nv_bfloat16*)a[i].Thl;
        q.out = (__nv_bfloat16*)a[i].out; q.ldo = a[i].ldo; q.acc_debug = a[i].acc_debug;
        q.N = (int)a[i].N; q.r = a[i].r; q.groups = ((int)a[i].N + 31) / 32; q.cluster_begin = begin; q.clusters = pl.clusters[i];
        begin += pl.clusters[i];
    }
    const int grid = begin * pl.S;
    if (planes == 3) return launch_small_t<1, 3, false>(p, grid, pl.smem, stream);
    return NTP == 1 ? launch_small_nt<1, 1>(p, grid, pl.smem, stream) : launch_small_nt<2, 1>(p, grid, pl.smem, stream);
}

}  // namespace bwla
