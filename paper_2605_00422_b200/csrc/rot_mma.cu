// Online OKT (Sec. 3.1) on the warp-level tensor-core path, with what follows it fused in: the per-token quantiser
// (Sec. 4.1), the bf16 rounding of the weight-only operating point, or the final binarisation of weight rows (Alg. 2).
//
//   X = reshape(x_t, n1 x n2) (row-major),   Z^T = P2^T X^T  [d][a],   Y^T = Z^T P1  [d][c]
//
// Both contractions deliver fp32 accuracy from 16-bit MMAs (m16n8k16, fp32 accumulators).  First: x is bf16 already, P2 is
// the sum of three bf16 terms (all 24 bits): three products.  Second: Z and P1 are sums of two fp16 terms (22 bits), scaled by
// powers of two so that no term meets the ends of fp16's exponent range (P1 to a largest magnitude in [2^13, 2^14), Z by the
// bound |Z| <= n2 max|P2| max|x|): three products (hi hi, hi lo, lo hi) where bf16 terms need six.  The scales leave exactly,
// with one multiplication, before the quantiser.  The tensor core truncates when it adds to its accumulator, a bias that
// grows with every step: every 32 values of the contraction start from zero (small products first) and are added to the
// running sum with ordinary rounded additions.  (With in-core accumulation over the whole depth the error was 9.7e-7 of a
// token's full scale at 160 x 160.)
//
// Work split.  A warp owns 16 rows d: Z^T of its rows only needs its rows of P2^T, and Y^T of its rows only needs its rows of
// Z^T, so nothing but x, the largest |x| and the absmax of Y is shared between warps, and the accumulators of the first
// contraction are the A operand of the second as they stand (more than 64 columns are dealt to 2 or 4 warps, which exchange
// their parts of Z^T through shared memory).  The warps of a token are a group with a barrier of its own; where shared memory
// allows, several groups of a CTA work on tokens of their own and share the constants, so that one group's barriers and
// stores run under another's MMAs.  A token whose warps or operands do not fit one CTA is spread over a cluster of up to
// eight, which share the two maxima through distributed shared memory.  CTAs stay on their SMs and take tokens in turn;
// the next token's x is fetched (cp.async) under the second contraction of this one.
//
// The blocks beside the rotation CTAs evaluate T = V x for the PSP low-rank branch (prologue_roles.cuh).
//
// Launched with programmatic stream serialisation: the layer's constants are fetched before the preceding kernel of the
// stream has finished; x is read, and everything is stored, after it.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "bwla_common.cuh"
#include "prologue_roles.cuh"
#include "rot_mma.cuh"

namespace bwla {

enum { kRotQuant = 0, kRotBf16 = 1, kRotBinarize = 2, kRotDigits = 3 };

// What the warps and CTAs of a token exchange: one per group, behind its operand tiles.  [token parity][warp of the token]
struct RotShared {
    uint32_t xmax[2][64];                 // bits of the largest |x|
    float amax[2][64], vmin[2][64];       // largest |Y| (asymmetric quantiser: largest and smallest Y)
    double wsum[kRotMaxWarps];
    double slot_sum[2][8];
    int qsum[2][3];
};
static_assert(sizeof(RotShared) <= kRotRedBytes, "RotShared");

// once per layer: P1, P2 (fp32) -> exponents (of max|P2|; by which P1 is scaled), the bf16 terms of P2^T and the fp16 terms of
// P1^T, rows as they lie in shared memory
__global__ void __launch_bounds__(256) prepare_rot_kernel(RotGeom g, const float* __restrict__ P1, const float* __restrict__ P2,
                                                         uint8_t* __restrict__ prepared) {
    __shared__ uint32_t red[8];
    const int e2 = exponent_of(block_absmax(P2, g.n2 * g.n2, red)), e1 = factor_exponent(block_absmax(P1, g.n1 * g.n1, red));
    if (blockIdx.x == 0 && threadIdx.x == 0) { reinterpret_cast<int*>(prepared)[0] = e2; reinterpret_cast<int*>(prepared)[1] = e1; }
    const int rows2 = g.n2p, rows1 = g.na * 8;
    uint8_t* t2 = prepared + kRotHeader;
    uint8_t* t1 = t2 + (size_t)3 * rows2 * g.s2;
    const int tid = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    split_factor<false>(P2, g.n2, 0, rows2, g.n2p, 1.f, [&](int r, int k2) { return t2 + (size_t)r * g.s2 + 4 * k2; }, (size_t)rows2 * g.s2, tid, nt);
    split_factor<true>(P1, g.n1, 0, rows1, rows1, pow2f(e1), [&](int r, int k2) { return t1 + (size_t)r * g.s1 + 4 * k2; }, (size_t)rows1 * g.s1, tid, nt);
}

int launch_prepare_rot(const RotGeom& g, const float* P1, const float* P2, void* prepared, cudaStream_t stream) {
    ProfScope prof(kProfPrepare, stream);
    prepare_rot_kernel<<<32, 256, 0, stream>>>(g, P1, P2, (uint8_t*)prepared);
    return after_launch();
}

// ---------------------------------------------------------------------------------------------
// per call
// ---------------------------------------------------------------------------------------------
struct RotKernelParams {
    RotGeom g;
    int groups;                     // groups of warps per CTA, each with a token of its own
    const void* x; int64_t ldx;     // bf16, or fp32 where the kernel is instantiated for fp32 rows
    int x_vec;                      // rows can be read in 16-byte pieces
    int64_t M;
    int bits, asym;
    int n_problems;
    int clusters_per_problem;       // group i of a problem (counted over its clusters) takes tokens i, i + all groups, ...
    int rot_first, rot_ctas;        // rotation CTAs are blocks [rot_first, rot_first + rot_ctas)
    RotProblem prob[kRotMaxProblems];
    uint32_t* status;
    // low-rank blocks: problem i owns blocks [lr_begin[i], lr_begin[i + 1]) counted among the non-rotation blocks
    int lr_begin[kRotMaxProblems + 1];
    PrologueParams lr[kRotMaxProblems];
};

// NTW: 8-column tiles of a (first contraction) and of c (second) one warp owns, at most.  EXCH: the columns are dealt to
// several warps, which exchange Z^T through shared memory.  F32: x is fp32 (three bf16 terms, taken one after the other
// through the same shared memory).
template <int NTW, bool EXCH, int MODE, bool F32>
__global__ void __launch_bounds__(32 * kRotMaxWarps, 1) rot_mma_kernel(const __grid_constant__ RotKernelParams p) {
    extern __shared__ __align__(16) uint8_t smem[];
    const int b = (int)blockIdx.x;
    if (MODE != kRotBinarize && (b < p.rot_first || b >= p.rot_first + p.rot_ctas)) {
        // ---------------- T = V x blocks ----------------
        const int lb = b < p.rot_first ? b : b - p.rot_ctas;
        int i = 0;
        while (i + 1 < p.n_problems && lb >= p.lr_begin[i + 1]) ++i;
        if (lb >= p.lr_begin[p.n_problems]) return;
        lowrank_block(p.lr[i], lb - p.lr_begin[i], reinterpret_cast<float*>(smem));
        return;
    }
    const RotGeom& g = p.g;
    const int lane = threadIdx.x & 31;
    const int rank = g.dc > 1 ? (int)cluster_ctarank() : 0;
    const int cl = (b - p.rot_first) / g.dc;
    const int prob_i = cl / p.clusters_per_problem;
    if (prob_i >= p.n_problems) return;               // (padding CTAs of the grid: whole clusters)
    const RotProblem& pr = p.prob[prob_i];
    // the group of warps this thread works in
    const int W = g.warps, T = 32 * W;
    const int group = (int)(threadIdx.x >> 5) / W, warp = (int)(threadIdx.x >> 5) - group * W, tid = 32 * warp + lane;
    const int64_t stride = (int64_t)p.clusters_per_problem * p.groups;
    const int64_t tok0 = (int64_t)(cl - prob_i * p.clusters_per_problem) * p.groups + group;
    uint8_t* const gs = smem + g.group_off + group * g.group_bytes;
    RotShared& sh = *reinterpret_cast<RotShared*>(gs + g.red_rel);
    auto barrier = [&]() { named_barrier(1 + group, T); };

    const int rows2 = g.dtc * 16, rows1 = g.na * 8;
    const int part2 = rows2 * g.s2, part1 = rows1 * g.s1;             // one term of this CTA's rows of P2^T; of P1^T
    uint8_t* const p2s = smem;
    uint8_t* const p1s = smem + g.p1_off;
    uint8_t* const xs = gs;
    uint8_t* const zs = gs + g.z_rel;

    // ---- the layer's constants (they do not depend on the preceding kernel, except that the factors of a binarisation may be what it has
    //      made), and the zeros around x ----
    if (MODE == kRotBinarize) griddep_wait();
    int e2, e1;
    if (pr.prepared) {
        const uint8_t* t2 = pr.prepared + kRotHeader + (size_t)rank * part2;
        const size_t all2 = (size_t)g.n2p * g.s2;                     // (the last CTA of a cluster may have fewer rows)
        const int own2 = min(part2, (g.n2p - rank * rows2) * g.s2);
        const uint8_t* t1 = pr.prepared + kRotHeader + 3 * all2;
        for (int i = 16 * threadIdx.x; i < own2; i += 16 * blockDim.x) {
            cp_async16(smem_u32(p2s + i), t2 + i);
            cp_async16(smem_u32(p2s + part2 + i), t2 + all2 + i);
            cp_async16(smem_u32(p2s + 2 * part2 + i), t2 + 2 * all2 + i);
        }
        for (int i = 16 * threadIdx.x; i < 2 * part1; i += 16 * blockDim.x) cp_async16(smem_u32(p1s + i), t1 + i);
        e2 = __ldg(reinterpret_cast<const int*>(pr.prepared));
        e1 = __ldg(reinterpret_cast<const int*>(pr.prepared) + 1);
    } else {
        uint32_t* const red = reinterpret_cast<RotShared*>(smem + g.group_off + g.red_rel)->xmax[0];
        e2 = exponent_of(block_absmax(pr.P2, g.n2 * g.n2, red));
        e1 = factor_exponent(block_absmax(pr.P1, g.n1 * g.n1, red));
        __syncthreads();                              // (the words of `red` are cleared below)
        split_factor<false>(pr.P2, g.n2, rank * rows2, rows2, g.n2p, 1.f, [&](int r, int k2) { return p2s + r * g.s2 + 4 * k2; }, part2, threadIdx.x, blockDim.x);
        split_factor<true>(pr.P1, g.n1, 0, rows1, rows1, pow2f(e1), [&](int r, int k2) { return p1s + r * g.s1 + 4 * k2; }, part1, threadIdx.x, blockDim.x);
    }
    const int cpr = g.n2 >> 3, chunks = g.n1 * cpr;   // 16-byte chunks (of bf16) per row of X, and in all
    auto zero_padding = [&]() {                       // what the contractions read of X beyond n1 x n2
        const int per = g.s2 >> 4;                    // (rows beyond n1 become columns of Z^T that EXCH drops)
        for (int i = tid; !EXCH && i < (rows1 - g.n1) * per; i += T) *reinterpret_cast<uint4*>(xs + g.n1 * g.s2 + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
        if (g.n2p != g.n2)
            for (int i = tid; i < g.n1; i += T) *reinterpret_cast<uint4*>(xs + i * g.s2 + 16 * cpr) = make_uint4(0u, 0u, 0u, 0u);
    };
    // x may be what the preceding kernel is writing, so it is read only behind the wait below; but its lines can be asked into the
    // L2, where those writes go anyway: address translation and, where x is older, the trip to HBM are over by then
    if (tok0 < p.M) {
        const uint8_t* xt = reinterpret_cast<const uint8_t*>(p.x) + tok0 * p.ldx * (F32 ? 4 : 2);
        for (int i = 128 * tid; i < g.K * (F32 ? 4 : 2); i += 128 * T) prefetch_l2_line(xt + i);
    }
    zero_padding();
    for (int i = tid; i < (int)(sizeof(RotShared) / 4); i += T) reinterpret_cast<uint32_t*>(&sh)[i] = 0u;
    __syncthreads();
    if (g.dc > 1) { cluster_arrive_release(); cluster_wait_acquire(); }   // every CTA of the cluster runs: its slots may be written
    // (The signs, scales and shifts of a binarisation are constants of the calls behind it, which read constants before they wait: they
    // start when this kernel has ended.)
    if (MODE != kRotBinarize) griddep_launch_dependents();
    int ntok = tok0 < p.M ? (int)((p.M - tok0 + stride - 1) / stride) : 0;
    // this thread's chunks of X: tid, tid + T, ...; (row, column) advance without divisions
    const int ch_a0 = tid / cpr, ch_c0 = tid - ch_a0 * cpr, ch_da = T / cpr, ch_dc = T - ch_da * cpr;
    auto for_chunks = [&](auto&& f) {
        int c = ch_c0;
        uint8_t* at = xs + ch_a0 * g.s2 + 16 * ch_c0;
        const int step = ch_da * g.s2 + 16 * ch_dc, wrap = g.s2 - 16 * cpr;
#pragma unroll 1
        for (int i = tid; i < chunks; i += T) {
            f(i, at);
            at += step; c += ch_dc;
            if (c >= cpr) { c -= cpr; at += wrap; }
        }
    };
    auto fetch_x = [&](int64_t t) {                   // bf16 rows go to shared memory as they are
        const uint16_t* xt = reinterpret_cast<const uint16_t*>(p.x) + t * p.ldx;
        if (p.x_vec) {
            for_chunks([&](int i, uint8_t* dst) { cp_async16(smem_u32(dst), xt + 8 * i); });
        } else {
            for_chunks([&](int i, uint8_t* dst) {
                for (int j = 0; j < 8; ++j) reinterpret_cast<uint16_t*>(dst)[j] = xt[8 * i + j];
            });
        }
    };
    auto load_f32 = [&](const float* src, float (&v)[8]) {
        if (p.x_vec) {
            const float4 lo = __ldg(reinterpret_cast<const float4*>(src)), hi = __ldg(reinterpret_cast<const float4*>(src) + 1);
            v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w; v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = __ldg(src + j);
        }
    };
    // term `which` of fp32 row t, in place of x; returns this thread's largest |x| (bits)
    auto put_term = [&](int64_t t, int which) -> uint32_t {
        const float* xf = reinterpret_cast<const float*>(p.x) + t * p.ldx;
        uint32_t m = 0u;
        for_chunks([&](int i, uint8_t* at) {
            float v[8];
            load_f32(xf + 8 * i, v);
            uint32_t w[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                m = max(m, max(__float_as_uint(v[2 * j]) & 0x7FFFFFFFu, __float_as_uint(v[2 * j + 1]) & 0x7FFFFFFFu));
                uint32_t h, mid, l;
                split3_pair(v[2 * j], v[2 * j + 1], h, mid, l);
                w[j] = which == 0 ? h : which == 1 ? mid : l;
            }
            *reinterpret_cast<uint4*>(at) = make_uint4(w[0], w[1], w[2], w[3]);
        });
        return m;
    };
    // largest |x| of the chunks this thread has fetched (every CTA of the cluster has all of x and looks at its share)
    auto own_max = [&]() -> uint32_t {
        uint32_t m = 0u, part = 0u;
        for_chunks([&](int, uint8_t* src) {
            if (part == (uint32_t)rank) {
                const uint4 v = *reinterpret_cast<const uint4*>(src);
                m = __vmaxu2(m, __vmaxu2(__vmaxu2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu), __vmaxu2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu)));
            }
            if (++part == (uint32_t)g.dc) part = 0u;
        });
        return max(m & 0xFFFFu, m >> 16) << 16;
    };
    // a warp's word into the slot of this warp in every CTA of the cluster; the token barrier (CTAs' or cluster's) follows
    auto publish = [&](void* slots, uint32_t v) {
        uint32_t* s = reinterpret_cast<uint32_t*>(slots) + rank * W + warp;
        if (g.dc == 1) { if (lane == 0) *s = v; }
        else if (lane < g.dc) st_shared_cluster_u32(map_shared_rank(smem_u32(s), (uint32_t)lane), v);
    };
    auto token_barrier = [&]() {
        if (g.dc == 1) barrier();
        else { cluster_arrive_release(); cluster_wait_acquire(); }
    };
    auto slots_max = [&](const void* slots) -> uint32_t {             // (the words are bits of non-negative values)
        const volatile uint32_t* s = reinterpret_cast<const volatile uint32_t*>(slots);
        return __reduce_max_sync(0xFFFFFFFFu, max(s[lane], s[lane + 32]));
    };

    const int dtl = EXCH ? warp / g.cw : warp, cw = EXCH ? warp - dtl * g.cw : 0;
    const int nt0 = cw * NTW;                                         // this warp's first column tile
    const int gq = lane >> 2, tq = lane & 3;                          // accumulator rows gq, gq + 8; columns 2 tq, 2 tq + 1
    const int d0 = (rank * g.dtc + dtl) * 16;
    const bool row_hi_ok = d0 + 8 < g.n2, row_lo_ok = d0 < g.n2;      // (a warp may have no rows at all)
    const uint32_t a_off = (uint32_t)(lane & 15), a_col = (uint32_t)(lane >> 4) * 16u;
    const uint32_t b_row = (uint32_t)(((lane >> 4) << 3) + (lane & 7)), b_col = (uint32_t)((lane >> 3) & 1) * 16u;
    const uint32_t a2_addr = smem_u32(p2s) + (uint32_t)(dtl * 16 + a_off) * g.s2 + a_col;
    const uint32_t bx_addr = smem_u32(xs) + (uint32_t)(nt0 * 8 + b_row) * g.s2 + b_col;
    const uint32_t b1_addr = smem_u32(p1s) + (uint32_t)(nt0 * 8 + b_row) * g.s1 + b_col;
    const uint32_t az_addr = smem_u32(zs) + (uint32_t)(dtl * 16 + a_off) * g.s1 + a_col, az_lo = (uint32_t)(rows2 * g.s1);
    const int ksteps2 = g.n2p >> 4, ksteps1 = g.na >> 1;
    const int qmax = (1 << (p.bits - 1)) - 1;
    const bool asym = p.asym != 0;
    // Where this lane's codes go, for its two columns (parity e) of tile 0 and row gq; a tile further is 8 n2 further, which
    // is a multiple of 64.  Interleaved layout: inside each group of 32, byte 4 (k % 8) + (k % 32) / 8; with n2 a multiple
    // of 16, rows gq and gq + 8 are neighbouring bytes.
    const bool interleave = (MODE == kRotQuant || MODE == kRotDigits) && pr.codes_layout != 0;
    const bool pairs16 = interleave && (g.n2 & 15) == 0 && row_hi_ok;
    const bool plain_codes = interleave && (g.n2 & 15) == 0 && row_hi_ok && (nt0 + NTW) * 8 <= g.n1 && !pr.y;
    int lim[2], off_lo[2], off_hi[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int c = nt0 * 8 + 2 * tq + e, k0 = c * g.n2 + d0, k1 = k0 + 8;
        lim[e] = row_lo_ok ? min(g.n1, (nt0 + NTW) * 8) - c : 0;            // tile j exists in this lane when 8 j < lim
        off_lo[e] = interleave ? (k0 & ~31) + 4 * gq + ((k0 & 31) >> 3) : k0 + gq;
        off_hi[e] = interleave ? (k1 & ~31) + 4 * gq + ((k1 & 31) >> 3) : k1 + gq;
    }

    // sum over the token's warps and CTAs, in a fixed order
    auto total_sum = [&](double v, int slot) -> double {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        barrier();                                    // the sums may still be read from the call before
        if (lane == 0) sh.wsum[warp] = v;
        barrier();
        double s = 0.0;
        for (int w = 0; w < W; ++w) s += sh.wsum[w];
        if (g.dc > 1) {
            if (tid < g.dc) {
                const uint32_t dst = map_shared_rank(smem_u32(&sh.slot_sum[slot][rank]), (uint32_t)tid);
                const uint64_t bits = (uint64_t)__double_as_longlong(s);
                st_shared_cluster_u32(dst, (uint32_t)bits);
                st_shared_cluster_u32(dst + 4, (uint32_t)(bits >> 32));
            }
            cluster_arrive_release(); cluster_wait_acquire();
            s = 0.0;
            for (int c = 0; c < g.dc; ++c) s += *reinterpret_cast<volatile double*>(&sh.slot_sum[slot][c]);
        }
        return s;
    };
    // acc += (one or two steps of 16 values of the contraction) A terms x B, in chains that start from zero with the smallest
    // products, two column tiles side by side.  `terms` lists (A term, B fragments) from small to large.
    // Up to 32 columns the splits are a large part of the error: chains are 16 values long, the second contraction's small products have one
    // of their own, with lo lo among them (32 x 32: 1.45e-7 -> 1.14e-7 of a row's 2-norm, six bf16 products 1.17e-7; one token 3.7 -> 3.8 us).
    constexpr bool FINE = !EXCH && NTW <= 4;
    float acc[NTW][4];
    auto clear = [&]() {
#pragma unroll
        for (int j = 0; j < NTW; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[j][i] = 0.f;
    };
    const float zero4[4] = {0.f, 0.f, 0.f, 0.f};
    auto load_b = [&](uint32_t (&f)[4], uint32_t at, bool both) {
        if (both) ldsm_x4(f, at);
        else ldsm_x2(f, at);
    };
    // acc += rows of P2^T (its TERMS largest terms) times what lies in x's place
    auto stage_a = [&](auto terms_) {
        constexpr int TERMS = decltype(terms_)::value;
        auto step = [&](int kk, auto two_) {
            constexpr int S = decltype(two_)::value ? 2 : 1;
            uint32_t fa[S][TERMS][4];
#pragma unroll
            for (int h = 0; h < S; ++h)
#pragma unroll
                for (int q = 0; q < TERMS; ++q) ldsm_x4(fa[h][q], a2_addr + q * part2 + 32 * (kk + h));
#pragma unroll
            for (int j = 0; j < NTW; j += 2) {
                uint32_t f[S][4];
#pragma unroll
                for (int h = 0; h < S; ++h) load_b(f[h], bx_addr + (uint32_t)(j * 8) * g.s2 + 32 * (kk + h), j + 1 < NTW);
                float t[2][4];
#pragma unroll
                for (int q = TERMS - 1; q >= 0; --q)
#pragma unroll
                    for (int h = 0; h < S; ++h)
#pragma unroll
                        for (int jj = 0; jj < (j + 1 < NTW ? 2 : 1); ++jj)
                            mma_16816<false>(t[jj], fa[h][q], f[h][2 * jj], f[h][2 * jj + 1], (q == TERMS - 1 && h == 0) ? zero4 : t[jj]);
                add4(acc[j], t[0]);
                if (j + 1 < NTW) add4(acc[j + 1 < NTW ? j + 1 : j], t[1]);
            }
        };
        int kk = 0;
        if constexpr (!FINE) {
#pragma unroll 1
            for (; kk + 1 < ksteps2; kk += 2) step(kk, std::true_type{});
        }
#pragma unroll 1
        for (; kk < ksteps2; ++kk) step(kk, std::false_type{});
    };
    // acc += (terms of Z^T, one or two steps of 16 values of a) times the terms of P1: lo hi, hi lo, hi hi
    auto stage_c = [&](int kk, auto two_, const uint32_t (*zh)[4], const uint32_t (*zl)[4]) {
        constexpr int S = decltype(two_)::value ? 2 : 1;
#pragma unroll
        for (int j = 0; j < NTW; j += 2) {
            uint32_t fh[S][4], fl[S][4];
#pragma unroll
            for (int h = 0; h < S; ++h) {
                const uint32_t at = b1_addr + (uint32_t)(j * 8) * g.s1 + 32 * (kk + h);
                load_b(fh[h], at, j + 1 < NTW);
                load_b(fl[h], at + part1, j + 1 < NTW);
            }
            float t[2][4];
            if constexpr (FINE) {
                float u[2][4];
#pragma unroll
                for (int jj = 0; jj < 2; ++jj) {
                    mma_16816<true>(u[jj], zl[0], fl[0][2 * jj], fl[0][2 * jj + 1], zero4);
                    mma_16816<true>(u[jj], zl[0], fh[0][2 * jj], fh[0][2 * jj + 1], u[jj]);
                    mma_16816<true>(u[jj], zh[0], fl[0][2 * jj], fl[0][2 * jj + 1], u[jj]);
                    mma_16816<true>(t[jj], zh[0], fh[0][2 * jj], fh[0][2 * jj + 1], zero4);
                    add4(t[jj], u[jj]);
                    add4(acc[j + jj], t[jj]);
                }
                continue;
            }
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int h = 0; h < S; ++h)
#pragma unroll
                    for (int jj = 0; jj < (j + 1 < NTW ? 2 : 1); ++jj)
                        mma_16816<true>(t[jj], q == 0 ? zl[h] : zh[h], q == 1 ? fl[h][2 * jj] : fh[h][2 * jj],
                                        q == 1 ? fl[h][2 * jj + 1] : fh[h][2 * jj + 1], (q == 0 && h == 0) ? zero4 : t[jj]);
            add4(acc[j], t[0]);
            if (j + 1 < NTW) add4(acc[j + 1 < NTW ? j + 1 : j], t[1]);
        }
    };
    // token `it`'s code sum leaves behind the first barrier of the token after it
    auto flush_qsum = [&](int64_t t, int par) {
        // every CTA of the cluster leaves its own part of the sum; the consumer adds the parts
        if ((MODE == kRotQuant || MODE == kRotDigits) && pr.qsum && tid < kQsumParts && (tid == rank || (rank == 0 && tid >= g.dc))) {
#pragma unroll
            for (int pl = 0; pl < (MODE == kRotDigits ? 3 : 1); ++pl) {
                pr.qsum[(pl * p.M + t) * kQsumParts + tid] = tid == rank ? sh.qsum[par][pl] : 0;
                if (tid == rank) sh.qsum[par][pl] = 0;
            }
        }
    };

    // (what the lanes need to know of their places is worked out by now, with the preceding kernel still running)
    uint32_t pin[6] = {a2_addr, bx_addr, b1_addr, az_addr, (uint32_t)off_lo[0], (uint32_t)off_hi[1]};
    asm volatile("" ::"r"(pin[0]), "r"(pin[1]), "r"(pin[2]), "r"(pin[3]), "r"(pin[4]), "r"(pin[5]), "r"(ntok), "r"(ch_a0), "r"(ch_da), "r"(lim[0]), "r"(lim[1]) : "memory");
    if (warp == 0 && tok0 < p.M) {
        if (lane == 0) touch(reinterpret_cast<const uint8_t*>(p.x) + tok0 * p.ldx * (F32 ? 4 : 2));
        if (lane == 1 && p.status) touch(p.status);
        if (lane == 2 && (MODE == kRotQuant || MODE == kRotDigits)) touch(pr.codes + tok0 * (int64_t)g.K);
        if (lane == 3 && MODE == kRotBf16) touch(pr.yhat + tok0 * (int64_t)g.K);
    }
    griddep_wait();                                   // x may be the output of the preceding kernel
    // (the look at the status word takes a trip to the L2: the first token's x is on its way by then)
    if (!F32 && ntok > 0) fetch_x(tok0);
    const int first_tokens = ntok;
    if (MODE == kRotBinarize) {
        if (b == 0 && threadIdx.x < kStatusBytes / 4) p.status[threadIdx.x] = 0u;     // this call clears its status words itself
    } else if (p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0) {
        ntok = 0;                                                                     // the call already failed
    }
    if (ntok < first_tokens) cp_async_wait_all();
    // Pass -1 only takes in the first token's x.
#pragma unroll 1
    for (int it = F32 ? 0 : -1; it < ntok; ++it) {
        const int par = it & 1;
        const int64_t t = tok0 + (int64_t)it * stride;
        const bool more = it + 1 < ntok, live = F32 || it >= 0;
        if (live) {
        // ---- Z^T of this warp's rows and columns
        clear();
        if (!F32) {
            if (row_lo_ok) stage_a(std::integral_constant<int, 3>{});
            barrier();                                // x is no longer needed
        } else {
            if (it > 0 && g.alias_z) zero_padding();
            publish(sh.xmax[par], __reduce_max_sync(0xFFFFFFFFu, put_term(t, 0)));
            token_barrier();
            if (row_lo_ok) stage_a(std::integral_constant<int, 3>{});
            barrier();
            put_term(t, 1);
            barrier();
            if (row_lo_ok) stage_a(std::integral_constant<int, 2>{});
            barrier();
            put_term(t, 2);
            barrier();
            if (row_lo_ok) stage_a(std::integral_constant<int, 1>{});
            barrier();
        }
        if (it > 0) flush_qsum(t - stride, par ^ 1);
        }
        const bool fetch_late = EXCH && g.alias_z;
        if (!F32 && more && live && !fetch_late) fetch_x(t + stride);
        // ---- the two fp16 terms of Z^T: accumulators of two column tiles are one A operand (16 values of a)
        const int ex = exponent_of(__uint_as_float(slots_max(sh.xmax[par])));
        const int z_exp = max(-126, min(126, 15 - (32 - __clz(g.n2 - 1)) - (e2 + 1) - (ex + 1)));
        const float z_scale = pow2f(z_exp);
        if (live) {
        uint32_t zh[(NTW + 1) / 2][4], zl[(NTW + 1) / 2][4];
#pragma unroll
        for (int j = 0; j < NTW; ++j) {
            mul2(acc[j][0], acc[j][1], z_scale);
            mul2(acc[j][2], acc[j][3], z_scale);
            uint32_t h0, l0, h1, l1;
            split2_pair(acc[j][0], acc[j][1], h0, l0);      // row gq
            split2_pair(acc[j][2], acc[j][3], h1, l1);      // row gq + 8
            if (!EXCH) {
                zh[j >> 1][2 * (j & 1)] = h0; zh[j >> 1][2 * (j & 1) + 1] = h1;
                zl[j >> 1][2 * (j & 1)] = l0; zl[j >> 1][2 * (j & 1) + 1] = l1;
            } else if (nt0 + j < g.na) {
                // (columns a >= n1 come from whatever lies behind x: they become zeros)
                const int a = (nt0 + j) * 8 + 2 * tq;
                const uint32_t keep = a + 1 < g.n1 ? 0xFFFFFFFFu : a < g.n1 ? 0xFFFFu : 0u;
                h0 &= keep; l0 &= keep; h1 &= keep; l1 &= keep;
                uint8_t* at = zs + (dtl * 16 + gq) * g.s1 + ((nt0 + j) * 8 + 2 * tq) * 2;
                *reinterpret_cast<uint32_t*>(at) = h0;
                *reinterpret_cast<uint32_t*>(at + 8 * g.s1) = h1;
                *reinterpret_cast<uint32_t*>(at + az_lo) = l0;
                *reinterpret_cast<uint32_t*>(at + az_lo + 8 * g.s1) = l1;
            }
        }
        if (EXCH) barrier();
        // ---- Y^T of this warp's rows and columns
        clear();
        if (row_lo_ok) {
            if (!EXCH) {
#pragma unroll
                for (int kk = 0; kk < NTW / 2; kk += FINE ? 1 : 2) {
                    if (!FINE && kk + 1 < NTW / 2) stage_c(kk, std::true_type{}, &zh[kk], &zl[kk]);
                    else stage_c(kk, std::false_type{}, &zh[kk], &zl[kk]);
                }
            } else {
                uint32_t fzh[2][4], fzl[2][4];
                int kk = 0;
#pragma unroll 1
                for (; kk + 1 < ksteps1; kk += 2) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) { ldsm_x4(fzh[h], az_addr + 32 * (kk + h)); ldsm_x4(fzl[h], az_addr + az_lo + 32 * (kk + h)); }
                    stage_c(kk, std::true_type{}, fzh, fzl);
                }
                if (kk < ksteps1) {
                    ldsm_x4(fzh[0], az_addr + 32 * kk); ldsm_x4(fzl[0], az_addr + az_lo + 32 * kk);
                    stage_c(kk, std::false_type{}, fzh, fzl);
                }
            }
        }
        if (EXCH && nt0 + NTW > g.na) {               // tiles beyond P1's rows hold anything
#pragma unroll
            for (int j = 0; j < NTW; ++j)
                if (nt0 + j >= g.na) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
        }
        if (fetch_late) {
            barrier();                                // Z^T is no longer needed: its place is x's again
            if (!F32 && more) { zero_padding(); fetch_x(t + stride); }
        }
        // ---- back to true scale (exact: powers of two), then what the caller wants of Y
        const int ey = -(z_exp + e1), ey1 = max(-126, min(127, ey)), ey2 = max(-126, min(127, ey - ey1));
        const float f1 = pow2f(ey1);
#pragma unroll
        for (int j = 0; j < NTW; ++j) { mul2(acc[j][0], acc[j][1], f1); mul2(acc[j][2], acc[j][3], f1); }
        if (ey2 != 0) {
            const float f2 = pow2f(ey2);
#pragma unroll
            for (int j = 0; j < NTW; ++j) { mul2(acc[j][0], acc[j][1], f2); mul2(acc[j][2], acc[j][3], f2); }
        }
        }
        float amax = 0.f, vmin = 0.f;                 // asymmetric: amax holds the largest value, zero included
        if (MODE == kRotQuant && live) {
            // Padding rows and columns are exact zeros, which changes neither reduction: the largest magnitude is at least zero
            // and the asymmetric range contains zero by definition.
            if (!asym) {
#pragma unroll
                for (int j = 0; j < NTW; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i) amax = fmaxf(amax, fabsf(acc[j][i]));
            } else {
#pragma unroll
                for (int j = 0; j < NTW; ++j)
#pragma unroll
                    for (int i = 0; i < 4; ++i) { amax = fmaxf(amax, acc[j][i]); vmin = fminf(vmin, acc[j][i]); }
            }
            // non-negative (NaNs aside), so their bit patterns order like the values
            publish(sh.amax[par], __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax)));
            if (asym) publish(sh.vmin[par], __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(fmaxf(-vmin, 0.f))));
        }
        if (MODE == kRotDigits && live) {
            // the values of the weight-only operating point are bf16; their largest magnitude as bits, NaNs included
            uint32_t top = 0u;
#pragma unroll
            for (int j = 0; j < NTW; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[j][i] = __bfloat162float(__float2bfloat16_rn(acc[j][i]));
                    top = max(top, __float_as_uint(acc[j][i]) & 0x7FFFFFFFu);
                }
            publish(sh.amax[par], __reduce_max_sync(0xFFFFFFFFu, top));
        }
        // the next token's x has had the second contraction to arrive (and so have the constants, before the first)
        if (!F32) {
            cp_async_wait_all();
            if (more) publish(sh.xmax[par ^ 1], __reduce_max_sync(0xFFFFFFFFu, own_max()));
            if (!live) __syncthreads();               // the constants are complete, for every group
            token_barrier();
            if (!live) continue;
        }
        if (MODE == kRotQuant) {
            amax = __uint_as_float(slots_max(sh.amax[par]));
            if (asym) vmin = -__uint_as_float(slots_max(sh.vmin[par]));
            // symmetric: codes in [-qmax, qmax] around zero.  Asymmetric (Sec. 4.1): u = rne(y * inv) + zero in [0, 2^b - 1]
            // with an integer zero point; what is stored is u - 2^(b-1) (+ the caller's bias), so that it fits int8.
            float inv = 0.f, scale = 1.f, zero_f = 0.f, half_f = 0.f, levels = 0.f;
            if (!asym) {
                if (amax != 0.f) { inv = __fdiv_rn((float)qmax, amax); scale = __fdiv_rn(amax, (float)qmax); }
            } else {
                levels = (float)((1 << p.bits) - 1);
                const float range = __fsub_rn(amax, vmin);
                if (range != 0.f) { inv = __fdiv_rn(levels, range); scale = __fdiv_rn(range, levels); }
                const float tz = __fmul_rn(-vmin, inv);
                zero_f = fminf(fmaxf(__fadd_rn(__fadd_rn(tz, 12582912.f), -12582912.f), 0.f), levels);
                half_f = (float)(1 << (p.bits - 1));
            }
            // With B = 1.5 * 2^23 + an even integer, fl(v + B) = B + rne(v) for |v| < 2^22: one addition rounds to nearest-even
            // and leaves the integer in the low mantissa bits.  Everything added to the rounded product (zero point, shift of
            // the stored code) goes into B except its parity bit, which is added to the bit pattern.  The stored byte is the
            // low byte of the pattern, and the patterns themselves are summed for the code sum: every one is 0x4B400000 + the
            // stored code.  Symmetric codes need no clamp (|y| * inv is at most qmax up to rounding, which rounds to qmax);
            // the rounding of an asymmetric zero point can push a code one step out of its range.
            const float store_shift = (float)pr.code_bias - half_f;
            const int shift_i = (int)(zero_f + store_shift);                 // small integer, exact
            const uint32_t odd = (uint32_t)(shift_i & 1);
            const float bias_even = 12582912.f + (float)(shift_i - (int)odd);
            const float lo_b = 12582912.f + store_shift - (float)odd, hi_b = lo_b + levels;
            uint32_t usum = 0u;
            int counted = 0;
            int8_t* ct = pr.codes + t * (int64_t)g.K;
            const int tile_step = 8 * g.n2;
            // (the product is rounded before the addition, as the definition says: packed multiplications were seen to be
            // contracted with the packed additions behind them, the scalar ones are not)
            auto code_words = [&](const float (&y)[4], uint32_t (&w)[4]) {
                float v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = __fmul_rn(y[i], inv);
                add2(v[0], v[1], bias_even, bias_even); add2(v[2], v[3], bias_even, bias_even);
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = __float_as_uint(v[i]);
            };
            auto clamp_words = [&](uint32_t (&w)[4]) {
#pragma unroll
                for (int i = 0; i < 4; ++i) w[i] = __float_as_uint(fminf(fmaxf(__uint_as_float(w[i]), lo_b), hi_b)) + odd;
            };
            if (plain_codes) {
                // the usual case: every row and column of the warp exists, codes in the contraction's order
                int8_t *c0 = ct + off_lo[0], *c1 = ct + off_lo[1];
                counted = 4 * NTW;
#pragma unroll
                for (int j = 0; j < NTW; ++j) {
                    uint32_t w[4];
                    code_words(acc[j], w);
                    if (asym) clamp_words(w);
                    usum += w[0] + w[1];
                    usum += w[2] + w[3];
                    *reinterpret_cast<uint16_t*>(c0) = (uint16_t)__byte_perm(w[0], w[2], 0x0040);
                    *reinterpret_cast<uint16_t*>(c1) = (uint16_t)__byte_perm(w[1], w[3], 0x0040);
                    c0 += tile_step; c1 += tile_step;
                }
            } else {
#pragma unroll
                for (int j = 0; j < NTW; ++j) {
                    uint32_t w[4];
                    code_words(acc[j], w);
                    if (asym) clamp_words(w);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        if (8 * j < lim[e]) {
                            usum += w[e]; ++counted;
                            ct[off_lo[e] + j * tile_step] = (int8_t)w[e];
                            if (row_hi_ok) {
                                usum += w[2 + e]; ++counted;
                                ct[off_hi[e] + j * tile_step] = (int8_t)w[2 + e];
                            }
                            if (pr.y) {
                                float* yt = pr.y + t * (int64_t)g.K + (nt0 * 8 + 2 * tq + e) * g.n2 + d0 + gq + j * tile_step;
                                yt[0] = acc[j][e];
                                if (row_hi_ok) yt[8] = acc[j][2 + e];
                            }
                        }
                    }
                }
            }
            if (pr.qsum) {
                int local = (int)(usum - (uint32_t)counted * (0x4B400000u + (uint32_t)pr.code_bias));
                local = __reduce_add_sync(0xFFFFFFFFu, local);
                if (lane == 0 && local != 0) atomicAdd(&sh.qsum[par][0], local);
            }
            if (tid == 0 && rank == 0) {
                pr.scales[t] = scale;
                if (pr.zp) pr.zp[t] = shift_i;
            }
        } else if (MODE == kRotDigits) {
            // The weight-only operating point for few tokens (gemm_small.cu): q = rne(value * 2^(21 - exponent of the largest)), a
            // 23-bit integer, as three signed base-256 digits.  Values down to 2^-14 of the largest are exact, smaller ones
            // within 2^-23 of it: what an fp32 sum of the values would round away.  (A token with an infinity or a NaN in it
            // gets a NaN scale.)
            const uint32_t top = slots_max(sh.amax[par]);
            const int es = 21 - exponent_of(__uint_as_float(top)), es2 = max(es - 126, 0);      // (to 148: in two factors)
            const float mult = pow2f(min(es, 126)), mult2 = pow2f(es2);
            const int64_t plane = p.M * (int64_t)g.K;
            int8_t* ct = pr.codes + t * (int64_t)g.K;
            const int tile_step = 8 * g.n2;
            int s0 = 0, s1 = 0, s2 = 0;               // sums of q, of q without its last digit, ... (wrap-around arithmetic)
#pragma unroll
            for (int j = 0; j < NTW; ++j) {
                int q0[4], q1[4], q2[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    q0[i] = __float_as_int(__fadd_rn(acc[j][i] * mult * mult2, 12582912.f)) - 0x4B400000;      // (the products are exact)
                    q1[i] = (q0[i] + 128) >> 8;
                    q2[i] = (q1[i] + 128) >> 8;
                }
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (8 * j < lim[e]) {
                        s0 += q0[e]; s1 += q1[e]; s2 += q2[e];
                        if (row_hi_ok) { s0 += q0[2 + e]; s1 += q1[2 + e]; s2 += q2[2 + e]; }
                        if (pairs16) {
                            int8_t* at = ct + off_lo[e] + j * tile_step;
                            *reinterpret_cast<uint16_t*>(at) = (uint16_t)__byte_perm(q0[e], q0[2 + e], 0x0040);
                            *reinterpret_cast<uint16_t*>(at + plane) = (uint16_t)__byte_perm(q1[e], q1[2 + e], 0x0040);
                            *reinterpret_cast<uint16_t*>(at + 2 * plane) = (uint16_t)__byte_perm(q2[e], q2[2 + e], 0x0040);
                        } else {
                            int8_t* at = ct + off_lo[e] + j * tile_step;
                            at[0] = (int8_t)q0[e]; at[plane] = (int8_t)q1[e]; at[2 * plane] = (int8_t)q2[e];
                            if (row_hi_ok) {
                                at = ct + off_hi[e] + j * tile_step;
                                at[0] = (int8_t)q0[2 + e]; at[plane] = (int8_t)q1[2 + e]; at[2 * plane] = (int8_t)q2[2 + e];
                            }
                        }
                    }
                }
            }
            const int d[3] = {s0 - 256 * s1, s1 - 256 * s2, s2};
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) {
                const int local = __reduce_add_sync(0xFFFFFFFFu, d[pl]);
                if (lane == 0 && local != 0) atomicAdd(&sh.qsum[par][pl], local);
            }
            if (tid == 0 && rank == 0) pr.scales[t] = top >= 0x7F800000u ? __uint_as_float(0x7FC00000u) : pow2f(es2 - es) * pow2f(-es2);
        } else if (MODE == kRotBf16) {
            // the weight-only operating point: bf16 values (layout 1: inside each group of 32, position 2 (k % 16) +
            // (k % 32) / 16), and where asked for their sum
            // (in fp64: sums in two floats cost the call without a shift, which has no sum, registers, 8.4 -> 9.0 us at 73 tokens of 64 x 64)
            __nv_bfloat16* yt = pr.yhat + t * (int64_t)g.K;
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < NTW; ++j) {
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    if (8 * j < lim[e]) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (h == 0 || row_hi_ok) {
                                const int k = off_lo[e] + 8 * h + j * 8 * g.n2;
                                const __nv_bfloat16 v = __float2bfloat16_rn(acc[j][2 * h + e]);
                                yt[pr.codes_layout ? (k & ~31) + 2 * (k & 15) + ((k >> 4) & 1) : k] = v;
                                if (pr.ysum) s += (double)__bfloat162float(v);
                            }
                        }
                    }
                }
            }
            if (pr.ysum) {
                s = total_sum(s, par);
                if (tid == 0 && rank == 0) pr.ysum[t] = (float)s;
            }
        } else {
            // Alg. 2, last step: the row's mean, its mean absolute deviation, and the signs about the mean
            // (in fp64: sums in two floats, one chain of dependent additions a thread, took longer, us: 15505 rows of 32 x 32 98 for 90, 1998 of
            // 32 x 64 27.6 for 25.3, 2348 of 86 x 128 187 for 172)
            double s = 0.0;
#pragma unroll
            for (int j = 0; j < NTW; ++j)             // (padding rows and columns are zeros)
#pragma unroll
                for (int i = 0; i < 4; ++i) s += (double)acc[j][i];
            const double mean = total_sum(s, 0) / (double)g.K;
            double dev = 0.0;
            uint32_t mine = 0u;                       // ballot number `lane` of the warp: column tile, row half, column parity
#pragma unroll
            for (int j = 0; j < NTW; ++j) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double x = (double)acc[j][i] - mean;
                    if (8 * j < lim[i & 1] && (i < 2 || row_hi_ok)) dev += fabs(x);
                    const uint32_t word = __ballot_sync(0xFFFFFFFFu, x > 0.0);
                    if (lane == 4 * j + i) mine = word;
                }
            }
            dev = total_sum(dev, 1) / (double)g.K;
            if (tid == 0 && rank == 0) { pr.mu[t] = (float)mean; pr.alpha[t] = (float)dev; }
            // bit 4 r + q of a ballot is row r (of the half), column pair q: the eight rows of a column are one byte of the row
            uint8_t* bytes = reinterpret_cast<uint8_t*>(pr.packed) + t * (int64_t)(g.K >> 3);
            const int j = lane >> 2, e = lane & 1, h = (lane >> 1) & 1;
            if (j < NTW && (h ? row_hi_ok : row_lo_ok)) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int c = (nt0 + j) * 8 + 2 * q + e;
                    uint32_t v = (mine >> q) & 0x11111111u;
                    v = (v | (v >> 3)) & 0x03030303u;
                    v = (v | (v >> 6)) & 0x000F000Fu;
                    v = (v | (v >> 12)) & 0xFFu;
                    if (c < g.n1) bytes[(c * g.n2 + d0 + 8 * h) >> 3] = (uint8_t)v;
                }
            }
        }
    }
    if ((MODE == kRotQuant || MODE == kRotDigits) && ntok > 0) {
        barrier();
        flush_qsum(tok0 + (int64_t)(ntok - 1) * stride, (ntok - 1) & 1);
    }
    if (MODE == kRotBinarize) __threadfence();       // (see above: complete in memory, not only issued)
    // nobody leaves while a neighbour may still store into its shared memory
    if (g.dc > 1) { cluster_arrive_release(); cluster_wait_acquire(); }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
bool rot_accepts_x(const void* x, int64_t ldx) { return (reinterpret_cast<uintptr_t>(x) & 15) == 0 && ldx % 8 == 0; }

typedef void (*RotKernel)(const RotKernelParams);

template <int MODE, bool F32>
static RotKernel pick_kernel(const RotGeom& g) {
    if (g.cw == 1)
        return g.ntw <= 2 ? rot_mma_kernel<2, false, MODE, F32> : g.ntw <= 4 ? rot_mma_kernel<4, false, MODE, F32>
             : g.ntw <= 6 ? rot_mma_kernel<6, false, MODE, F32> : rot_mma_kernel<8, false, MODE, F32>;
    if (MODE != kRotBinarize && g.ntw <= 4) return rot_mma_kernel<MODE == kRotBinarize ? 5 : 4, true, MODE, F32>;
    return g.ntw <= 5 ? rot_mma_kernel<5, true, MODE, F32> : g.ntw <= 6 ? rot_mma_kernel<6, true, MODE, F32>
         : g.ntw <= 7 ? rot_mma_kernel<7, true, MODE, F32> : rot_mma_kernel<8, true, MODE, F32>;
}

// How many clusters of the kernel the device holds at once (asked once per kernel, size and thread).
int resident_clusters(const void* k, int dc, int threads, size_t smem) {
    struct Known { const void* k; int dc, threads, dev, n; size_t smem; };
    static thread_local Known known[64];
    static thread_local int used = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    for (int i = 0; i < 64 && i < used; ++i)
        if (known[i].k == k && known[i].dc == dc && known[i].threads == threads && known[i].dev == dev && known[i].smem == smem) return known[i].n;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRotMaxSmem) != cudaSuccess) { cudaGetLastError(); return 0; }
    int n = 0;
    if (dc == 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) { cudaGetLastError(); return 0; }
        n *= sm_count();
    } else {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(dc * sm_count()), 1, 1);
        cfg.blockDim = dim3((unsigned)threads, 1, 1);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute a[1];
        a[0].id = cudaLaunchAttributeClusterDimension;
        a[0].val.clusterDim.x = (unsigned)dc; a[0].val.clusterDim.y = 1; a[0].val.clusterDim.z = 1;
        cfg.attrs = a; cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    }
    known[used % 64] = Known{k, dc, threads, dev, n, smem};
    ++used;
    return n;
}

// Few tokens: one group per CTA, so that they spread over the SMs; from there on as many as there are tokens for.
static int choose_groups(const RotGeom& g, int64_t M, int n_problems) {
    const int sms = std::max(1, sm_count());
    return (int)std::max<int64_t>(1, std::min<int64_t>(g.max_groups, (M * n_problems + sms - 1) / sms));
}

static int launch_rot_kernel(RotKernel k, const RotGeom& g, RotKernelParams& p, size_t smem, int lr_total, cudaStream_t stream) {
    const int threads = 32 * g.warps * p.groups;
    smem = std::max(smem, (size_t)(g.group_off + p.groups * g.group_bytes));
    const int room = resident_clusters((const void*)k, g.dc, threads, smem) / p.n_problems;
    if (room < 1) return cuda_fail(cudaErrorInvalidConfiguration);
    p.clusters_per_problem = (int)std::min<int64_t>((p.M + p.groups - 1) / p.groups, room);
    p.rot_ctas = p.n_problems * p.clusters_per_problem * g.dc;
    // (clusters that take tokens in turn hold their SMs to the end: the T = V x blocks then go first in block order)
    const bool stay = (int64_t)p.clusters_per_problem * p.groups < p.M;
    p.rot_first = (stay && lr_total > 0) ? (lr_total + g.dc - 1) / g.dc * g.dc : 0;
    int grid = p.rot_first ? p.rot_first + p.rot_ctas : p.rot_ctas + lr_total;
    grid = (grid + g.dc - 1) / g.dc * g.dc;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    // Clusters that stay are placed on an empty device: next to blocks of the kernel before they did not all fit at once, and
    // a cluster that starts when the others are through doubles the launch.
    attrs[0].val.programmaticStreamSerializationAllowed = (stay && g.dc > 1) ? 0u : launch_overlap_allowed();
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = (unsigned)g.dc; attrs[1].val.clusterDim.y = 1; attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = g.dc > 1 ? 2 : 1;
    ProfScope prof(kProfRotateQuant, stream);
    void* args[1] = {&p};
    cudaError_t e = cudaLaunchKernelExC(&cfg, (const void*)k, args);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}

static RotKernel rot_kernel_of(const RotGeom& g, const RotProblem& pr) {
    return pr.yhat ? pick_kernel<kRotBf16, false>(g) : pr.digits ? pick_kernel<kRotDigits, false>(g) : pick_kernel<kRotQuant, false>(g);
}

// Whether the device holds a cluster for every token at once, and the geometry that is spread for the time of one token.
static bool few_geometry(const RotGeom& base, int64_t M, int n_problems, const RotProblem* problems, RotGeom* g) {
    return M * n_problems <= sm_count() && few_tokens_geometry(base, !problems[0].prepared, g, [&](const RotGeom& t) {
        // (behind another kernel a cluster finds its place later than single CTAs do, where these are possible half of the SMs must be
        // left: 32 tokens of 108 x 128 in clusters of four 36 us a call, in CTAs 28)
        return t.dc == 1 || ((base.dc > 1 || 2 * M * n_problems * t.dc <= sm_count()) && M * n_problems <= resident_clusters((const void*)rot_kernel_of(t, problems[0]), t.dc, 32 * t.warps, (size_t)(t.group_off + t.group_bytes)));
    });
}
int rot_few_cluster(const RotGeom& base, int64_t M, int n_problems, const RotProblem* problems) {
    RotGeom g = base;
    return few_geometry(base, M, n_problems, problems, &g) ? g.dc : 1;
}

int launch_rot(const RotGeom& base, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems,
               const RotProblem* problems, const OktLowrank* lowrank, uint32_t* status, cudaStream_t stream, int behind) {
    if (M == 0 || n_problems == 0) return BWLA_OK;
    if (n_problems > kRotMaxProblems || M >= ((int64_t)1 << 31)) return BWLA_ERR_INVALID_ARG;
    const bool vec = rot_accepts_x(x, ldx);
    // ---- T = V x: beside the rotation, or before it in launches of its own.  Every kernel of the chain waits for its predecessor before it
    //      ends, so the contraction still finds T complete. ----
    OktLowrank beside[kRotMaxProblems] = {};          // what is left for blocks of the rotation's own launch
    bool any = false;
    for (int i = 0; lowrank && i < n_problems; ++i)
        if (lowrank[i].V && lowrank[i].r > 0 && lowrank[i].Thl) { beside[i] = lowrank[i]; any = true; }
    // on the tcgen05 tensor cores, for all linears that it takes at once
    auto on_tcgen05 = [&]() -> int {
        OktLowrank batch[kRotMaxProblems];
        int nb = 0;
        any = false;
        for (int i = 0; i < n_problems; ++i) {
            if (!beside[i].V) continue;
            if (lowrank_umma_takes(x, M, base.K, ldx, beside[i])) { batch[nb++] = beside[i]; beside[i] = OktLowrank{}; }
            else any = true;
        }
        return nb > 0 ? launch_lowrank_umma(x, M, base.K, ldx, nb, batch, status, stream) : BWLA_OK;
    };
    // as blocks of a launch of their own: `all`, or the wide tiles, whose registers do not fit beside the rotation
    auto own_launch = [&](bool all) -> int {
        for (int i = 0; i < n_problems; ++i) {
            if (!beside[i].V) continue;
            PrologueParams probe{};
            size_t bytes = 0;
            plan_lowrank(probe, x, M, base.K, ldx, beside[i], kRotMaxWarps, kRotMaxSmem, &bytes);
            if (!all && probe.lr_wide != 3) continue;
            const int st = launch_prologue(x, M, base.K, ldx, nullptr, 0, nullptr, 0, bits, nullptr, 0, nullptr, nullptr, beside[i].V, beside[i].r,
                                           beside[i].Thl, beside[i].lr_part, beside[i].lr_count ? beside[i].lr_count - kLrCounterWord : nullptr, stream);
            if (st != BWLA_OK) return st;
            beside[i] = OktLowrank{};
        }
        return BWLA_OK;
    };
    int st = M > 64 ? on_tcgen05() : BWLA_OK;
    if (st != BWLA_OK) return st;
    // ---- the kernel: while the device holds a cluster for every token, mma.sync, spread for the time of one token ----
    RotGeom g = base;
    const bool few = few_geometry(base, M, n_problems, problems, &g);
    // rot_rows.cu where it can and is no less exact and faster (T beside it by the warp-level MMA blocks only)
    auto rows_faster = [&]() {
        const int sms = sm_count();
        const bool t_first = M > 64 && lowrank && lowrank[0].r > 0;
        if (!few) return rot_rows_faster(base, problems[0].yhat != nullptr, !problems[0].prepared, any && M <= 64, t_first, M * n_problems, sms);
        if (problems[0].prepared || behind == 0 || M < 3 || sms < 1) return false;
        const int at_once = resident_clusters((const void*)rot_kernel_of(g, problems[0]), g.dc, 32 * g.warps, (size_t)(g.group_off + g.group_bytes)) * g.dc;
        const int per_sm = std::max(1, at_once / sms);
        return rot_rows_crowded(base, t_first, M * n_problems, (int)((M * n_problems * g.dc + per_sm - 1) / per_sm), behind, sms);
    };
    if (vec && rot_rows_exact(base, any) && rows_faster() && rot_rows_supports(base, n_problems, problems)) {
        if (any && M > 64) {
            st = own_launch(true);
            if (st != BWLA_OK) return st;
        }
        bool fits = true;
        for (int i = 0; i < n_problems; ++i) {
            if (!beside[i].V) continue;
            PrologueParams probe{};
            size_t bytes = 0;
            plan_lowrank(probe, x, M, base.K, ldx, beside[i], kRotMaxWarps, kRotMaxSmem, &bytes);
            fits = fits && (probe.lr_wide == 2 || probe.lr_wide == 4);
        }
        if (fits) return launch_rot_rows(base, x, M, ldx, bits, asym, n_problems, problems, beside, status, stream);
    }
    if (!few && vec) {
        RotRowsGeom rows;
        bool okt = rot_okt_factors(base) && !problems[0].yhat && !problems[0].digits && !rot_rows_geometry(base.n1, base.n2, 1, &rows);
        for (int i = 0; i < n_problems; ++i) okt = okt && (problems[i].many || !problems[i].prepared);
        OktGeom og;
        if (okt && okt_geometry(base.n1, base.n2, &og)) {
            st = own_launch(false);
            return st != BWLA_OK ? st : launch_okt(og, x, M, ldx, bits, asym, n_problems, problems, beside, status, stream);
        }
        // (which has no blocks for T beside it: with those, up to 64 tokens, the rounds of mma.sync are shorter than two more launches unless a
        // token takes a cluster; three linears with rank 64, 64 tokens: 64 x 128 39 | 52 us, 160 x 160 92 | 81)
        if (rot_umma_supports(base, n_problems, problems) && !(any && base.dc == 1)) {
            st = on_tcgen05();
            if (st == BWLA_OK) st = own_launch(true);
            return st != BWLA_OK ? st : launch_rot_umma(base, x, M, ldx, bits, asym, n_problems, problems, status, stream);
        }
    }
    st = own_launch(false);
    if (st != BWLA_OK) return st;
    RotKernelParams p{};
    p.g = g; p.x = x; p.ldx = ldx; p.x_vec = vec; p.M = M; p.bits = bits; p.asym = asym; p.n_problems = n_problems;
    p.status = status;
    p.groups = choose_groups(g, M, n_problems);
    size_t smem = 0;
    int lr_total = 0;
    for (int i = 0; i < n_problems; ++i) {
        p.prob[i] = problems[i];
        p.lr_begin[i] = lr_total;
        if (beside[i].V) {
            size_t lr_smem = 0;
            lr_total += plan_lowrank(p.lr[i], x, M, g.K, ldx, beside[i], g.warps * p.groups, kRotMaxSmem, &lr_smem);
            smem = std::max(smem, lr_smem);
        }
    }
    for (int i = n_problems; i <= kRotMaxProblems; ++i) p.lr_begin[i] = lr_total;
    return launch_rot_kernel(rot_kernel_of(g, problems[0]), g, p, smem, lr_total, stream);
}

int launch_rot_binarize(const RotGeom& g, const void* w, int dtype, int64_t N, int64_t ldw, const RotProblem& problem, uint32_t* status,
                        cudaStream_t stream) {
    if (N >= ((int64_t)1 << 31)) return BWLA_ERR_INVALID_ARG;
    bool taken = false;
    const int st = launch_rows_binarize(g, w, dtype, N, ldw, problem, status, &taken, stream);
    if (taken) return st;
    RotKernelParams p{};
    p.g = g; p.x = w; p.ldx = ldw; p.M = N; p.bits = 8; p.n_problems = 1; p.prob[0] = problem;
    p.status = status; p.groups = choose_groups(g, N, 1);
    p.x_vec = (reinterpret_cast<uintptr_t>(w) & 15) == 0 && ldw % (dtype == BWLA_DTYPE_F32 ? 4 : 8) == 0;
    RotKernel k = dtype == BWLA_DTYPE_F32 ? pick_kernel<kRotBinarize, true>(g) : pick_kernel<kRotBinarize, false>(g);
    return launch_rot_kernel(k, g, p, 0, 0, stream);
}

}  // namespace bwla
