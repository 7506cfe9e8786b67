// Online OKT (Sec. 3.1) for many tokens on the tcgen05 tensor cores, with the per-token quantiser (Sec. 4.1), the bf16 rounding of the
// weight-only operating point or the final binarisation of weight rows (Alg. 2) fused in, for factors of up to 128 x 128 (host_plans.h has
// the rule).
//
//   X = reshape(x_t, n1 x n2) (row-major),   V = P1^T X  [c][b],   Y = V P2  [c][d]
//
// The lanes of tensor memory are output rows c, of two tokens side by side where n1 <= 64, so that a lane's outputs are neighbours in
// memory, all four lane quarters have work and V meets P2 as the A operand where it lies.  (rot_umma.cu has Z^T = P2^T X^T first and rows
// d on the lanes: 80 of 128 lanes for n2 = 80, and codes that have to be gathered from eight lanes.)
//   first:  A = three bf16 terms of P1^T, B = x as TMA brings it (rows of k = a, N along the row); a step's tokens one after the other,
//           each into its own lanes
//   second: A = two fp16 terms of V in tensor memory, B = two fp16 terms of P2^T; three products
// Small products first.  V is scaled by a power of two of the token (its largest magnitude goes to [2^14, 2^15)), which leaves exactly
// with the scale of P2.  The tensor core truncates when it adds to its accumulator, so the first contraction is summed in two chains and the
// second in three (two for more than 80 rows and columns: host_plans.h), in accumulators of their own, and added with rounded additions.  (With two
// for the second 64 x 80 has 1.56e-7 of a row's 2-norm and 64 x 128 1.74e-7; with three 1.44e-7 and 1.55e-7.)
//
// The terms of V take the place of the first of its accumulators (a warp writes the lanes and columns that it has read), the third chain of
// Y that of the second.  Up to 80 columns there is a second pair for the next step's V; the MMAs then run a step ahead and are never waited for:
//   MMA warps   one issues V(0), V(1), and V(i + 2) behind Y(i), the other Y(i)
//   ALU warps   step i: V(i) to registers, the token's largest magnitude, two fp16 terms to tensor memory    (Y(i) may start)
//                       Y(i-1) to registers, the token's extremes, codes                                      (Y(i) may be written)
// With more columns Y(i-1) is read first and quantised under the MMAs of Y(i) and V(i+1).
//
// Bounds: up to 80 columns the ALU warps' instructions (a step of two tokens of 64 x 64 4000 cycles, 1000 of them MMAs); beyond, the chain V, exchange
// and terms, Y of a token (86 x 128: 6200 cycles, 3100 of them MMAs).  4096 tokens of 64 x 80 50 us (rot_mma.cu, whose MMAs take eight
// times as long, 86); of 86 x 128 113 (okt_umma.cu 137).  An MMA of 51 cycles took 110 to issue from run-time loops of one elected thread.
//
// Up to 64 x 80, fp32 rows of weights are split into three bf16 terms by the ALU warps, the next step's behind this step's V, and make six products with
// P1's; mean and mean absolute deviation are summed in fp64, and a lane's signs are neighbouring bits.
//
// Launched with programmatic stream serialisation: the factors are fetched before the preceding kernel of the stream has finished; x is
// read, and everything is stored, after it.  Every wait on an mbarrier is bounded (umma_wait.cuh); a warp whose wait ran out goes on
// through the token barriers without working.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "bwla_common.cuh"
#include "prologue_roles.cuh"
#include "rot_mma.cuh"
#include "tensor_map.cuh"
#include "umma_ptx.cuh"
#include "umma_wait.cuh"

namespace bwla {

namespace rr {
constexpr int kControl = 128;             // threads of the four control warps
// registers with two chunks a warp: 96 a thread at launch (640 x 96 = 61440); 128 x 32 + 512 x 112 = 61440 after the split
constexpr int kRegsControl = 32, kRegsAlu = 112;
constexpr int kSlots = 20;                // warps of a token, at most
constexpr int kNotFinite = 14 + 127 - 255;       // the exponent of V's scale where its largest magnitude is no number
struct Shared {
    uint64_t fac_full;                    // the prepared factors have landed
    uint64_t x_full[2], x_empty[2];       // a step's x has landed; the MMAs that read it have completed
    uint64_t v_full[2], y_full;           // the accumulators hold V, Y
    uint64_t v_empty[2];                  // V's terms have been read
    uint64_t y_free, y_read[2];           // Y has been read (for the warp that issues Y; by step parity for the one that issues V)
    uint64_t a_ready[2];                  // the terms of V are in tensor memory (by step parity: the ALU warps may be a step ahead)
    uint64_t out_full[2], out_free[2];    // the step's outputs and code sums are staged; have left
    uint32_t vmax[2][2][kSlots], ymax[2][2][kSlots], ymin[2][2][kSlots];       // [step parity][token][warp of the token]
    double dev[2][2][kSlots];             // ... sums of a binarisation's deviations
    int qsum[2][2];                       // code sums of the step's tokens
    uint32_t tmem_slot;
    int abort_flag, skip;
};
static_assert(sizeof(Shared) <= kRotRowsSharedBytes, "Shared");
}  // namespace rr

struct RotRowsParams {
    RotRowsGeom g;
    int64_t M;
    int bits;
    int n_problems, ctas_per_problem;
    const void* x; int64_t ldx; int x_vec;        // fp32 rows; whether they can be read in 16-byte pieces
    // T = V x beside the rotation (up to 64 tokens): problem i owns blocks [lr_begin[i], lr_begin[i + 1]) behind the rotation's
    int rot_ctas, lr_begin[kRotMaxProblems + 1];
    PrologueParams lr[kRotMaxProblems];
    RotProblem prob[kRotMaxProblems];
    uint32_t* status;
};

__device__ __forceinline__ float max_nan(float a, float b) {       // (a NaN if one of them is)
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// Where columns 2 k2, 2 k2 + 1 of row r lie in an operand of `rows` rows, 32 columns (64 bytes, swizzled) an atom.
__host__ __device__ __forceinline__ int rot_rows_place(int rows, int r, int k2) {
    return ((k2 >> 4) * rows + r) * 64 + ((((k2 >> 2) ^ (r >> 1)) & 3) << 4) + 4 * (k2 & 3);
}
// The terms of both factors as the kernel wants them; returns the exponent of P2's scale.  `red`: a word per warp.
__device__ __forceinline__ int rot_rows_split(const RotRowsGeom& g, const float* P1, const float* P2, uint8_t* image, uint32_t* red, int tid, int threads) {
    const int e2 = factor_exponent(block_absmax(P2, g.n2 * g.n2, red));
    split_factor<true>(P2, g.n2, 0, g.n2, 32 * g.atoms2, pow2f(e2), [&](int r, int k2) { return image + rot_rows_place(g.n2, r, k2); },
                       (size_t)g.atoms2 * g.n2 * 64, tid, threads);
    split_factor<false>(P1, g.n1, 0, g.lanes, 32 * g.atoms1, 1.f, [&](int r, int k2) { return image + g.p1_off + rot_rows_place(g.lanes, r, k2); },
                        (size_t)g.atoms1 * g.lanes * 64, tid, threads);
    return e2;
}
__global__ void __launch_bounds__(256) prepare_rows_kernel(RotRowsGeom g, const float* __restrict__ P1, const float* __restrict__ P2, uint8_t* __restrict__ prepared) {
    __shared__ uint32_t red[8];
    const int e2 = rot_rows_split(g, P1, P2, prepared + kRotHeader, red, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
    if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<int*>(prepared) = e2;
}
int launch_prepare_rows(const RotRowsGeom& g, const float* P1, const float* P2, void* prepared, cudaStream_t stream) {
    ProfScope prof(kProfPrepare, stream);
    prepare_rows_kernel<<<32, 256, 0, stream>>>(g, P1, P2, (uint8_t*)prepared);
    return after_launch();
}

// Steps of 16 values of the contractions: the first has two chains of sums, the second two or three (RotRowsGeom::y_chains).
__host__ __device__ constexpr int chain_end(int ks, int chains, int h) { return (ks * (h + 1) + chains - 1) / chains; }

// The MMAs of one product of the first contraction (one term of P1^T, one of x) into chain H, KS steps of 16 in all.  Unrolled: the issuing
// warp shares its scheduler with five others, and with run-time loops an MMA of 51 cycles took 110 to issue.
template <int KS, int H, bool FRESH>
__device__ __forceinline__ void issue_v(bool one, uint32_t v, uint32_t a, uint32_t a_hi, uint32_t blk, uint32_t b, uint32_t b_hi, uint32_t idesc,
                                        uint32_t skip_lo, uint32_t skip_hi) {
    constexpr int K0 = H == 0 ? 0 : chain_end(KS, 2, 0), K1 = chain_end(KS, 2, H);
    a += (uint32_t)(K0 >> 1) * blk;
#pragma unroll
    for (int k = K0; k < K1; ++k) {
        const uint32_t at = a + 2u * (k & 1), bt = b + 64u * (uint32_t)k;
        if (FRESH && k == K0) warp_mma_f16_ss_lanes<false>(one, v, at, a_hi, bt, b_hi, idesc, skip_lo, skip_hi);
        else warp_mma_f16_ss_lanes<true>(one, v, at, a_hi, bt, b_hi, idesc, skip_lo, skip_hi);
        if (k & 1) a += blk;
    }
}
// All products of a token into chain H, small ones first; XT: x has three terms, `x_term` apart.
template <int KS, int H, bool XT>
__device__ __forceinline__ void issue_token(bool one, uint32_t v, uint32_t a, uint32_t a_hi, uint32_t blk, uint32_t b, uint32_t b_hi, uint32_t idesc,
                                            uint32_t skip_lo, uint32_t skip_hi, uint32_t x_term) {
    const uint32_t term = (uint32_t)((KS + 1) / 2) * blk;
    issue_v<KS, H, true>(one, v, a + 2u * term, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi);
    if constexpr (XT) {
        issue_v<KS, H, false>(one, v, a + term, a_hi, blk, b + x_term, b_hi, idesc, skip_lo, skip_hi);
        issue_v<KS, H, false>(one, v, a, a_hi, blk, b + 2u * x_term, b_hi, idesc, skip_lo, skip_hi);
    }
    issue_v<KS, H, false>(one, v, a + term, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi);
    if constexpr (XT) issue_v<KS, H, false>(one, v, a, a_hi, blk, b + x_term, b_hi, idesc, skip_lo, skip_hi);
    issue_v<KS, H, false>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi);
}
template <int H, bool XT>
__device__ __forceinline__ void issue_token(int ks, bool one, uint32_t v, uint32_t a, uint32_t a_hi, uint32_t blk, uint32_t b, uint32_t b_hi, uint32_t idesc,
                                            uint32_t skip_lo, uint32_t skip_hi, uint32_t x_term) {
    switch (ks) {
        case 3: return issue_token<3, H, XT>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi, x_term);
        case 4: return issue_token<4, H, XT>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi, x_term);
        case 5: return issue_token<5, H, XT>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi, x_term);
        case 6: return issue_token<6, H, XT>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi, x_term);
        case 7: return issue_token<7, H, XT>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi, x_term);
        default: return issue_token<8, H, XT>(one, v, a, a_hi, blk, b, b_hi, idesc, skip_lo, skip_hi, x_term);
    }
}
// One product of the second contraction: 16 columns of V have left 8 of the first term and 8 of the second.
template <int KS, int CHAINS, bool FRESH>
__device__ __forceinline__ void issue_y(bool one, uint32_t y0, uint32_t y1, uint32_t y2, uint32_t a, uint32_t b, uint32_t b_hi, uint32_t blk, uint32_t idesc) {
    constexpr int E0 = chain_end(KS, CHAINS, 0), E1 = chain_end(KS, CHAINS, 1);
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        const uint32_t bt = b + 2u * (k & 1), y = k < E0 ? y0 : k < E1 ? y1 : y2;
        if (FRESH && (k == 0 || k == E0 || k == E1)) warp_mma_f16_ts<false>(one, y, a + 16u * (uint32_t)k, bt, b_hi, idesc);
        else warp_mma_f16_ts<true>(one, y, a + 16u * (uint32_t)k, bt, b_hi, idesc);
        if (k & 1) b += blk;
    }
}
template <int KS, int CHAINS = KS == 2 ? 2 : 3>
__device__ __forceinline__ void issue_outputs(bool one, uint32_t y0, uint32_t y1, uint32_t y2, uint32_t a, uint32_t b, uint32_t b_hi, uint32_t blk, uint32_t idesc) {
    const uint32_t term = (uint32_t)((KS + 1) / 2) * blk;
    issue_y<KS, CHAINS, true>(one, y0, y1, y2, a + 8u, b, b_hi, blk, idesc);          // lo hi
    issue_y<KS, CHAINS, false>(one, y0, y1, y2, a, b + term, b_hi, blk, idesc);       // hi lo
    issue_y<KS, CHAINS, false>(one, y0, y1, y2, a, b, b_hi, blk, idesc);              // hi hi
}

// MODE: the symmetric or the asymmetric quantiser, the weight-only operating point, or the binarisation of weight rows.  CH: 16-column
// chunks of a warp.  F32: x is fp32.
enum { kRowsSym = 0, kRowsAsym = 1, kRowsBf16 = 2, kRowsBinarize = 3 };
template <int MODE, int CH, bool F32 = false>
__global__ void __launch_bounds__(CH == 1 ? 768 : 640, 1)
rot_rows_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ RotRowsParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int NC = 16 * CH, NV = CH == 1 ? 2 : 1;
    const RotRowsGeom& g = p.g;
    rr::Shared& sh = *reinterpret_cast<rr::Shared*>(smem + g.sh_off);
    volatile int* abort_flag = &sh.abort_flag;
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    if (MODE != kRowsBinarize && (int)blockIdx.x >= p.rot_ctas) {
        // ---------------- T = V x blocks (two and one chunks of K in registers: 80 a thread) ----------------
        const int lb = (int)blockIdx.x - p.rot_ctas;
        int j = 0;
        while (j + 1 < p.n_problems && lb >= p.lr_begin[j + 1]) ++j;
        if (p.lr[j].lr_wide == 4) lowrank_mma_role<4, 1, false>(p.lr[j], lb - p.lr_begin[j], reinterpret_cast<float*>(smem));
        else lowrank_mma_role<2, 2, false>(p.lr[j], lb - p.lr_begin[j], reinterpret_cast<float*>(smem));
        return;
    }
    const int prob_i = (int)blockIdx.x / p.ctas_per_problem;
    const RotProblem& pr = p.prob[prob_i];
    const int64_t first = (int)blockIdx.x - prob_i * p.ctas_per_problem;      // steps first, first + CTAs, ...
    const int64_t steps_all = (p.M + g.tps - 1) / g.tps;
    const int alu_warps = 4 * g.groups;

    if (threadIdx.x == 0) {
        sh.abort_flag = 0;
        mbar_init(&sh.fac_full, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.x_full[i], F32 ? alu_warps : 1); mbar_init(&sh.x_empty[i], 1);
            mbar_init(&sh.v_full[i], 1); mbar_init(&sh.v_empty[i], 1);
            mbar_init(&sh.a_ready[i], alu_warps); mbar_init(&sh.y_read[i], alu_warps);
            mbar_init(&sh.out_full[i], alu_warps); mbar_init(&sh.out_free[i], 1);
            for (int j = 0; j < 2; ++j) sh.qsum[i][j] = 0;
        }
        mbar_init(&sh.y_full, 1); mbar_init(&sh.y_free, alu_warps);
        fence_barrier_init();
    }
    if (warp == 2) {
        tmem_alloc(&sh.tmem_slot, 512);
        tmem_relinquish();
    }
    // ---- the layer's factors (they do not depend on the preceding kernel; those of a binarisation may be what it has made) ----
    if (MODE == kRowsBinarize) griddep_wait();
    int e2;
    if (pr.many) {
        e2 = __ldg(reinterpret_cast<const int*>(pr.many));
        if (threadIdx.x == 0) {
            fence_proxy_async();
            mbar_expect_tx(&sh.fac_full, (uint32_t)g.x_off);
            tma_bulk_g2s(smem, pr.many + kRotHeader, (uint32_t)g.x_off, &sh.fac_full);
        }
    } else {
        e2 = rot_rows_split(g, pr.P1, pr.P2, smem, sh.vmax[0][0], threadIdx.x, blockDim.x);
        fence_proxy_async();
    }
    if (MODE == kRowsBinarize) {
        // (no dependent starts before this kernel has ended: its outputs are constants of the calls behind it, which they read before they
        // wait; this call clears its status words itself)
        if (blockIdx.x == 0 && threadIdx.x < kStatusBytes / 4) p.status[threadIdx.x] = 0u;
    } else if (threadIdx.x == 0) {
        // the call (or one before it) already failed: one answer for all warps, looked up while the factors and the tensor memory are on their way (a
        // failure of the kernel before that comes later is not seen, and this one's work is then done for nothing)
        sh.skip = p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&sh.tmem_slot);
    if (MODE != kRowsBinarize) {
        // (dependents start when every CTA has its tensor memory: one that got a CTA's columns first would wait for this grid with them)
        griddep_launch_dependents();
        griddep_wait();                               // x may be the output of the preceding kernel
    }
    const int n = (MODE == kRowsBinarize || !sh.skip) && first < steps_all ? (int)((steps_all - first + p.ctas_per_problem - 1) / p.ctas_per_problem) : 0;

    if (warp < 4) {
    if (CH == 2) set_regs_dec<rr::kRegsControl>();
    if (warp == 0) {
        // ---------------- x ----------------
        if (!F32 && elect_one()) {
            tma_prefetch_desc(&x_map);
            for (int i = 0; i < n; ++i) {
                const int b = g.xb == 2 ? i & 1 : 0;
                const uint32_t use = (uint32_t)(g.xb == 2 ? i >> 1 : i);
                if (!wait_or_abort(&sh.x_empty[b], (use & 1u) ^ 1u, abort_flag)) { give_up(p.status, abort_flag, 0x510); break; }
                const int t0 = (int)((first + (int64_t)i * p.ctas_per_problem) * g.tps);
                uint8_t* dst = smem + g.x_off + b * g.atoms2 * 8192;
                mbar_expect_tx(&sh.x_full[b], (uint32_t)(g.atoms2 * 8192));
                for (int a = 0; a < g.atoms2; ++a) tma_load_3d(dst + a * 8192, &x_map, 32 * a, 0, t0, &sh.x_full[b]);
            }
            if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);
        }
    } else if (warp == 1) {
        // ---------------- MMAs of the first contraction ----------------
        const bool one = elect_one();
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(g.n2 >> 3) << 17) | ((128u >> 4) << 24);
        const uint64_t d_p1 = smem_desc_kmajor(smem_u32(smem + g.p1_off), 64), d_x = smem_desc_mnmajor64(smem_u32(smem + g.x_off), 8192u);
        const uint32_t p1_hi = (uint32_t)(d_p1 >> 32), x_hi = (uint32_t)(d_x >> 32);
        const uint32_t blk1 = (uint32_t)(g.lanes * 64) >> 4, n2 = (uint32_t)g.n2;
        bool ok = true;
        if (pr.many && !warp_wait(&sh.fac_full, 0u, abort_flag)) { give_up(p.status, abort_flag, 0x521); ok = false; }
        for (int i = 0; i < n && ok; ++i) {
            const int b = g.xb == 2 ? i & 1 : 0;
            const uint32_t use = (uint32_t)(g.xb == 2 ? i >> 1 : i);
            if (!warp_wait(&sh.x_full[b], use & 1u, abort_flag)) { give_up(p.status, abort_flag, 0x520); break; }
            if (i >= NV && !warp_wait(&sh.v_empty[i % NV], (uint32_t)((i / NV - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x524); break; }
            tc_fence_after();
            const uint32_t v = tmem + (uint32_t)((i % NV) * 2) * n2, x0 = (uint32_t)d_x + (uint32_t)(b * g.atoms2) * (8192u >> 4);
            const uint32_t x_term = F32 ? (uint32_t)g.atoms2 * (8192u >> 4) : 0u;
            auto chain = [&](auto h_) {
                constexpr int H = decltype(h_)::value;
                for (int tk = 0; tk < g.tps; ++tk) {
                    // the token's lanes (what the other lanes would add, rows outside P1's terms times this token, is not a zero where x
                    // holds an infinity)
                    const uint32_t skip_lo = tk == 1 ? 0xFFFFFFFFu : 0u, skip_hi = g.tps == 2 && tk == 0 ? 0xFFFFFFFFu : 0u;
                    issue_token<H, F32>(g.ks1, one, v + (uint32_t)H * n2, (uint32_t)d_p1 - (uint32_t)tk * blk1, p1_hi, blk1, x0 + (uint32_t)tk * 256u, x_hi, idesc,
                                        skip_lo, skip_hi, x_term);
                }
            };
            chain(std::integral_constant<int, 0>{});
            // (the third chain of Y(i - NV) lay where the second of V goes)
            if (i >= NV && g.y_chains == 3 && !warp_wait(&sh.y_read[(i - NV) & 1], (uint32_t)(((i - NV) >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x525); break; }
            tc_fence_after();
            chain(std::integral_constant<int, 1>{});
            if (one) { tc_commit(&sh.x_empty[b]); tc_commit(&sh.v_full[i % NV]); }
            __syncwarp();
        }
    } else if (warp == 2) {
        // ---------------- MMAs of the second ----------------
        const bool one = elect_one();
        const uint32_t idesc = (1u << 4) | ((uint32_t)(g.n2 >> 3) << 17) | ((128u >> 4) << 24);
        const uint64_t d_p2 = smem_desc_kmajor(smem_u32(smem), 64);
        const uint32_t p2_hi = (uint32_t)(d_p2 >> 32), blk2 = (uint32_t)(g.n2 * 64) >> 4, n2 = (uint32_t)g.n2;
        for (int i = 0; i < n; ++i) {
            if (!warp_wait(&sh.a_ready[i & 1], (uint32_t)((i >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x522); break; }
            if (i >= 1 && !warp_wait(&sh.y_free, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x523); break; }
            tc_fence_after();
            const uint32_t a = tmem + (uint32_t)((i % NV) * 2) * n2, y = tmem + (uint32_t)(NV * 2) * n2;
            const uint32_t p2 = (uint32_t)d_p2, y1 = y + n2, y2 = a + n2;
            if (CH == 1) {
                switch (g.ks2) {
                    case 2: issue_outputs<2>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    case 3: issue_outputs<3>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    case 4: issue_outputs<4>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    default: issue_outputs<5>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                }
            } else if (g.y_chains == 3) {
                switch (g.ks2) {
                    case 6: issue_outputs<6>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    case 7: issue_outputs<7>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    default: issue_outputs<8>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                }
            } else {
                switch (g.ks2) {
                    case 6: issue_outputs<6, 2>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    case 7: issue_outputs<7, 2>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                    default: issue_outputs<8, 2>(one, y, y1, y2, a, p2, p2_hi, blk2, idesc); break;
                }
            }
            if (one) { tc_commit(&sh.v_empty[i % NV]); tc_commit(&sh.y_full); }
            __syncwarp();
        }
    } else if (warp == 3 && MODE != kRowsBinarize) {
        // ---------------- code sums and staged outputs of a step ----------------
        for (int i = 0; i < n; ++i) {
            const int par = i & 1;
            if (!warp_wait(&sh.out_full[par], (uint32_t)((i >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x540); break; }
            const int64_t t0 = (first + (int64_t)i * p.ctas_per_problem) * g.tps;
            const int tokens = (int)min((int64_t)g.tps, p.M - t0);
            if (g.staged && lane == 0) {
                const int size = g.out_bytes / g.tps;
                uint8_t* dst = MODE == kRowsBf16 ? reinterpret_cast<uint8_t*>(pr.yhat) : reinterpret_cast<uint8_t*>(pr.codes);
                bulk_s2g(dst + t0 * size, smem + g.st_off + par * g.out_bytes, (uint32_t)(tokens * size));
            }
            if (MODE != kRowsBf16 && pr.qsum) {
                const int tk = lane >> 3, part = lane & 7;
                static_assert(kQsumParts == 8, "a lane per part");
                const int sum = tk < 2 ? sh.qsum[par][tk] : 0;
                __syncwarp();
                if (part == 0 && tk < 2) sh.qsum[par][tk] = 0;
                if (tk < tokens) pr.qsum[(t0 + tk) * kQsumParts + part] = part == 0 ? sum : 0;
            }
            if (g.staged && lane == 0) bulk_wait_read();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.out_free[par]);
        }
        if (g.staged && lane == 0) bulk_wait_all();
    }
    } else {
        if (CH == 2) set_regs_inc<rr::kRegsAlu>();
        // ---------------- everything between and behind the MMAs ----------------
        const int w = warp - 4, q = w & 3, wc = w >> 2;
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        const int tk = q * 32 / g.lanes;              // this quarter's token of the step
        const int c = (q * 32 + lane) & (g.lanes - 1);
        const bool valid = c < g.n1;
        const int slots = g.groups * (g.lanes >> 5), slot = wc * (g.lanes >> 5) + (q & ((g.lanes >> 5) - 1));
        const int c0 = NC * wc, have = min(NC, g.n2 - c0);            // this warp's columns of V
        // Its columns of Y.  Where rows are whole groups of 32 outputs and a warp has 16 columns, they are those that make 16 (or, of bf16
        // values, 32) neighbouring bytes of the contractions' order: a half of a group, four (eight) columns of every eight (sixteen).
        constexpr int RUN = MODE == kRowsBf16 ? 8 : 4;
        const bool gather = MODE != kRowsBinarize && CH == 1 && (g.n2 & 31) == 0;
        const int y0 = gather ? 32 * (wc >> 1) + RUN * (wc & 1) : c0;
        auto column = [&](int e) { return y0 + (gather ? e % RUN + (32 / (16 / RUN)) * (e / RUN) : e); };
        bool ok = true;
        int z_exp = 0;
        auto token_barrier = [&]() { named_barrier(1 + tk, g.groups * g.lanes); };
        // ---- fp32 rows: eight values of step `i` to the three terms in x's place (rows beyond n1 and M are zeros)
        const int cpr = g.n2 >> 3, alu_threads = 32 * alu_warps;
        // (the L2 is asked for a step's rows three steps before it: 5120 x 5120 143 us without, 129 with (sums in two floats); the first pass over new pages 255 and 194)
        auto ask_x = [&](int i) {
            if (!F32 || !p.x_vec || threadIdx.x != rr::kControl || i >= n) return;
            const int64_t t = (first + (int64_t)i * p.ctas_per_problem) * g.tps;
            for (int j = 0; j < g.tps && t + j < p.M; ++j)
                prefetch_l2_bulk(reinterpret_cast<const float*>(p.x) + (t + j) * p.ldx, (uint32_t)(g.K * 4));
        };
        auto load_x = [&](int i, int j, float (&f)[8]) {
            const int r = j / cpr, a = r & (g.lanes - 1);
            const int64_t t = (first + (int64_t)i * p.ctas_per_problem) * g.tps + r / g.lanes;
            if (a < g.n1 && t < p.M) {
                const float* src = reinterpret_cast<const float*>(p.x) + t * p.ldx + a * g.n2 + 8 * (j - r * cpr);
                if (p.x_vec) {
                    const float4 lo = __ldg(reinterpret_cast<const float4*>(src)), hi = __ldg(reinterpret_cast<const float4*>(src) + 1);
                    f[0] = lo.x; f[1] = lo.y; f[2] = lo.z; f[3] = lo.w; f[4] = hi.x; f[5] = hi.y; f[6] = hi.z; f[7] = hi.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) f[e] = __ldg(src + e);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) f[e] = 0.f;
            }
        };
        auto put_x = [&](int j, const float (&f)[8]) {
            const int r = j / cpr, ch = j - r * cpr;
            uint8_t* const at = smem + g.x_off + (ch >> 2) * 8192 + r * 64 + (((ch ^ (r >> 1)) & 3) << 4);
            uint32_t h[4], m[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) split3_pair(f[2 * e], f[2 * e + 1], h[e], m[e], l[e]);
            *reinterpret_cast<uint4*>(at) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(at + g.atoms2 * 8192) = make_uint4(m[0], m[1], m[2], m[3]);
            *reinterpret_cast<uint4*>(at + 2 * g.atoms2 * 8192) = make_uint4(l[0], l[1], l[2], l[3]);
        };
        auto x_done = [&]() {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.x_full[0]);
        };
        // (128 n2 / 8 pieces a step for 8 n2 threads: two a thread)
        if (F32 && n > 0) {
            ask_x(1); ask_x(2);
            float f[2][8];
            const int j = threadIdx.x - rr::kControl;
            const bool two = j + alu_threads < 128 * cpr;
            load_x(0, j, f[0]);
            if (two) load_x(0, j + alu_threads, f[1]);
            put_x(j, f[0]);
            if (two) put_x(j + alu_threads, f[1]);
            x_done();
        }
#pragma unroll 1
        for (int i = 0; i <= n; ++i) {
            const int par = i & 1, pi = par ^ 1;
            const int64_t t = (first + (int64_t)(i - 1) * p.ctas_per_problem) * g.tps + tk;       // of Y
            float v[NC], y[NC];
            float f1 = 1.f, amax = 0.f, vmin = 0.f;
            auto load_v = [&]() {
                if (ok && !warp_wait(&sh.v_full[i % NV], (uint32_t)((i / NV) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x531); ok = false; }
                float m = 0.f;
                if (ok) {
                    tc_fence_after();
                    const uint32_t src = tmem + lane_addr + (uint32_t)((i % NV) * 2 * g.n2 + c0);
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch)
                        if (16 * ch < have) {
                            uint32_t u[16];
                            tmem_ld_words<16>(src + 16 * ch, reinterpret_cast<uint32_t*>(v) + 16 * ch);
                            tmem_ld_words<16>(src + (uint32_t)g.n2 + 16 * ch, u);
                            tc_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; e += 2) {
                                add2(v[16 * ch + e], v[16 * ch + e + 1], __uint_as_float(u[e]), __uint_as_float(u[e + 1]));
                                m = max_nan(m, max_nan(fabsf(v[16 * ch + e]), fabsf(v[16 * ch + e + 1])));
                            }
                        }
                }
                const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, valid ? __float_as_uint(m) : 0u);
                if (lane == 0) sh.vmax[par][tk][slot] = top;
            };
            auto convert = [&]() {
                const uint32_t top = __reduce_max_sync(0xFFFFFFFFu, lane < slots ? *reinterpret_cast<volatile uint32_t*>(&sh.vmax[par][tk][lane]) : 0u);
                z_exp = max(-126, min(126, 14 + 127 - (int)(top >> 23)));      // (kNotFinite where V holds an infinity or a NaN)
                const float scale = pow2f(z_exp);
                if (ok) {
                    const uint32_t dst = tmem + lane_addr + (uint32_t)((i % NV) * 2 * g.n2 + c0);
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch)
                        if (16 * ch < have) {
                            uint32_t h[8], l[8];
#pragma unroll
                            for (int e = 0; e < 8; ++e) {
                                mul2(v[16 * ch + 2 * e], v[16 * ch + 2 * e + 1], scale);
                                split2_pair(v[16 * ch + 2 * e], v[16 * ch + 2 * e + 1], h[e], l[e]);
                            }
                            tmem_st_32x8(dst + 16 * ch, h);
                            tmem_st_32x8(dst + 16 * ch + 8, l);
                        }
                    tc_wait_st();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.a_ready[par]);
            };
            auto load_y = [&](int ze) {
                if (ok && !warp_wait(&sh.y_full, (uint32_t)((i - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x530); ok = false; }
                uint32_t top = 0u, bottom = 0u;
                if (ok) {
                    tc_fence_after();
                    const uint32_t src = tmem + lane_addr + (uint32_t)(NV * 2 * g.n2 + y0);
                    uint32_t* const yw = reinterpret_cast<uint32_t*>(y);
                    const uint32_t third = tmem + lane_addr + (uint32_t)(((i - 1) % NV) * 2 * g.n2 + g.n2 + y0);
                    auto load = [&](uint32_t at, uint32_t* w) {
                        if (gather) {
#pragma unroll
                            for (int r = 0; r < 16 / RUN; ++r) tmem_ld_words<RUN>(at + (32 / (16 / RUN)) * r, w + RUN * r);
                        } else {
                            tmem_ld_words<16>(at, w);
                        }
                    };
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch)
                        if (16 * ch < have) {
                            uint32_t u[16];
                            load(src + 16 * ch, yw + 16 * ch);
                            load(src + (uint32_t)g.n2 + 16 * ch, u);
                            tc_wait_ld();
#pragma unroll
                            for (int e = 0; e < 16; e += 2) add2(y[16 * ch + e], y[16 * ch + e + 1], __uint_as_float(u[e]), __uint_as_float(u[e + 1]));
                            if (g.y_chains == 3) {
                                load(third + 16 * ch, u);
                                tc_wait_ld();
#pragma unroll
                                for (int e = 0; e < 16; e += 2) add2(y[16 * ch + e], y[16 * ch + e + 1], __uint_as_float(u[e]), __uint_as_float(u[e + 1]));
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < 16; ++e) y[16 * ch + e] = 0.f;
                        }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) { mbar_arrive(&sh.y_free); mbar_arrive(&sh.y_read[pi]); }
                if (!ok) return;
                const int ey = -(ze + e2), ey1 = max(-126, min(127, ey)), ey2 = max(-126, min(127, ey - ey1));
                f1 = pow2f(ey1);
                if (ey2 != 0) {                               // scales at the ends of fp32's range
                    const float f2 = pow2f(ey2);
#pragma unroll
                    for (int e = 0; e < NC; ++e) y[e] = y[e] * f1 * f2;
                    f1 = 1.f;
                }
                if (MODE == kRowsBf16 || MODE == kRowsBinarize) {
                    // the sum of the values goes where the quantiser's two extremes go
                    if (MODE == kRowsBinarize || pr.ysum) {
                        double s = 0.0, s1 = 0.0;             // (of the scaled, or the rounded values; two chains)
#pragma unroll
                        for (int e = 0; e < NC; e += 2) {
                            s += (double)(MODE == kRowsBinarize ? y[e] : __bfloat162float(__float2bfloat16_rn(y[e] * f1)));
                            s1 += (double)(MODE == kRowsBinarize ? y[e + 1] : __bfloat162float(__float2bfloat16_rn(y[e + 1] * f1)));
                        }
                        s = warp_sum(valid ? s + s1 : 0.0);
                        top = (uint32_t)__double2loint(s); bottom = (uint32_t)__double2hiint(s);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < NC; e += 2) {
                        if (MODE == kRowsSym) amax = fmaxf(amax, fmaxf(fabsf(y[e]), fabsf(y[e + 1])));
                        else { amax = fmaxf(amax, fmaxf(y[e], y[e + 1])); vmin = fminf(vmin, fminf(y[e], y[e + 1])); }
                    }
                    if (!valid) amax = vmin = 0.f;            // (rows beyond P1's hold anything)
                    // non-negative (NaNs aside), so their bit patterns order like the values
                    top = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax * f1));
                    if (MODE == kRowsAsym) bottom = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(fmaxf(-vmin * f1, 0.f)));
                }
                if (lane == 0) { sh.ymax[par][tk][slot] = top; if (MODE != kRowsSym) sh.ymin[par][tk][slot] = bottom; }
            };
            // ---- the step before: codes, scale and code sum, or bf16 values
            auto emit = [&](int ze) {
                const uint32_t s0 = lane < slots ? *reinterpret_cast<volatile uint32_t*>(&sh.ymax[par][tk][lane]) : 0u;
                const uint32_t s1 = MODE != kRowsSym && lane < slots ? *reinterpret_cast<volatile uint32_t*>(&sh.ymin[par][tk][lane]) : 0u;
                if (ok && i >= 3 && !warp_wait(&sh.out_free[pi], (uint32_t)((((i - 1) >> 1) - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x534); ok = false; }
                if (ok && t < p.M) {
                    const bool writer = slot == 0;                // of the token's scalars
                    uint8_t* const stage = smem + g.st_off + pi * g.out_bytes + tk * (g.out_bytes / g.tps);
                    const int k0 = c * g.n2 + y0;
                    if (MODE == kRowsBf16) {
                        if (writer && pr.ysum) {
                            const double s = warp_sum(__hiloint2double((int)s1, (int)s0));
                            if (lane == 0) pr.ysum[t] = (float)s;
                        }
                        // layout 1: inside each group of 32, position 2 (k % 16) + (k % 32) / 16
                        uint16_t* const yt = g.staged ? reinterpret_cast<uint16_t*>(stage) : reinterpret_cast<uint16_t*>(pr.yhat + t * (int64_t)g.K);
                        if (!valid) {
                        } else if (pr.codes_layout && !g.staged) {
                            uint4* const at = reinterpret_cast<uint4*>(yt + (k0 & ~31) + 2 * (k0 & 15));
                            if (CH == 1) {
                                uint32_t o[8];
#pragma unroll
                                for (int e = 0; e < 8; ++e) o[e] = cvt_bf16x2_rn(y[e] * f1, y[8 + e] * f1);
                                at[0] = make_uint4(o[0], o[1], o[2], o[3]); at[1] = make_uint4(o[4], o[5], o[6], o[7]);
                            } else {
#pragma unroll
                                for (int s = 0; s < 4; ++s) {
                                    uint32_t o[4];
#pragma unroll
                                    for (int e = 0; e < 4; ++e) o[e] = cvt_bf16x2_rn(y[(4 * s + e) % NC] * f1, y[(16 + 4 * s + e) % NC] * f1);
                                    at[s] = make_uint4(o[0], o[1], o[2], o[3]);
                                }
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < NC; ++e) {
                                const int k = c * g.n2 + column(e);
                                if (e < have) yt[pr.codes_layout ? (k & ~31) + 2 * (k & 15) + ((k >> 4) & 1) : k] = __bfloat16_as_ushort(__float2bfloat16_rn(y[e] * f1));
                            }
                        }
                    } else {
                        amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, s0));
                        if (MODE == kRowsAsym) vmin = -__uint_as_float(__reduce_max_sync(0xFFFFFFFFu, s1));
                        // The quantiser of rot_mma.cu with the same roundings: fl(v + 1.5 * 2^23 + shift) leaves rne(v) + shift in the low
                        // mantissa bits, the low byte is stored.
                        const float levels = MODE == kRowsSym ? (float)((1 << (p.bits - 1)) - 1) : (float)((1 << p.bits) - 1);
                        const float range = MODE == kRowsSym ? amax : __fsub_rn(amax, vmin);
                        const float inv = range != 0.f ? __fdiv_rn(levels, range) : 0.f;
                        float zero_f = 0.f, half_f = 0.f;
                        if (MODE == kRowsAsym) {
                            const float tz = __fmul_rn(-vmin, inv);
                            zero_f = fminf(fmaxf(__fadd_rn(__fadd_rn(tz, 12582912.f), -12582912.f), 0.f), levels);
                            half_f = (float)(1 << (p.bits - 1));
                        }
                        const float store_shift = (float)pr.code_bias - half_f;
                        const int shift_i = (int)(zero_f + store_shift);
                        const uint32_t odd = (uint32_t)(shift_i & 1);
                        // (every code is shifted to c + 128 - bias >= 0: the bits of 1.5 * 2^23 below bit 16 are zero, so four codes make a word by
                        // multiply-adds and nothing carries from one byte into the next)
                        const float bias = 12582912.f + (float)(shift_i - (int)odd + 128 - pr.code_bias);
                        const float lo = 12582912.f + store_shift - (float)odd + (float)(128 - pr.code_bias), hi = lo + levels;
                        if (writer && lane == 0) {
                            pr.scales[t] = range != 0.f ? __fdiv_rn(range, levels) : 1.f;
                            if (pr.zp) pr.zp[t] = shift_i;
                        }
                        if (pr.y && valid) {
#pragma unroll
                            for (int e = 0; e < NC; ++e)
                                if (e < have) pr.y[t * (int64_t)g.K + c * g.n2 + column(e)] = y[e] * f1;
                        }
                        // fl(y inv) = fl(y_scaled (f inv)): f is a power of two, and where f inv leaves fp32's normal range the values are too
                        // small against the token's largest for any code but zero
                        const float f_inv = inv * f1;
                        if (MODE == kRowsSym && (ze == rr::kNotFinite || inv > 3.402823466e38f)) {
                            // as the other kernels have it: the code of a NaN is -1, and where the token is so small that inv overflows codes are 0
                            // (the words below are put together by additions, which neither pattern may carry into)
#pragma unroll
                            for (int e = 0; e < NC; ++e) {
                                const float c0 = __fmul_rn(y[e], f_inv);
                                y[e] = y[e] != y[e] ? -1.f : fabsf(c0) <= 128.f ? c0 : 0.f;
                            }
                        } else {
#pragma unroll
                            for (int e = 0; e < NC; ++e) y[e] = __fmul_rn(y[e], f_inv);
                        }
#pragma unroll
                        for (int e = 0; e < NC; e += 2) add2(y[e], y[e + 1], bias, bias);
                        if (MODE == kRowsAsym)
#pragma unroll
                            for (int e = 0; e < NC; ++e) y[e] = fminf(fmaxf(y[e], lo), hi);
                        // w0 + 2^8 w1 has 0x8B40 above its two bytes; that of the lower pair is taken off the upper one
                        const uint32_t top = MODE == kRowsAsym ? 0x74C00000u + 0x01010101u * odd : 0x74C00000u;
                        uint32_t sum = 0u;
                        auto word = [&](int e0, int e1, int e2_, int e3) -> uint32_t {      // four codes, the first lowest
                            const uint32_t p01 = __float_as_uint(y[e1 % NC]) * 256u + __float_as_uint(y[e0 % NC]);
                            const uint32_t p23 = __float_as_uint(y[e3 % NC]) * 256u + __float_as_uint(y[e2_ % NC]);
                            const uint32_t o = p23 * 65536u + (p01 + top);
                            sum = __dp4a(o, 0x01010101u, sum);
                            return pr.code_bias ? o - 0x01010101u * (uint32_t)(128 - pr.code_bias) : o ^ 0x80808080u;
                        };
                        uint8_t* const ct = g.staged ? stage : reinterpret_cast<uint8_t*>(pr.codes) + t * (int64_t)g.K;
                        if (pr.codes_layout && !g.staged) {
                            // inside each group of 32, byte 4 j + i holds k = j + 8 i
                            uint4* const at = reinterpret_cast<uint4*>(ct + (k0 & ~31) + 4 * (k0 & 7));
                            if (CH == 1) {
                                uint32_t o[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) o[j] = word(j, 4 + j, 8 + j, 12 + j);
                                if (valid) at[0] = make_uint4(o[0], o[1], o[2], o[3]);
                            } else {
#pragma unroll
                                for (int s = 0; s < 2; ++s) {
                                    uint32_t o[4];
#pragma unroll
                                    for (int j = 0; j < 4; ++j) o[j] = word(4 * s + j, 8 + 4 * s + j, 16 + 4 * s + j, 24 + 4 * s + j);
                                    if (valid) at[s] = make_uint4(o[0], o[1], o[2], o[3]);
                                }
                            }
                        } else if (pr.codes_layout) {
                            // 16 columns are half of a group: two bytes of every four
#pragma unroll
                            for (int ch = 0; ch < CH; ++ch) {
                                if (16 * ch >= have) break;
                                const int kc = k0 + 16 * ch;
                                const uint32_t at = smem_u32(ct) + (uint32_t)((kc & ~31) + 2 * ((kc >> 4) & 1));
                                uint32_t o[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) o[j] = word(16 * ch + 2 * j, 16 * ch + 8 + 2 * j, 16 * ch + 2 * j + 1, 16 * ch + 9 + 2 * j);
                                // Rows start n2 bytes apart, so that every eighth lane has the same bank: lanes 8 r ... start at word r.
                                const int r = lane >> 3;
                                const uint32_t half = r & 1 ? 0x5432u : 0x3210u;
                                uint32_t w[4];
#pragma unroll
                                for (int j = 0; j < 4; ++j) w[j] = r & 2 ? o[(j + 1) & 3] : o[j];
#pragma unroll
                                for (int j = 0; j < 4; ++j) o[j] = __byte_perm(w[j], w[(j + 1) & 3], half);
#pragma unroll
                                for (int j = 0; j < 8; ++j) {
                                    const uint32_t to = at + 4u * (uint32_t)((j + r) & 7);
                                    if (valid) st_shared_u16(to, j & 1 ? o[j >> 1] >> 16 : o[j >> 1]);
                                }
                            }
                        } else {
                            // natural order: runs of four columns are neighbours
#pragma unroll
                            for (int e = 0; e < NC; e += 4) {
                                if (e >= have) break;
                                const uint32_t o = word(e, e + 1, e + 2, e + 3);
                                if (valid) *reinterpret_cast<uint32_t*>(ct + c * g.n2 + column(e)) = o;
                            }
                        }
                        if (pr.qsum) {
                            const int own = (int)sum - have * 128;                // (less the bias)
                            const int local = __reduce_add_sync(0xFFFFFFFFu, valid ? own : 0);
                            if (lane == 0 && local != 0) atomicAdd(&sh.qsum[pi][tk], local);
                        }
                    }
                }
                if (g.staged) fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.out_full[pi]);
            };
            // ---- the step before, a binarisation (Alg. 2, last step): the row's mean, its mean absolute deviation, and the signs about the mean
            auto binarize = [&]() {
                const uint32_t s0 = lane < slots ? *reinterpret_cast<volatile uint32_t*>(&sh.ymax[par][tk][lane]) : 0u;
                const uint32_t s1 = lane < slots ? *reinterpret_cast<volatile uint32_t*>(&sh.ymin[par][tk][lane]) : 0u;
                const double mean = warp_sum(__hiloint2double((int)s1, (int)s0)) / (double)g.K;          // (of the scaled values)
                const float below = __double2float_rd(mean);                                             // (a float is above the mean where it is above this)
                double dev = 0.0, dev1 = 0.0;
                uint32_t bits = 0u;
#pragma unroll
                for (int e = 0; e < NC; e += 2) {
                    bits |= (y[e] > below ? 1u << (e & 31) : 0u) | (y[e + 1] > below ? 2u << (e & 31) : 0u);
                    dev += fabs((double)y[e] - mean);
                    dev1 += fabs((double)y[e + 1] - mean);
                }
                if (ok && valid && t < p.M) {
                    reinterpret_cast<uint16_t*>(pr.packed)[(t * (int64_t)g.K + c * g.n2 + y0) >> 4] = (uint16_t)bits;
                }
                dev = warp_sum(valid ? dev + dev1 : 0.0);
                if (lane == 0) sh.dev[par][tk][slot] = dev;
                token_barrier();
                if (slot == 0) {
                    const double all = warp_sum(lane < slots ? *reinterpret_cast<volatile double*>(&sh.dev[par][tk][lane]) : 0.0);
                    if (lane == 0 && ok && t < p.M) {
                        pr.mu[t] = (float)(mean * (double)f1);
                        pr.alpha[t] = (float)(all / (double)g.K * (double)f1);
                    }
                }
            };
            const int ze = z_exp;
            if (MODE == kRowsBinarize) {
                if (i < n) {
                    // the next step's rows are on their way while this step's V is waited for; its accumulation has read x then
                    float f[2][8];
                    const int j = threadIdx.x - rr::kControl;
                    const bool more = F32 && i + 1 < n, two = j + alu_threads < 128 * cpr;
                    ask_x(i + 3);
                    if (more) { load_x(i + 1, j, f[0]); if (two) load_x(i + 1, j + alu_threads, f[1]); }
                    load_v();
                    if (more) { put_x(j, f[0]); if (two) put_x(j + alu_threads, f[1]); x_done(); }
                    token_barrier();
                    convert();
                }
                if (i > 0) load_y(ze);
                if (i > 0) token_barrier();
                if (i > 0) binarize();
            } else if (NV == 2) {
                // (one exchange for both: Y(i - 1) has had the end of the step before to complete)
                if (i < n) load_v();
                if (i > 0) load_y(ze);
                token_barrier();
                if (i < n) convert();
                if (i > 0) emit(ze);
            } else {
                if (i > 0) load_y(ze);
                if (i < n) load_v();
                token_barrier();
                if (i < n) convert();
                if (i > 0) emit(ze);
            }
        }
        if (!ok) *abort_flag = 1;
        if (MODE == kRowsBinarize) __threadfence();   // (see above: complete in memory, not only issued)
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
}

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
bool rot_rows_supports(const RotGeom& base, int n_problems, const RotProblem* problems) {
    for (int i = 0; i < n_problems; ++i)
        if (problems[i].digits || problems[i].packed || (problems[i].prepared && !problems[i].many)) return false;
    RotRowsGeom g;
    return rot_rows_geometry(base.n1, base.n2, problems[0].yhat ? 2 : 1, &g);
}

typedef void (*RotRowsKernel)(const CUtensorMap, const RotRowsParams);

static int make_x_map(CUtensorMap* xm, const RotRowsGeom& g, const void* x, int64_t M, int64_t ldx) {
    const uint64_t dims[3] = {(uint64_t)g.n2, (uint64_t)g.n1, (uint64_t)M};
    const uint64_t strides[2] = {(uint64_t)g.n2 * 2, (uint64_t)ldx * 2};
    const uint32_t box[3] = {32, (uint32_t)g.lanes, (uint32_t)g.tps};
    return make_map(xm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, x, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
}

// lr_blocks, lr_smem: of the T = V x blocks beside the rotation
static int launch_rows_kernel(RotRowsKernel k, const CUtensorMap& xm, RotRowsParams& p, int lr_blocks, size_t lr_smem, cudaStream_t stream) {
    RotRowsGeom& g = p.g;
    const int threads = rr::kControl + 128 * g.groups;
    // (a step a CTA: one x, so that blocks of the kernels before and behind find room beside these)
    if (g.xb == 2 && (p.M + g.tps - 1) / g.tps * p.n_problems + lr_blocks <= sm_count()) rot_rows_places(g, 1, 1);
    p.ctas_per_problem = rot_rows_ctas(resident_clusters((const void*)k, 1, threads, (size_t)g.total), sm_count(), p.n_problems, (p.M + g.tps - 1) / g.tps);
    if (p.ctas_per_problem < 1) return cuda_fail(cudaErrorInvalidConfiguration);
    cudaLaunchConfig_t cfg{};
    p.rot_ctas = p.n_problems * p.ctas_per_problem;
    cfg.gridDim = dim3((unsigned)(p.rot_ctas + lr_blocks), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = std::max((size_t)g.total, lr_smem);
    cfg.stream = stream;
    cudaLaunchAttribute attrs[1];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attrs[0].val.programmaticStreamSerializationAllowed = launch_overlap_allowed();
    cfg.attrs = attrs;
    cfg.numAttrs = 1;
    ProfScope prof(kProfRotateQuant, stream);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, xm, p);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}

int launch_rot_rows(const RotGeom& base, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems, const RotProblem* problems,
                    const OktLowrank* beside, uint32_t* status, cudaStream_t stream) {
    RotRowsParams p{};
    if (!rot_rows_geometry(base.n1, base.n2, problems[0].yhat ? 2 : 1, &p.g)) return BWLA_ERR_INVALID_ARG;
    const RotRowsGeom& g = p.g;
    p.M = M; p.bits = bits; p.n_problems = n_problems; p.status = status;
    for (int i = 0; i < n_problems; ++i) p.prob[i] = problems[i];
    CUtensorMap xm;
    const int st = make_x_map(&xm, g, x, M, ldx);
    if (st != BWLA_OK) return st;
    static const RotRowsKernel kernels[3][2] = {{rot_rows_kernel<kRowsSym, 1>, rot_rows_kernel<kRowsSym, 2>},
                                         {rot_rows_kernel<kRowsAsym, 1>, rot_rows_kernel<kRowsAsym, 2>},
                                         {rot_rows_kernel<kRowsBf16, 1>, rot_rows_kernel<kRowsBf16, 2>}};
    const RotRowsKernel k = kernels[problems[0].yhat ? kRowsBf16 : asym ? kRowsAsym : kRowsSym][g.chunks - 1];
    int lr_blocks = 0;
    size_t lr_smem = 0;
    for (int i = 0; i < n_problems; ++i) {
        p.lr_begin[i] = lr_blocks;
        if (!beside[i].V) continue;
        size_t bytes = 0;
        lr_blocks += plan_lowrank(p.lr[i], x, M, g.K, ldx, beside[i], (rr::kControl + 128 * g.groups) / 32, kRotMaxSmem, &bytes);
        lr_smem = std::max(lr_smem, bytes);
    }
    for (int i = n_problems; i <= kRotMaxProblems; ++i) p.lr_begin[i] = lr_blocks;
    return launch_rows_kernel(k, xm, p, lr_blocks, lr_smem, stream);
}

// Weight rows (fp32 or bf16): signs, scale and shift of each.  False in *taken: sizes or rows that rot_mma.cu has to take.
int launch_rows_binarize(const RotGeom& base, const void* w, int dtype, int64_t N, int64_t ldw, const RotProblem& problem, uint32_t* status, bool* taken,
                         cudaStream_t stream) {
    RotRowsParams p{};
    const bool f32 = dtype == BWLA_DTYPE_F32;
    *taken = (f32 || rot_accepts_x(w, ldw)) && rot_rows_binarizes(base, f32, N, sm_count()) && rot_rows_geometry(base.n1, base.n2, 0, &p.g, f32 ? 3 : 1);
    if (!*taken) return BWLA_OK;
    p.M = N; p.bits = 8; p.n_problems = 1; p.prob[0] = problem; p.status = status; p.x = w; p.ldx = ldw;
    p.x_vec = (reinterpret_cast<uintptr_t>(w) & 15) == 0 && ldw % 4 == 0;
    CUtensorMap xm{};
    if (!f32) {
        const int st = make_x_map(&xm, p.g, w, N, ldw);
        if (st != BWLA_OK) return st;
    }
    return launch_rows_kernel(f32 ? rot_rows_kernel<kRowsBinarize, 1, true> : rot_rows_kernel<kRowsBinarize, 1>, xm, p, 0, 0, stream);
}

}  // namespace bwla
