// Online OKT (Sec. 3.1) for many tokens on the tcgen05 tensor cores, with the per-token quantiser (Sec. 4.1) or the bf16
// rounding of the weight-only operating point fused in.  rot_mma.cu serves fewer tokens, every other mode and small factors, okt_umma.cu
// those between (host_plans.h has the rule).
//
//   X = reshape(x_t, n1 x n2) (row-major),   Z^T = P2^T X^T  [d][a],   Y^T = Z^T P1  [d][c]
//
// The same sums of products as in rot_mma.cu: x against the three bf16 terms of P2, then two fp16 terms of Z against two of P1 (three
// products), small products first.  Z is scaled by a power of two per row d (its largest magnitude goes to [2^14, 2^15)), which
// leaves exactly, row by row, with the scale of P1.
//
// The tensor core truncates when it adds to its accumulator, so each contraction is summed in two chains, one in each of two
// accumulators, and added with a rounded addition.  (One chain, with the accumulators of two steps in turn, took 68 us for a call of
// 64 x 80 and 4096 tokens instead of 91, but left 2.15e-7 of a row's 2-norm against 1.80e-7 of okt_umma.cu's six bf16 products and 1.50e-7
// of two chains; 160 x 160: 9.9e-7 of a token's full scale.)
//
// What bounds it: 160 x 160 takes 60 MMAs of 128 x 160 x 16 a token and CTA (80 cycles each, 80 of the 128 rows in use); what the
// ALU warps do with every value of Z and Y, in lock step and with five barriers a step, takes about twice that (2048 tokens of
// 160 x 160: 209 us; on mma.sync 505, whose operands are re-read from shared memory as fast as it delivers).
// MMAs and the work around them run side by side:
//   MMA thread    Z(0), Y(0), Z(1), Y(1), ...          Z(i) and Y(i) share the accumulators
//   16 ALU warps  step i: Y(i-1) to registers, its largest magnitude published  (accumulators free: Z(i) may start)
//                         Y(i-1) quantised and stored
//                         Z(i) to two fp16 terms in tensor memory               (Y(i) may start)
// A step is 1, 2 or 4 tokens, so that it fills up to 160 columns (64 x 128: 2 tokens).  Factors whose terms do not fit one CTA
// (or with n2 > 128) are split by rows d over a cluster of two, which share nothing but the largest magnitudes.
//
// Launched with programmatic stream serialisation: the factors are fetched before the preceding kernel of the stream has
// finished; x is read, and everything is stored, after it.  Every wait is bounded (umma_wait.cuh).
#include <cuda_bf16.h>

#include <algorithm>

#include "bwla_common.cuh"
#include "rot_mma.cuh"
#include "tensor_map.cuh"
#include "umma_ptx.cuh"
#include "umma_wait.cuh"

namespace bwla {

namespace ru {
constexpr int kAluWarps = 16;
constexpr int kThreads = 128 + 32 * kAluWarps;       // 640
// registers: 96 a thread at launch (640 x 96 = 61440); 128 x 56 + 512 x 104 = 60416 after the split (without it the two-chain
// variant keeps values in local memory: 2048 tokens of 160 x 160 236 -> 209 us)
constexpr int kRegsControl = 56, kRegsAlu = 104;
constexpr int kChunks = 5;                // 8-column chunks of a step one ALU warp owns, at most
struct Shared {
    uint64_t x_full[2], x_empty[2];       // a step's x has landed; the MMAs that read it have completed
    uint64_t z_full, y_full;              // the accumulators hold Z, Y
    uint64_t d_free;                      // ... have been read
    uint64_t a_ready;                     // the terms of Z are in tensor memory
    uint64_t row_full[2][4];              // the exponents of a lane quarter's rows are there
    uint64_t out_full[2], out_free[2];    // the step's outputs and code sums are staged; have left
    uint64_t max_full[2];                 // all warps of the token (both CTAs) have left their maxima
    uint32_t amax[2][32], vmin[2][32];    // [step parity][CTA][column part][lane quarter]
    uint8_t zexp[2][4][32][4];            // biased exponents of the rows' largest |Z|: [step parity][quarter][lane][column part]
    int qsum[2][4];                       // code sums of the step's tokens
    uint32_t tmem_slot;
    int abort_flag;
};
static_assert(sizeof(Shared) <= kRotUmmaSharedBytes, "Shared");
}  // namespace ru

struct RotUmmaParams {
    RotUmmaGeom g;
    int64_t M;
    int bits;
    int n_problems, clusters_per_problem;
    RotProblem prob[kRotMaxProblems];
    uint32_t* status;
};

namespace {
__device__ __forceinline__ void tmem_ld_32x8(uint32_t taddr, uint32_t* v) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st_32x4(uint32_t taddr, const uint32_t (&v)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
// A word into the shared memory of a CTA of the cluster, counted (4 bytes) on a barrier of that CTA.
__device__ __forceinline__ void st_async_u32(uint32_t cluster_addr, uint32_t v, uint32_t cluster_bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(cluster_addr), "r"(v), "r"(cluster_bar) : "memory");
}
__device__ __forceinline__ bool warp_wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
    for (uint32_t i = 0; i < kWaitLimit; ++i) {
        const bool done = mbar_try_wait_cluster(bar, parity, kParkNs);
        if (__all_sync(0xFFFFFFFFu, done)) return true;
        if (*abort_flag) return false;
    }
    return false;
}
// The warp's columns of the sum of both chains, whose accumulators are `other` columns apart.
template <int NC>
__device__ __forceinline__ void load_sums(uint32_t src, uint32_t other, int cw, float (&v)[NC * 8]) {
#pragma unroll
    for (int j = 0; j < NC; ++j)
        if (8 * j < cw) tmem_ld_32x8(src + 8 * j, reinterpret_cast<uint32_t*>(v) + 8 * j);
#pragma unroll
    for (int j = 0; j < NC; j += 2) {
        if (8 * j < cw) {
            const bool both = j + 1 < NC && 8 * (j + 1) < cw;
            uint32_t u[16] = {};
            tmem_ld_32x8(src + other + 8 * j, u);
            if (both) tmem_ld_32x8(src + other + 8 * (j + 1), u + 8);
            tc_wait_ld();
#pragma unroll
            for (int e = 0; e < 8; e += 2)
                add2(v[8 * j + e], v[8 * j + e + 1], __uint_as_float(u[e]), __uint_as_float(u[e + 1]));
            if (both && j + 1 < NC)
#pragma unroll
                for (int e = 0; e < 8; e += 2)
                    add2(v[8 * (j + 1 < NC ? j + 1 : j) + e], v[8 * (j + 1 < NC ? j + 1 : j) + e + 1], __uint_as_float(u[8 + e]), __uint_as_float(u[9 + e]));
        }
    }
}
}  // namespace

// MODE: the symmetric or the asymmetric quantiser, or the weight-only operating point.
enum { kSym = 0, kAsym = 1, kBf16 = 2 };
template <int MODE>
__global__ void __launch_bounds__(ru::kThreads, 1)
rot_umma_kernel(const __grid_constant__ CUtensorMap x_map, const __grid_constant__ RotUmmaParams p) {
    extern __shared__ __align__(1024) uint8_t smem[];
    constexpr int NC = ru::kChunks;
    const RotUmmaGeom& g = p.g;
    ru::Shared& sh = *reinterpret_cast<ru::Shared*>(smem + g.sh_off);
    volatile int* abort_flag = &sh.abort_flag;
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const int rank = g.dc > 1 ? (int)cluster_ctarank() : 0;
    const int cl = (int)blockIdx.x / g.dc;
    const int prob_i = cl / p.clusters_per_problem;
    const RotProblem& pr = p.prob[prob_i];
    const int64_t first = cl - (int64_t)prob_i * p.clusters_per_problem;      // steps first, first + clusters, ...
    const int64_t steps_all = (p.M + g.tps - 1) / g.tps;
    int n = first < steps_all ? (int)((steps_all - first + p.clusters_per_problem - 1) / p.clusters_per_problem) : 0;
    const int rows = min(g.dt, g.n2 - rank * g.dt);

    // ---- the layer's factors (they do not depend on the preceding kernel): rows of 64 bytes, swizzled ----
    int e1;
    if (pr.prepared) {
        const uint8_t* t2 = pr.prepared + kRotHeader;
        const size_t all2 = (size_t)g.n2 * g.s2;
        const uint8_t* t1 = t2 + 3 * all2;
        e1 = __ldg(reinterpret_cast<const int*>(pr.prepared) + 1);
        const int cpr2 = g.n2 >> 3;
        for (int i = threadIdx.x; i < 3 * rows * cpr2; i += ru::kThreads) {
            const int rr = i / cpr2, ch = i - rr * cpr2, term = rr / rows, r = rr - term * rows;
            uint8_t* dst = smem + ((term * g.atoms2 + (ch >> 2)) * g.dt + r) * 64 + (((ch ^ (r >> 1)) & 3) << 4);
            cp_async16(smem_u32(dst), t2 + term * all2 + (size_t)(rank * g.dt + r) * g.s2 + 16 * ch);
        }
        const int cpr1 = g.nc >> 3;
        for (int i = threadIdx.x; i < 2 * g.nc * cpr1; i += ru::kThreads) {
            const int rr = i / cpr1, ch = i - rr * cpr1, term = rr / g.nc, r = rr - term * g.nc;
            uint8_t* dst = smem + g.p1_off + ((term * g.atoms1 + (ch >> 2)) * g.nc + r) * 64 + (((ch ^ (r >> 1)) & 3) << 4);
            cp_async16(smem_u32(dst), t1 + (size_t)term * g.nc * g.s1 + (size_t)r * g.s1 + 16 * ch);
        }
    }
    else {
        e1 = factor_exponent(block_absmax(pr.P1, g.n1 * g.n1, sh.amax[0]));
        split_factor<false>(pr.P2, g.n2, rank * g.dt, rows, g.n2, 1.f, [&](int r, int k2) {
            return smem + ((k2 >> 4) * g.dt + r) * 64 + ((((k2 >> 2) ^ (r >> 1)) & 3) << 4) + 4 * (k2 & 3);
        }, (size_t)g.atoms2 * g.dt * 64, threadIdx.x, ru::kThreads);
        split_factor<true>(pr.P1, g.n1, 0, g.nc, g.nc, pow2f(e1), [&](int r, int k2) {
            return smem + g.p1_off + ((k2 >> 4) * g.nc + r) * 64 + ((((k2 >> 2) ^ (r >> 1)) & 3) << 4) + 4 * (k2 & 3);
        }, (size_t)g.atoms1 * g.nc * 64, threadIdx.x, ru::kThreads);
    }
    if (threadIdx.x == 0) {
        sh.abort_flag = 0;
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.x_full[i], 1); mbar_init(&sh.x_empty[i], 1);
            mbar_init(&sh.max_full[i], g.dc == 1 ? ru::kAluWarps : 1);
            mbar_init(&sh.out_full[i], ru::kAluWarps); mbar_init(&sh.out_free[i], 1);
            for (int j = 0; j < 4; ++j) { sh.qsum[i][j] = 0; mbar_init(&sh.row_full[i][j], 4); }
        }
        mbar_init(&sh.z_full, 1); mbar_init(&sh.y_full, 1);
        mbar_init(&sh.d_free, ru::kAluWarps); mbar_init(&sh.a_ready, ru::kAluWarps);
        fence_barrier_init();
    }
    if (warp == 2) {
        tmem_alloc(&sh.tmem_slot, 512);
        tmem_relinquish();
    }
    cp_async_wait_all();
    fence_proxy_async();
    tc_fence_before();
    __syncthreads();
    if (g.dc > 1) { cluster_arrive_release(); cluster_wait_acquire(); }       // the other CTA's barriers stand
    tc_fence_after();
    const uint32_t tmem = *reinterpret_cast<volatile uint32_t*>(&sh.tmem_slot);
    griddep_launch_dependents();
    griddep_wait();                                   // x may be the output of the preceding kernel
    if (p.status && *reinterpret_cast<volatile uint32_t*>(p.status) != 0) n = 0;      // the call already failed

    // phase of step i's accumulators
    auto phase_of = [](int i) { return (uint32_t)(i & 1); };
    if (warp < 4) {
    set_regs_dec<ru::kRegsControl>();
    if (warp == 0) {
        // ---------------- x ----------------
        if (elect_one()) {
            tma_prefetch_desc(&x_map);
            const int atom_bytes = g.ntot * 64;
            for (int i = 0; i < n; ++i) {
                const int b = g.xb == 2 ? i & 1 : 0;
                const uint32_t use = (uint32_t)(g.xb == 2 ? i >> 1 : i);
                if (!wait_or_abort(&sh.x_empty[b], (use & 1u) ^ 1u, abort_flag)) { give_up(p.status, abort_flag, 0x210); break; }
                const int t0 = (int)((first + (int64_t)i * p.clusters_per_problem) * g.tps);
                uint8_t* dst = smem + g.x_off + b * g.atoms2 * atom_bytes;
                mbar_expect_tx(&sh.x_full[b], (uint32_t)(g.atoms2 * atom_bytes));
                for (int a = 0; a < g.atoms2; ++a) tma_load_3d(dst + a * atom_bytes, &x_map, 32 * a, 0, t0, &sh.x_full[b]);
            }
            if (*abort_flag) for (int i = 0; i < 500; ++i) __nanosleep(100);
        }
    } else if (warp == 1) {
        // ---------------- MMAs (all lanes in step: see umma_ptx.cuh) ----------------
        const bool one = elect_one();
        const uint32_t idesc_a = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(g.ntot >> 3) << 17) | ((128u >> 4) << 24);
        const uint32_t idesc_c = (1u << 4) | ((uint32_t)(g.nc >> 3) << 17) | ((128u >> 4) << 24);
        const uint64_t d_p2 = smem_desc_kmajor(smem_u32(smem), 64), d_p1 = smem_desc_kmajor(smem_u32(smem + g.p1_off), 64);
        const uint64_t d_x = smem_desc_kmajor(smem_u32(smem + g.x_off), 64);
        const uint32_t desc_hi = (uint32_t)(d_p2 >> 32);                      // (the same for all three)
        const uint32_t blk2 = (uint32_t)(g.dt * 64) >> 4, blkx = (uint32_t)(g.ntot * 64) >> 4, blk1 = (uint32_t)(g.nc * 64) >> 4;
        const int ks2 = g.n2 >> 4, ks1 = g.nc >> 4, half2 = (ks2 + 1) >> 1, half1 = (ks1 + 1) >> 1;
        for (int i = 0; i < n; ++i) {
            const int b = g.xb == 2 ? i & 1 : 0;
            const uint32_t use = (uint32_t)(g.xb == 2 ? i >> 1 : i);
            if (!warp_wait(&sh.x_full[b], use & 1u, abort_flag)) { give_up(p.status, abort_flag, 0x220); break; }
            if (i >= 1 && !warp_wait(&sh.d_free, phase_of(i) ^ 1u, abort_flag)) { give_up(p.status, abort_flag, 0x221); break; }
            tc_fence_after();
            const uint32_t x0 = (uint32_t)d_x + (uint32_t)(b * g.atoms2) * blkx;
#pragma unroll 1
            for (int term = 2; term >= 0; --term) {
                uint32_t at = (uint32_t)d_p2 + (uint32_t)(term * g.atoms2) * blk2, bt = x0;
#pragma unroll 2
                for (int k = 0; k < ks2; ++k) {
                    warp_mma_f16_ss(one, k >= half2 ? tmem + (uint32_t)g.ntot : tmem, at, desc_hi, bt, desc_hi, idesc_a, (term == 2 && (k == 0 || k == half2)) ? 0u : 1u);
                    at += k & 1 ? blk2 - 2u : 2u;
                    bt += k & 1 ? blkx - 2u : 2u;
                }
            }
            warp_commit(one, &sh.x_empty[b]);
            warp_commit(one, &sh.z_full);
            if (!warp_wait(&sh.a_ready, (uint32_t)(i & 1), abort_flag)) { give_up(p.status, abort_flag, 0x222); break; }
            tc_fence_after();
            for (int tk = 0; tk < g.tps; ++tk) {
                const uint32_t a = tmem + (uint32_t)(2 * g.ntot + tk * (g.np >> 1)), y = tmem + (uint32_t)(tk * g.np);
                // lo hi, hi lo, hi hi
#pragma unroll 1
                for (int q = 0; q < 3; ++q) {
                    uint32_t at = a + (q == 0 ? (uint32_t)(g.ntot >> 1) : 0u), bt = (uint32_t)d_p1 + (q == 1 ? (uint32_t)g.atoms1 * blk1 : 0u);
#pragma unroll 2
                    for (int k = 0; k < ks1; ++k) {
                        warp_mma_f16_ts(one, k >= half1 ? y + (uint32_t)g.ntot : y, at, bt, desc_hi, idesc_c, (q == 0 && (k == 0 || k == half1)) ? 0u : 1u);
                        at += 8u;
                        bt += k & 1 ? blk1 - 2u : 2u;
                    }
                }
            }
            warp_commit(one, &sh.y_full);
        }
    } else if (warp == 3) {
        // ---------------- code sums and staged outputs of a step ----------------
        for (int i = 0; i < n; ++i) {
            const int par = i & 1;
            if (!warp_wait(&sh.out_full[par], (uint32_t)((i >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x240); break; }
            const int64_t t0 = (first + (int64_t)i * p.clusters_per_problem) * g.tps;
            const int tokens = (int)min((int64_t)g.tps, p.M - t0);
            if (g.staged && lane == 0) {
                const int size = g.out_bytes / g.tps;
                uint8_t* dst = MODE == kBf16 ? reinterpret_cast<uint8_t*>(pr.yhat) : reinterpret_cast<uint8_t*>(pr.codes);
                bulk_s2g(dst + t0 * size, smem + g.st_off + par * g.out_bytes, (uint32_t)(tokens * size));
            }
            if (MODE != kBf16 && pr.qsum) {
                // every CTA of the cluster leaves its own part of the sum; the consumer adds the parts
                const int tk = lane >> 3, part = lane & 7;
                static_assert(kQsumParts == 8, "a lane per part");
                const int sum = sh.qsum[par][tk];
                __syncwarp();
                if (part == 0) sh.qsum[par][tk] = 0;
                if (tk < tokens && (part == rank || (rank == 0 && part >= g.dc))) pr.qsum[(t0 + tk) * kQsumParts + part] = part == rank ? sum : 0;
            }
            if (g.staged && lane == 0) bulk_wait_read();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.out_free[par]);
        }
        if (g.staged && lane == 0) bulk_wait_all();
    }
    } else {
        set_regs_inc<ru::kRegsAlu>();
        // ---------------- everything between and behind the MMAs ----------------
        // A warp issues an instruction about every six cycles here (four warps a scheduler), so instructions a value are what
        // counts: no scaling pass over Y (a row's power of two goes into the quantiser's factor), one read of Z, no
        // conditions on single values where whole chunks exist, two columns a store.
        const int w = warp - 4, q = w & 3, wc = w >> 2;
        const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
        const int cw = g.ntot >> 2;                   // columns of the step this warp owns
        const int tk = wc * g.tps >> 2;               // their token
        const int c_base = wc * cw - tk * g.np;       // first of them within the token
        const bool some = q * 32 < rows, valid = q * 32 + lane < rows;        // (16 lanes at a time)
        const int d = rank * g.dt + q * 32 + lane;
        const int parts = 4 / g.tps;                  // warps of a token in a lane quarter
        const int have = some ? min(cw, g.nc - c_base) : 0;                   // columns that hold sums (a multiple of 8), and
        const int exist = some ? min(cw, g.n1 - c_base) : 0;                  // that are outputs (either may be negative)
        float f1 = 1.f;                               // power of two that brings this lane's row of y to true scale
        int z_exp = 0;
        bool ok = true;
#pragma unroll 1
        for (int i = 0; i <= n && ok; ++i) {
            const int pi = (i - 1) & 1;
            const int64_t t = (first + (int64_t)(i - 1) * p.clusters_per_problem) * g.tps + tk;
            float amax = 0.f, vmin = 0.f;
            float y[NC * 8];
            if (i > 0) {
                // ---- Y of the step before to registers; its extremes to the token's other warps
                if (!warp_wait(&sh.y_full, phase_of(i - 1), abort_flag)) { give_up(p.status, abort_flag, 0x230); ok = false; break; }
                tc_fence_after();
                const uint32_t src = tmem + lane_addr + (uint32_t)(wc * cw);
                if (some) load_sums<NC>(src, (uint32_t)g.ntot, cw, y);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.d_free);
                const int ey = -(z_exp + e1), ey1 = max(-126, min(127, ey)), ey2 = max(-126, min(127, ey - ey1));
                f1 = pow2f(ey1);
                if (__any_sync(0xFFFFFFFFu, ey2 != 0)) {          // scales at the ends of fp32's range
                    const float f2 = pow2f(ey2);
#pragma unroll
                    for (int j = 0; j < NC * 8; ++j) y[j] = y[j] * f1 * f2;
                    f1 = 1.f;
                }
                auto publish = [&](uint32_t m, uint32_t v) {
                    uint32_t* slot = &sh.amax[pi][rank * 16 + w];
                    uint32_t* slot_v = &sh.vmin[pi][rank * 16 + w];
                    if (g.dc == 1) {
                        if (lane == 0) { *slot = m; *slot_v = v; mbar_arrive(&sh.max_full[pi]); }
                    } else {
                        // (asynchronous stores that count on the barrier: an arrival with release at cluster scope waits for this
                        // warp's codes of the step before to reach global memory, about 1000 cycles)
                        constexpr uint32_t each = MODE == kSym ? 4u : 8u;
                        if (w == 0 && lane == 0) mbar_expect_tx(&sh.max_full[pi], 2u * ru::kAluWarps * each);
                        if (lane < 2) {
                            const uint32_t bar = map_shared_rank(smem_u32(&sh.max_full[pi]), (uint32_t)lane);
                            st_async_u32(map_shared_rank(smem_u32(slot), (uint32_t)lane), m, bar);
                            if (MODE != kSym) st_async_u32(map_shared_rank(smem_u32(slot_v), (uint32_t)lane), v, bar);
                        }
                    }
                };
                if (MODE == kBf16) {
                    if (pr.ysum) {
                        // the sum of the rounded values goes where the quantiser's two extremes go
                        double s = 0.0;
#pragma unroll
                        for (int j = 0; j < NC; ++j)
                            if (valid && 8 * j < have)
#pragma unroll
                                for (int e = 0; e < 8; ++e) s += (double)__bfloat162float(__float2bfloat16_rn(y[8 * j + e] * f1));
                        s = warp_sum(s);
                        publish((uint32_t)__double2loint(s), (uint32_t)__double2hiint(s));
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < NC; ++j)
                        if (8 * j < have)
#pragma unroll
                            for (int e = 0; e < 8; e += 2) {
                                const float a = y[8 * j + e], b = y[8 * j + e + 1];
                                if (MODE == kSym) amax = fmaxf(amax, fmaxf(fabsf(a), fabsf(b)));
                                else { amax = fmaxf(amax, fmaxf(a, b)); vmin = fminf(vmin, fminf(a, b)); }
                            }
                    if (!valid) amax = vmin = 0.f;                // (rows beyond P2's hold anything)
                    // non-negative (NaNs aside), so their bit patterns order like the values
                    publish(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(amax * f1)),
                            MODE == kAsym ? __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(fmaxf(-vmin * f1, 0.f))) : 0u);
                }
            }
            auto convert = [&]() -> bool {
                // ---- Z of this step: the power of two of every row, then its two fp16 terms, in place of the step before's (whose
                // MMAs have completed: this warp has seen Y above)
                const int zi = i & 1;
                if (!warp_wait(&sh.z_full, phase_of(i), abort_flag)) { give_up(p.status, abort_flag, 0x231); return false; }
                tc_fence_after();
                const uint32_t src = tmem + lane_addr + (uint32_t)(wc * cw);
                // (read twice, two chunks at a time: with all of Z in registers over the exchange they do not suffice)
                float z[16];
                auto load_two = [&](int j) { load_sums<2>(src + 8 * j, (uint32_t)g.ntot, cw - 8 * j, z); };
                if (some) {
                    float m = 0.f;
#pragma unroll
                    for (int j = 0; j < NC; j += 2) {
                        load_two(j);
#pragma unroll
                        for (int e = 0; e < 16; e += 2)
                            if (8 * j + e < cw) m = fmaxf(m, fmaxf(fabsf(z[e]), fabsf(z[e + 1])));
                    }
                    sh.zexp[zi][q][lane][wc] = (uint8_t)(__float_as_uint(m) >> 23);
                }
                __syncwarp();
                if (parts > 1) {
                    if (lane == 0) mbar_arrive(&sh.row_full[zi][q]);
                    if (!warp_wait(&sh.row_full[zi][q], (uint32_t)((i >> 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x233); return false; }
                }
                if (some) {
                    const uint32_t ex4 = *reinterpret_cast<const volatile uint32_t*>(&sh.zexp[zi][q][lane][0]);
                    uint32_t ex = 0u;
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if ((j * g.tps >> 2) == tk) ex = max(ex, (ex4 >> (8 * j)) & 0xFFu);
                    z_exp = max(-126, min(126, 14 + 127 - (int)ex));
                    const float z_scale = pow2f(z_exp);
                    const uint32_t dst = tmem + lane_addr + (uint32_t)(2 * g.ntot + (wc * cw >> 1));
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        if (j % 2 == 0) load_two(j);
                        if (8 * j < cw) {
                            uint32_t h[4], l[4];
                            const int at = 8 * (j & 1);
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                mul2(z[at + 2 * e], z[at + 2 * e + 1], z_scale);
                                split2_pair(z[at + 2 * e], z[at + 2 * e + 1], h[e], l[e]);
                            }
                            tmem_st_32x4(dst + 4 * j, h);
                            tmem_st_32x4(dst + (uint32_t)(g.ntot >> 1) + 4 * j, l);
                        }
                    }
                    tc_wait_st();
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.a_ready);
                return true;
            };
            // ---- the step before: codes, scale and code sum, or bf16 values
            auto finish = [&]() -> bool {
                if (i >= 3 && !warp_wait(&sh.out_free[pi], (uint32_t)((((i - 1) >> 1) - 1) & 1), abort_flag)) { give_up(p.status, abort_flag, 0x234); return false; }
                uint8_t* const stage = smem + g.st_off + pi * g.out_bytes + tk * (g.out_bytes / g.tps);
                if (MODE == kBf16) {
                    if (t < p.M && valid) {
                        // layout 1: inside each group of 32, position 2 (k % 16) + (k % 32) / 16; every other column has the same
                        // place in its group (2 n2 is a multiple of 32)
                        __nv_bfloat16* yt = g.staged ? reinterpret_cast<__nv_bfloat16*>(stage) : pr.yhat + t * (int64_t)g.K;
                        const int k0 = c_base * g.n2 + d, k1 = k0 + g.n2;
                        __nv_bfloat16* at0 = yt + (pr.codes_layout ? (k0 & ~31) + 2 * (k0 & 15) + ((k0 >> 4) & 1) : k0);
                        __nv_bfloat16* at1 = yt + (pr.codes_layout ? (k1 & ~31) + 2 * (k1 & 15) + ((k1 >> 4) & 1) : k1);
                        const int step = 2 * g.n2;
                        if (exist == NC * 8) {
#pragma unroll
                            for (int j = 0; j < NC * 8; j += 2) {
                                *at0 = __float2bfloat16_rn(y[j] * f1); *at1 = __float2bfloat16_rn(y[j + 1] * f1);
                                at0 += step; at1 += step;
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < NC * 8; j += 2) {
                                if (j < exist) *at0 = __float2bfloat16_rn(y[j] * f1);
                                if (j + 1 < exist) *at1 = __float2bfloat16_rn(y[j + 1] * f1);
                                at0 += step; at1 += step;
                            }
                        }
                    }
                    if (!pr.ysum) return true;
                }
                if (g.dc == 1 ? !warp_wait(&sh.max_full[pi], (uint32_t)(((i - 1) >> 1) & 1), abort_flag)
                              : !warp_wait_cluster(&sh.max_full[pi], (uint32_t)(((i - 1) >> 1) & 1), abort_flag)) {
                    give_up(p.status, abort_flag, 0x232); return false;
                }
                const bool mine = lane < 16 * g.dc && (((lane & 15) >> 2) * g.tps >> 2) == tk;
                const bool writer = rank == 0 && q == 0 && c_base == 0;       // of the token's scalars
                const uint32_t s0 = mine ? *reinterpret_cast<volatile uint32_t*>(&sh.amax[pi][lane]) : 0u;
                const uint32_t s1 = mine && MODE != kSym ? *reinterpret_cast<volatile uint32_t*>(&sh.vmin[pi][lane]) : 0u;
                if (t >= p.M) return true;
                if (MODE == kBf16) {
                    if (writer) {
                        const double s = warp_sum(__hiloint2double((int)s1, (int)s0));
                        if (lane == 0) pr.ysum[t] = (float)s;
                    }
                    return true;
                }
                amax = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, s0));
                if (MODE == kAsym) vmin = -__uint_as_float(__reduce_max_sync(0xFFFFFFFFu, s1));
                // The quantiser of rot_mma.cu with the same roundings: fl(v + 1.5 * 2^23 + shift) leaves rne(v) + shift in the low
                // mantissa bits, the low byte is stored, the patterns are summed.
                const float levels = MODE == kSym ? (float)((1 << (p.bits - 1)) - 1) : (float)((1 << p.bits) - 1);
                const float range = MODE == kSym ? amax : __fsub_rn(amax, vmin);
                const float inv = range != 0.f ? __fdiv_rn(levels, range) : 0.f;
                float zero_f = 0.f, half_f = 0.f;
                if (MODE == kAsym) {
                    const float tz = __fmul_rn(-vmin, inv);
                    zero_f = fminf(fmaxf(__fadd_rn(__fadd_rn(tz, 12582912.f), -12582912.f), 0.f), levels);
                    half_f = (float)(1 << (p.bits - 1));
                }
                const float store_shift = (float)pr.code_bias - half_f;
                const int shift_i = (int)(zero_f + store_shift);
                const uint32_t odd = (uint32_t)(shift_i & 1);
                const float bias_even = 12582912.f + (float)(shift_i - (int)odd);
                const float lo_b = 12582912.f + store_shift - (float)odd, hi_b = lo_b + levels;
                if (writer && lane == 0) {
                    pr.scales[t] = range != 0.f ? __fdiv_rn(range, levels) : 1.f;
                    if (pr.zp) pr.zp[t] = shift_i;
                }
                if (pr.y && valid) {
#pragma unroll
                    for (int j = 0; j < NC * 8; ++j)
                        if (j < exist) pr.y[t * (int64_t)g.K + (c_base + j) * g.n2 + d] = y[j] * f1;
                }
                // fl(y inv) = fl(y_row_scaled (f inv)): f is a power of two, and where f inv leaves fp32's normal range the row is too
                // small against the token's largest value for any code but zero
                const float f_inv = inv * f1;
                int code_sum = 0;                                 // of the stored codes less their bias
                const int whole = pr.codes_layout ? max(exist, 0) & ~7 : 0;
                if (whole > 0) {
                    // The usual case: whole chunks of outputs, in the contraction's order.  Four codes of a lane make a
                    // word by multiply-adds, every code shifted to c + 128 >= 0 (the bits of 1.5 * 2^23 below bit 16 are zero, so
                    // nothing carries from one byte into the next).  Lanes 8 apart have neighbouring bytes of a column: they swap
                    // words, and one of the two stores both lanes' codes of the first two columns, the other of the last two.
                    // (Conditions a column, selects and packing one by one took 31 half-rate instructions for four columns, 250
                    // cycles a scheduler.)
                    const int hb = (lane >> 3) & 1;
                    const uint32_t sel = hb ? 0x3726u : 0x5140u;
                    const int k0 = (c_base + 2 * hb) * g.n2 + (d & ~8), k1 = k0 + g.n2;
                    const int off0 = (k0 & ~31) + 4 * (k0 & 7) + ((k0 & 31) >> 3), off1 = (k1 & ~31) + 4 * (k1 & 7) + ((k1 & 31) >> 3);
                    const float b = bias_even + 128.f, lo = lo_b + 128.f, hi = hi_b + 128.f;
                    // w0 + 2^8 w1 has 0x8B40 above its two bytes; that of the lower pair is taken off the upper one
                    const uint32_t top = MODE == kAsym ? 0x74C00000u + 0x01010101u * odd : 0x74C00000u;
                    uint32_t sum = 0u;
                    auto all = [&](auto store) {
#pragma unroll
                        for (int j = 0; j < NC * 8; j += 4) {
                            if ((j & ~7) >= whole) break;
                            float v[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) v[e] = __fmul_rn(y[j + e], f_inv);
                            add2(v[0], v[1], b, b);
                            add2(v[2], v[3], b, b);
                            if (MODE == kAsym)
#pragma unroll
                                for (int e = 0; e < 4; ++e) v[e] = fminf(fmaxf(v[e], lo), hi);
                            const uint32_t p01 = __float_as_uint(v[1]) * 256u + __float_as_uint(v[0]);
                            const uint32_t p23 = __float_as_uint(v[3]) * 256u + __float_as_uint(v[2]);
                            const uint32_t word = p23 * 65536u + (p01 + top);
                            sum = __dp4a(word, 0x01010101u, sum);
                            const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, word, 8);
                            const uint32_t both = __byte_perm(word, other, sel) ^ 0x80808080u;
                            store(j, both);
                        }
                    };
                    if (g.staged) {
                        uint32_t at0 = smem_u32(stage) + off0, at1 = smem_u32(stage) + off1;
                        const uint32_t step = 4 * g.n2;
                        all([&](int, uint32_t both) {
                            if (valid) { st_shared_u16(at0, both); st_shared_u16(at1, both >> 16); }
                            at0 += step; at1 += step;
                        });
                    } else {
                        int8_t* at0 = pr.codes + t * (int64_t)g.K + off0;
                        const int delta = off1 - off0, step = 4 * g.n2;
                        all([&](int, uint32_t both) {
                            if (valid) { *reinterpret_cast<uint16_t*>(at0) = (uint16_t)both; *reinterpret_cast<uint16_t*>(at0 + delta) = (uint16_t)(both >> 16); }
                            at0 += step;
                        });
                    }
                    code_sum = (int)sum - whole * (128 + pr.code_bias);
                }
                if (whole < exist) {
                    int8_t* const ct = g.staged ? reinterpret_cast<int8_t*>(stage) : pr.codes + t * (int64_t)g.K;
#pragma unroll
                    for (int j = 0; j < NC * 8; ++j) {
                        if (j >= whole && j < exist) {
                            const float v = __fadd_rn(__fmul_rn(y[j], f_inv), bias_even);
                            uint32_t word = __float_as_uint(v);
                            if (MODE == kAsym) word = __float_as_uint(fminf(fmaxf(v, lo_b), hi_b)) + odd;
                            code_sum += (int)(word - (0x4B400000u + (uint32_t)pr.code_bias));
                            const int k = (c_base + j) * g.n2 + d;
                            if (valid) ct[pr.codes_layout ? (k & ~31) + 4 * (k & 7) + ((k & 31) >> 3) : k] = (int8_t)word;
                        }
                    }
                }
                if (pr.qsum) {
                    const int local = __reduce_add_sync(0xFFFFFFFFu, valid ? code_sum : 0);
                    if (lane == 0 && local != 0) atomicAdd(&sh.qsum[pi][tk], local);
                }
                return true;
            };
            if (i > 0) {
                if (!finish()) { ok = false; break; }
                if (g.staged) fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.out_full[pi]);
            }
            if (i < n && !convert()) { ok = false; break; }
        }
        if (!ok) *abort_flag = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 512);
    }
    // nobody leaves while the other CTA may still store into its shared memory
    if (g.dc > 1) { cluster_arrive_release(); cluster_wait_acquire(); }
}

typedef void (*Kernel)(const CUtensorMap, const RotUmmaParams);
bool rot_umma_supports(const RotGeom& base, int n_problems, const RotProblem* problems) {
    if (rot_mma_always(base)) return false;
    for (int i = 0; i < n_problems; ++i)
        if (problems[i].digits || problems[i].packed) return false;
    RotUmmaGeom u;
    return rot_umma_geometry(base, problems[0].yhat ? 2 : 1, &u);
}

int launch_rot_umma(const RotGeom& base, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems,
                    const RotProblem* problems, uint32_t* status, cudaStream_t stream) {
    RotUmmaParams p{};
    if (!rot_umma_geometry(base, problems[0].yhat ? 2 : 1, &p.g)) return BWLA_ERR_INVALID_ARG;
    const RotUmmaGeom& g = p.g;
    p.M = M; p.bits = bits; p.n_problems = n_problems; p.status = status;
    for (int i = 0; i < n_problems; ++i) p.prob[i] = problems[i];
    CUtensorMap xm;
    {
        const uint64_t dims[3] = {(uint64_t)g.n2, (uint64_t)g.n1, (uint64_t)M};
        const uint64_t strides[2] = {(uint64_t)g.n2 * 2, (uint64_t)ldx * 2};
        const uint32_t box[3] = {32, (uint32_t)g.np, (uint32_t)g.tps};
        const int st = make_map(&xm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, x, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_64B,
                                CU_TENSOR_MAP_L2_PROMOTION_L2_128B);
        if (st != BWLA_OK) return st;
    }
    const int mode = problems[0].yhat ? kBf16 : asym ? kAsym : kSym;
    const Kernel k = mode == kSym ? rot_umma_kernel<kSym> : mode == kAsym ? rot_umma_kernel<kAsym> : rot_umma_kernel<kBf16>;
    const int room = resident_clusters((const void*)k, g.dc, ru::kThreads, (size_t)g.total) / n_problems;
    if (room < 1) return cuda_fail(cudaErrorInvalidConfiguration);
    p.clusters_per_problem = (int)std::min<int64_t>((M + g.tps - 1) / g.tps, room);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(n_problems * p.clusters_per_problem * g.dc), 1, 1);
    cfg.blockDim = dim3(ru::kThreads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)g.total;
    cfg.stream = stream;
    cudaLaunchAttribute attrs[2];
    attrs[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    // clusters that stay are placed on an empty device (see rot_mma.cu)
    attrs[0].val.programmaticStreamSerializationAllowed = g.dc > 1 ? 0u : launch_overlap_allowed();
    attrs[1].id = cudaLaunchAttributeClusterDimension;
    attrs[1].val.clusterDim.x = (unsigned)g.dc; attrs[1].val.clusterDim.y = 1; attrs[1].val.clusterDim.z = 1;
    cfg.attrs = attrs;
    cfg.numAttrs = g.dc > 1 ? 2 : 1;
    ProfScope prof(kProfRotateQuant, stream);
    const cudaError_t e = cudaLaunchKernelEx(&cfg, k, xm, p);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e); }
    return after_launch();
}

}  // namespace bwla
