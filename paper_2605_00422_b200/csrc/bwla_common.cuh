// Shared declarations of the CUDA library: status handling, workspace layout, kernel launchers.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <algorithm>

#include "bwla.h"
#include "host_plans.h"

namespace bwla {

// ---------------------------------------------------------------------------------------------
// per-thread bookkeeping (the library keeps no process-global mutable state)
// ---------------------------------------------------------------------------------------------
extern thread_local int g_last_cuda_error;
extern thread_local int g_launch_count;

inline int cuda_fail(cudaError_t e) {
    g_last_cuda_error = (int)e;
    return BWLA_ERR_CUDA;
}

#define BWLA_CUDA_TRY(expr)                                   \
    do {                                                      \
        cudaError_t e__ = (expr);                             \
        if (e__ != cudaSuccess) return ::bwla::cuda_fail(e__); \
    } while (0)

// Checks the launch that has just been issued and counts it.
inline int after_launch() {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e);
    ++g_launch_count;
    return BWLA_OK;
}

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Number of SMs of the current device (cached per thread and device); 0 if it cannot be queried.
inline int sm_count() {
    static thread_local int cached_dev = -1, cached_n = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    if (dev != cached_dev) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { cudaGetLastError(); return 0; }
        cached_dev = dev; cached_n = n;
    }
    return cached_n;
}

// ---------------------------------------------------------------------------------------------
// optional per-kernel timing (bwla_profile_enable / bwla_profile_collect): CUDA events recorded on the launching
// stream right around each kernel launch, summed per kernel kind.  Off by default; not usable under stream capture.
// ---------------------------------------------------------------------------------------------
enum ProfKind { kProfRotateQuant = 0, kProfContraction = 2, kProfPrepare = 4,
                kProfPack = 5, kProfKinds = 8 };
// 1 unless per-kernel timing is on: timed kernels are launched fully serialised so that each event pair brackets
// one kernel alone.
unsigned launch_overlap_allowed();
void prof_begin(int kind, cudaStream_t stream);
void prof_end(int kind, cudaStream_t stream);
struct ProfScope {
    int kind; cudaStream_t stream;
    ProfScope(int k, cudaStream_t s) : kind(k), stream(s) { prof_begin(kind, stream); }
    ~ProfScope() { prof_end(kind, stream); }
};

// ---------------------------------------------------------------------------------------------
// workspace layout (byte offsets into the caller's scratch buffer; every section 256-byte aligned)
// ---------------------------------------------------------------------------------------------
constexpr int kStatusBytes = 256;        // word 0: status; words 1..: where a bounded wait gave up
// The code sum of a token is kept as kQsumParts partial sums (host_plans.h; one per CTA of the prologue cluster that quantised a slab
// of the token; unused parts are zero): the consumer adds them, the producers need no exchange.

constexpr int kLrCounterWord = 4;        // first of the arrival counters of split tiles of T among the status words

// T = V x for many tokens on the tensor cores (lowrank_umma.cu), for the problems of one group (all share x, M, K; every entry of
// `lowrank` has V, Thl and, where partial sums are needed, umma_part set).
struct OktLowrank;
bool lowrank_umma_takes(const void* x, int64_t M, int64_t K, int64_t ldx, const OktLowrank& lowrank);
int launch_lowrank_umma(const void* x, int64_t M, int64_t K, int64_t ldx, int n_problems, const OktLowrank* lowrank,
                        uint32_t* status, cudaStream_t stream);

struct Workspace {
    size_t status, scales, zp, qsum, T, lr_part, codes, total;
};

inline Workspace workspace_layout(int64_t M, int64_t K, int64_t N, int r, int bits) {
    Workspace w{};
    size_t off = 0;
    w.status = off; off += kStatusBytes;
    w.scales = off; off += align_up((size_t)M * 4, 256);
    w.zp = off;     off += align_up((size_t)M * 4, 256);        // per-token zero points (asymmetric activations)
    w.qsum = off;   off += align_up((size_t)M * 4 * kQsumParts, 256);
    const size_t lr_cols = (size_t)lowrank_cols(r);
    w.T = off;      off += align_up((size_t)M * lr_cols * 6, 256);     // bf16 [3][M][cols]
    w.lr_part = off; off += r > 0 ? lowrank_split_bytes(M, lowrank_cols(r)) : 0;
    // (the tcgen05 kernel for T leaves its partial sums where the rotation behind it puts the codes)
    w.codes = off;  off += align_up((size_t)M * (size_t)K, 256);
    (void)N; (void)bits;
    w.total = off;
    return w;
}

// Argument checks of bwla_w1ax_linear (everything that can be refused without touching the GPU, then the device check).
// BWLA_OK also for the empty problems M == 0 / N == 0, which the caller turns into a no-op.
int validate_linear_call(const void* x_bf16, int64_t M, int64_t K, int64_t ldx, const float* P1, int n1, const float* P2,
                         int n2, int bits, const uint32_t* packed, const float* alpha, const void* U_bf16,
                         const void* V_bf16, int r, const void* out_bf16, int64_t N, int64_t ldo, const void* workspace,
                         size_t workspace_bytes);

// ---------------------------------------------------------------------------------------------
// kernel launchers (each returns a BWLA status; all asynchronous on `stream`)
// ---------------------------------------------------------------------------------------------
int launch_pack_signs(const void* w, int dtype, int64_t N, int64_t K, int64_t ldw, uint32_t* packed,
                      cudaStream_t stream);
// rowsum[n] = sum_k sign(n,k) = 2 * popc(row n) - K
int launch_row_sums(const uint32_t* packed, int64_t N, int64_t K, int32_t* rowsum, cudaStream_t stream);

// One launch: fused rotate + absmax + quantise (skipped when codes == NULL) and T = V x (skipped when r == 0 or
// Thl == NULL).  codes_layout: 0 = natural k order, 1 = interleaved order used by the tensor-core contraction (inside
// each group of 32, position 4*j + i holds k = j + 8*i).  qsum (int32 [M][kQsumParts], partial sums) may be NULL.
// Thl: bf16 [3][M][cols], cols = lowrank_cols(r): T as the sum of three bf16 terms (exact for an fp32 T).
// lr_part / status (both may be NULL): scratch for the partial sums of T and the workspace status words (see kLrKSplitMax).
int launch_prologue(const void* x, int64_t M, int64_t K, int64_t ldx, const float* P1, int n1, const float* P2, int n2,
                    int bits, int8_t* codes, int codes_layout, float* scales, int32_t* qsum, const void* V, int r,
                    void* Thl, float* lr_part, uint32_t* status, cudaStream_t stream);

// ---- rotation + quantiser on the warp-level tensor-core path (rot_mma.cu; its geometry: host_plans.h) ----
constexpr int kRotMaxProblems = 4;          // linears that share one x and are rotated by one launch
struct RotProblem {
    const uint8_t* prepared;    // terms of P2^T and P1^T (launch_prepare_rot), or NULL: P1 and P2 are split by every CTA
    const float *P1, *P2;       // read only when `prepared` is NULL
    const uint8_t* many;        // beside `prepared`: the terms in the layout of rot_rows.cu, or for factors that it does not take of okt_umma.cu, or NULL
    // quantiser (yhat == NULL)
    int8_t* codes;              // [M][K]
    int codes_layout;           // 0: natural k order; 1: the interleaved order of the tensor-core contraction
    int32_t* zp;                // [M] zero points (asymmetric quantiser), or NULL
    int code_bias;              // added to every stored code and to the stored zero point (see launch_rot)
    float* scales;              // [M]
    int32_t* qsum;              // [M][kQsumParts] or NULL
    float* y;                   // [M][K] fp32 rotated activations before the quantiser, or NULL
    // weight-only operating point: bf16 values, or (digits; codes, scales and qsum are then [3][M][K], [M], [3][M][kQsumParts])
    // their fixed-point digits
    int digits;
    __nv_bfloat16* yhat;        // [M][K]
    float* ysum;                // [M] sums of the rounded values, or NULL
    // final binarisation
    uint32_t* packed; float *alpha, *mu;
};
// V == NULL: no T = V x.  lr_part, lr_count: of the blocks beside the rotation; umma_part: of lowrank_umma.cu, may overlap the codes.
struct OktLowrank { const void* V; int r; void* Thl; float* lr_part; uint32_t* lr_count; float* umma_part; };
// rows of x that start on 16 bytes (others are read element by element, and the tcgen05 V x kernel does not take them)
bool rot_accepts_x(const void* x, int64_t ldx);
int launch_prepare_rot(const RotGeom& g, const float* P1, const float* P2, void* prepared, cudaStream_t stream);
// One launch for up to kRotMaxProblems linears that read the same x: rotation + quantiser for each, and the T = V x
// blocks of those with a low-rank branch.
// asym == 0: symmetric codes in [-qmax, qmax], qmax = 2^(b-1) - 1.  asym == 1 (Sec. 4.1, per-token asymmetric): with
// u in [0, 2^b - 1] and the integer zero point z of the token, the stored code is u - 2^(b-1) + code_bias and the
// stored zero point z - 2^(b-1) + code_bias; a code minus the zero point times the scale is the value it stands for.
// behind: SMs that the kernel behind it takes at once (0: not known; only asked for with raw factors and few tokens).
int launch_rot(const RotGeom& g, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems,
               const RotProblem* problems, const OktLowrank* lowrank, uint32_t* status, cudaStream_t stream, int behind = 0);
// The same for many tokens, on the tcgen05 tensor cores (rot_umma.cu); x in 16-byte pieces.  launch_rot goes there by itself.
int rot_few_cluster(const RotGeom& g, int64_t M, int n_problems, const RotProblem* problems);      // CTAs of a cluster where it takes few tokens in clusters, or 1
bool rot_umma_supports(const RotGeom& g, int n_problems, const RotProblem* problems);
int launch_rot_umma(const RotGeom& g, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems,
                    const RotProblem* problems, uint32_t* status, cudaStream_t stream);
// Many tokens of factors up to 128 x 128 (rot_rows.cu; launch_rot goes there by itself); x in 16-byte pieces
bool rot_rows_supports(const RotGeom& g, int n_problems, const RotProblem* problems);
int launch_prepare_rows(const RotRowsGeom& g, const float* P1, const float* P2, void* prepared, cudaStream_t stream);
// (beside: the T = V x that its launch evaluates too, rows of V on 16 bytes)
int launch_rot_rows(const RotGeom& g, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems,
                    const RotProblem* problems, const OktLowrank* beside, uint32_t* status, cudaStream_t stream);
int launch_rows_binarize(const RotGeom& g, const void* w, int dtype, int64_t N, int64_t ldw, const RotProblem& problem, uint32_t* status, bool* taken,
                         cudaStream_t stream);
// how many clusters of a kernel the device holds at once
int resident_clusters(const void* kernel, int dc, int threads, size_t smem);
// ---- many tokens of factors up to 128 (okt_umma.cu; launch_rot goes there by itself) ----
// Geometry of the kernel for one pair of factor sizes.
struct OktGeom {
    int n1, n2, K;
    int n1p, n2p;           // n1, n2 rounded up to 16: columns of Z^T / Y^T, contraction depth of the first stage
    int atom2, atom1;       // bytes of one K-atom row (the swizzle span) of operands contracted over b / over a
    int dt_count, dt_rows;  // tiles of the rows d of P2^T (= tensor-memory lanes) and rows per tile (a multiple of 8)
    int cs_count, cs_cols;  // slabs of the rows c of P1^T (= output columns) and columns per slab (a multiple of 16)
    int p2t_bytes, p1t_bytes, x_bytes;      // one tile of P2^T terms, one slab of P1^T terms, one token's X tile
    int p1t_off, x_off, bar_off;            // shared-memory offsets (P2^T tile at 0)
    int tmem_cols, smem_bytes;
};
bool okt_geometry(int n1, int n2, OktGeom* out);
size_t okt_prepared_bytes(const OktGeom& g);
int launch_prepare_okt(const OktGeom& g, const float* P1, const float* P2, void* prepared, cudaStream_t stream);
int launch_okt(const OktGeom& g, const void* x, int64_t M, int64_t ldx, int bits, int asym, int n_problems,
               const RotProblem* problems, const OktLowrank* lowrank, uint32_t* status, cudaStream_t stream);
// Rows of weights (fp32 or bf16): packed signs, scale and shift of every row.
int launch_rot_binarize(const RotGeom& g, const void* w, int dtype, int64_t N, int64_t ldw, const RotProblem& problem, uint32_t* status,
                        cudaStream_t stream);

// qsum[t][0] = sum_k codes[t][k] (the other parts zero); optionally rewrites natural-order codes into the interleaved order.
int launch_prepare_codes(const int8_t* codes, int64_t M, int64_t K, int8_t* codes_interleaved, int32_t* qsum,
                         cudaStream_t stream);

struct GemmArgs {
    const int8_t* codes;      // [M][K]; natural order for the simple path
    const float* scales;      // [M]
    const int32_t* qsum;      // [M][kQsumParts] partial sums
    int64_t M, K, N;
    int bits;
    const uint32_t* packed;   // [N][K/32]
    const float* alpha;       // [N]
    const float* mu;          // [N] or NULL
    const int32_t* zp;        // [M] per-token zero points of the codes, or NULL (symmetric codes)
    const int32_t* rowsum;    // [N] sum_k sign(n,k) = 2 * popc(row n) - K; read only when zp is given
    const void* Thl;          // bf16 [3][M][lowrank_cols(r)] or NULL
    const void* U;            // bf16 [N][r] or NULL
    int r;
    void* out;                // bf16 [M][ldo] or NULL
    int64_t ldo;
    int32_t* acc_debug;       // [M][N] or NULL
    uint32_t* status;         // workspace status words
    // Contractions of a group that read the results of the same preceding kernel (the rotation launch): the first one
    // (kDepHead) lets the next kernel of the stream start only once it has itself seen that kernel complete, so the
    // others (kDepSibling) need not wait for their predecessor, a sibling, before they read: they run beside it.
    // kDepChain: the ordinary chain (wait for the predecessor before reading its results).
    int dep_mode;
    int sm_budget;            // SMs this launch should plan for (0: all): siblings share the device
    int rot_cluster;          // CTAs of a cluster of the rotation before (few tokens; 0: not known, or no clusters)
};
enum { kDepChain = 0, kDepHead = 1, kDepSibling = 2 };

// W1A16, the weight-only operating point (gemm_a16.cu): the bf16 contraction against the packed signs with the fused
// epilogue.  Thl as for the int8 contractions (NULL when r == 0).
// The same in persistent CTAs, yhat in the interleaved order (RotProblem::codes_layout 1)
bool a16_persistent_supports(int64_t K);
int launch_a16_persistent(const void* yhat, const float* ysum, int64_t M, int64_t K, int64_t N, const uint32_t* packed,
                          const float* alpha, const float* mu, const void* U, int r, const void* Thl, void* out, int64_t ldo,
                          uint32_t* status, cudaStream_t stream);
bool a16_supports(int64_t M, int64_t K, int64_t N, int r);
int launch_gemm_a16(const void* yhat, const float* ysum, int64_t M, int64_t K, int64_t N, const uint32_t* packed, const float* alpha,
                    const float* mu, const void* U, int r, const void* Thl, void* out, int64_t ldo, uint32_t* status,
                    cudaStream_t stream);

int launch_gemm_simple(const GemmArgs& a, cudaStream_t stream);

// One to four tokens: activation bit-planes against the packed sign words (and + popc), weights never expanded.
// a.codes in natural k order.
bool bitplane_supports(int64_t M, int64_t K, int64_t N, int r, int bits);
int launch_gemm_bitplane(const GemmArgs& a, cudaStream_t stream);

// Up to kSmallTokens tokens: warp-level int8 MMAs, all linears of a group (same M, K, bits; a.codes in the interleaved order) in one
// launch.  planes == 3: three digit planes per token (the weight-only operating point, up to kSmallDigitTokens).  *taken is false, and
// nothing has been launched, for shapes whose codes do not fit shared memory: those go to the tcgen05 kernels.
bool gemm_small_fits(const GemmArgs* a, int n, int planes);
int gemm_small_blocks(const GemmArgs& a);      // of one linear's launch, one an SM; 0 where it does not fit
int launch_gemm_small(const GemmArgs* a, int n, int planes, bool* taken, cudaStream_t stream);

// tcgen05 path with the fused epilogue.  codes_interleaved: int8 [M][K] in the interleaved order.
bool umma_supports(int64_t M, int64_t K, int64_t N, int r, int bits);
int launch_gemm_umma(const GemmArgs& a, const int8_t* codes_interleaved, cudaStream_t stream);
int gemm_umma_sms(const GemmArgs& a);          // that its launch takes at once, or 0
// The weight-only operating point for few tokens as three digit planes a value, a.codes int8 [3][M][K]: planes are tokens to the MMAs
bool umma_digits_supports(int64_t M, int64_t K, int64_t N, int r);
int launch_gemm_umma_digits(const GemmArgs& a, cudaStream_t stream);
// More than 64 tokens: the same contraction in CTAs that stay on their SM and take tiles of 128 rows x 128 tokens in turn.
bool umma_persistent_supports(int64_t M, int64_t K, int64_t N, int r);
// n linears with the same M and K, all of them or none with a low-rank branch; codes in the interleaved order
int launch_gemm_umma_persistent(const GemmArgs* a, int n, cudaStream_t stream);

}  // namespace bwla
