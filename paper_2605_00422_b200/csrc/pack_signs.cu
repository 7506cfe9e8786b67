// Binarisation of rotated/centred weights into packed sign words (Eq. 2-3: Sign(w) = +1 iff w > 0).
#include <cuda_bf16.h>

#include "bwla_common.cuh"

namespace bwla {

template <typename T>
__device__ __forceinline__ bool is_positive(T v);
template <>
__device__ __forceinline__ bool is_positive<float>(float v) { return v > 0.0f; }
template <>
__device__ __forceinline__ bool is_positive<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v) > 0.0f; }

// Bound: HBM (4 or 2 bytes in, one bit out per weight).  A thread reads 16 bytes of bf16 (32 of fp32) = eight weights and
// stores their eight signs as one byte: byte i of a row holds weights 8 i .. 8 i + 7, LSB first, which is the little-endian
// view of the words, so nothing is exchanged between lanes and a warp's store fills one 32-byte sector.  kPackUnroll such
// groups per thread are requested before the first is used: the loads in flight cover the latency (one load of 2 bytes
// per lane and step, the kernel below, ran at 0.85 TB/s on 25600 x 5120 bf16).
constexpr int kPackUnroll = 4;

// eight comparisons with zero -> one byte.  bf16: a packed comparison gives a 16-bit mask per value (false for NaN).
__device__ __forceinline__ uint32_t sign_byte(const uint4& v) {
    const uint32_t in[4] = {v.x, v.y, v.z, v.w};
    uint32_t acc = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        __nv_bfloat162 pair;
        *reinterpret_cast<uint32_t*>(&pair) = in[i];
        acc |= __hgt2_mask(pair, __nv_bfloat162(__nv_bfloat16_raw{0}, __nv_bfloat16_raw{0})) & (0x00020001u << (2 * i));
    }
    return (acc | (acc >> 16)) & 0xFFu;
}
__device__ __forceinline__ uint32_t sign_byte(const float4& a, const float4& b) {
    const float f[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t acc = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) acc |= f[i] > 0.f ? (1u << i) : 0u;
    return acc;
}

// `groups` groups of eight weights per row, rows of ldw weights (rows that lie back to back come as one long row).
template <typename T>
__global__ void __launch_bounds__(256) pack_signs_vec_kernel(const T* __restrict__ w, int64_t rows, int64_t groups, int64_t ldw,
                                                             uint8_t* __restrict__ packed) {
    const int64_t c0 = (int64_t)blockIdx.x * (256 * kPackUnroll) + threadIdx.x;
    for (int64_t row = blockIdx.y; row < rows; row += gridDim.y) {
        const uint4* src = reinterpret_cast<const uint4*>(w + row * ldw);
        uint8_t* dst = packed + row * groups;
        uint4 v[kPackUnroll][sizeof(T) / 2];
#pragma unroll
        for (int u = 0; u < kPackUnroll; ++u) {
            const int64_t c = c0 + 256 * u;
            if (c < groups) {
#pragma unroll
                for (int h = 0; h < (int)(sizeof(T) / 2); ++h) v[u][h] = __ldcs(src + c * (sizeof(T) / 2) + h);
            }
        }
#pragma unroll
        for (int u = 0; u < kPackUnroll; ++u) {
            const int64_t c = c0 + 256 * u;
            if (c < groups) {
                uint32_t b;
                if constexpr (sizeof(T) == 2) b = sign_byte(v[u][0]);
                else b = sign_byte(*reinterpret_cast<const float4*>(&v[u][0]), *reinterpret_cast<const float4*>(&v[u][1]));
                dst[c] = (uint8_t)b;
            }
        }
    }
    __threadfence();       // (the next call may read the words as constants, before it waits for this kernel's end)
}

// Rows whose start is not 16-byte aligned.  One warp produces one 32-bit word per step: lane l looks at weight
// 32*word + l, the ballot is the word (LSB-first).
template <typename T>
__global__ void __launch_bounds__(256) pack_signs_kernel(const T* __restrict__ w, int64_t N, int64_t words,
                                                         int64_t ldw, uint32_t* __restrict__ packed) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t total = N * words;
    for (int64_t i = warp; i < total; i += nwarps) {
        const int64_t n = i / words, wd = i - n * words;
        const bool pos = is_positive<T>(w[n * ldw + wd * 32 + lane]);
        const uint32_t word = __ballot_sync(0xFFFFFFFFu, pos);
        if (lane == 0) packed[i] = word;
    }
    __threadfence();
}

// One warp per row: the number of +1 weights minus the number of -1 weights.
__global__ void __launch_bounds__(256) row_sums_kernel(const uint32_t* __restrict__ packed, int64_t N, int64_t words,
                                                       int32_t* __restrict__ rowsum) {
    const int lane = threadIdx.x & 31;
    const int64_t row = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= N) return;
    int ones = 0;
    for (int64_t w = lane; w < words; w += 32) ones += __popc(packed[row * words + w]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ones += __shfl_xor_sync(0xFFFFFFFFu, ones, o);
    if (lane == 0) rowsum[row] = 2 * ones - (int32_t)(words * 32);
}

int launch_row_sums(const uint32_t* packed, int64_t N, int64_t K, int32_t* rowsum, cudaStream_t stream) {
    if (N == 0) return BWLA_OK;
    ProfScope prof(kProfPack, stream);
    row_sums_kernel<<<(unsigned)((N + 7) / 8), 256, 0, stream>>>(packed, N, K / 32, rowsum);
    return after_launch();
}

int launch_pack_signs(const void* w, int dtype, int64_t N, int64_t K, int64_t ldw, uint32_t* packed,
                      cudaStream_t stream) {
    const int64_t words = K / 32;
    const int64_t total = N * words;
    if (total == 0) return BWLA_OK;
    const int64_t esize = dtype == BWLA_DTYPE_F32 ? 4 : 2;
    if ((reinterpret_cast<uintptr_t>(w) & 15) == 0 && (ldw * esize) % 16 == 0) {
        int64_t rows = N, groups = K / 8;
        if (ldw == K) { groups *= N; rows = 1; }
        const int64_t gx = (groups + 256 * kPackUnroll - 1) / (256 * kPackUnroll);
        const dim3 grid((unsigned)gx, (unsigned)std::min<int64_t>(rows, 65535));
        if (gx < ((int64_t)1 << 31)) {
            ProfScope prof(kProfPack, stream);
            if (dtype == BWLA_DTYPE_F32)
                pack_signs_vec_kernel<float><<<grid, 256, 0, stream>>>((const float*)w, rows, groups, ldw, (uint8_t*)packed);
            else
                pack_signs_vec_kernel<__nv_bfloat16><<<grid, 256, 0, stream>>>((const __nv_bfloat16*)w, rows, groups, ldw, (uint8_t*)packed);
            return after_launch();
        }
    }
    const int warps_per_block = 8;
    int64_t blocks = (total + warps_per_block - 1) / warps_per_block;
    const int64_t cap = (int64_t)(sm_count() > 0 ? sm_count() : 128) * 16;   // the kernel strides over the rest
    if (blocks > cap) blocks = cap;
    ProfScope prof(kProfPack, stream);
    if (dtype == BWLA_DTYPE_F32)
        pack_signs_kernel<float><<<(unsigned)blocks, 256, 0, stream>>>((const float*)w, N, words, ldw, packed);
    else
        pack_signs_kernel<__nv_bfloat16><<<(unsigned)blocks, 256, 0, stream>>>((const __nv_bfloat16*)w, N, words,
                                                                             ldw, packed);
    return after_launch();
}

}  // namespace bwla
