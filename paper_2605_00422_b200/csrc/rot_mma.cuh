// Warp-level pieces of the rotation kernels: ldmatrix, fp16 MMAs, cp.async and the power-of-two scalings.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

#include "umma_ptx.cuh"

namespace bwla {

// (the same sum in every lane)
__device__ __forceinline__ double warp_sum(double s) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
    return s;
}
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x2(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr));
}
// d = A (16 x 16) * B (16 x 8) + c, fp32 accumulators; F16: fp16 operands, else bf16.  (Not volatile: a register-only
// instruction that the scheduler may interleave with the chains beside it.)
template <bool F16>
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, const float* c) {
    if constexpr (F16)
        asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
    else
        asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
            : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}
// two fp32 additions / multiplications in one instruction (each rounded to nearest)
__device__ __forceinline__ void add2(float& a0, float& a1, float b0, float b1) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tadd.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(b0), "f"(b1));
}
__device__ __forceinline__ void mul2(float& a0, float& a1, float b) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %2};\n\tmul.rn.f32x2 x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"
        : "+f"(a0), "+f"(a1) : "f"(b));
}
__device__ __forceinline__ void add4(float (&c)[4], const float (&t)[4]) {
    add2(c[0], c[1], t[0], t[1]);
    add2(c[2], c[3], t[2], t[3]);
}
// A load whose value nobody uses: it brings the translation of the page to this SM (the first access to a page costs about
// 1.5 us), which neither of the L2 prefetches does.  Goes past the L1, so nothing stale stays behind.
__device__ __forceinline__ void touch(const void* p) {
    uint32_t v;
    asm volatile("ld.volatile.global.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3));
    asm volatile("" ::"r"(v));
}
__device__ __forceinline__ void prefetch_l2_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void named_barrier(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Two fp32 values as one fp16 pair (low half: the first), and an fp16 pair's residual of the same two values.
__device__ __forceinline__ uint32_t cvt_f16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ void split2_pair(float a, float b, uint32_t& h, uint32_t& l) {
    h = cvt_f16x2(a, b);
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&h));
    l = cvt_f16x2(a - f.x, b - f.y);
}

__device__ __forceinline__ uint32_t cvt_bf16x2_rn(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// Two fp32 values into their three bf16 terms (all 24 bits), two per word.
__device__ __forceinline__ void split3_pair(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = cvt_bf16x2_rn(a, b);
    const float ra = a - __uint_as_float(h << 16), rb = b - __uint_as_float(h & 0xFFFF0000u);
    m = cvt_bf16x2_rn(ra, rb);
    l = cvt_bf16x2_rn(ra - __uint_as_float(m << 16), rb - __uint_as_float(m & 0xFFFF0000u));
}

// 2^e for -126 <= e <= 127
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }
// floor(log2 v) of a non-negative finite v (subnormals and zero: -127)
__device__ __forceinline__ int exponent_of(float v) { return (int)((__float_as_uint(v) >> 23) & 0xFFu) - 127; }

// Exponent by which P1 is scaled: its largest magnitude goes to [2^13, 2^14).
__device__ __forceinline__ int factor_exponent(float amax) { return min(13 - exponent_of(amax), 126); }

// Largest |v| of n floats (v 16-byte aligned), over the threads of the block; `red` has a word per warp.
__device__ __forceinline__ float block_absmax(const float* __restrict__ v, int n, uint32_t* red) {
    uint32_t m = 0u;
    const float4* v4 = reinterpret_cast<const float4*>(v);
#pragma unroll 4
    for (int i = threadIdx.x; i < (n >> 2); i += blockDim.x) {
        const float4 f = __ldg(v4 + i);
        m = max(m, max(max(__float_as_uint(f.x) & 0x7FFFFFFFu, __float_as_uint(f.y) & 0x7FFFFFFFu),
                       max(__float_as_uint(f.z) & 0x7FFFFFFFu, __float_as_uint(f.w) & 0x7FFFFFFFu)));
    }
    if ((int)threadIdx.x < (n & 3)) m = max(m, __float_as_uint(__ldg(v + (n & ~3) + threadIdx.x)) & 0x7FFFFFFFu);
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[w]);
    return __uint_as_float(m);
}

// The terms of rows [r0, r0 + rows) of factor^T (element (r, k) = P[k][r], times scale), zero outside n x n: blocks of `block`
// bytes, one per term, kp columns; columns 2 k2, 2 k2 + 1 of row r (counted from r0) go to place(r, k2).  Threads run along r, so
// the reads of P are coalesced.
template <bool F16, typename Place>
__device__ __forceinline__ void split_factor(const float* __restrict__ P, int n, int r0, int rows, int kp, float scale, Place place,
                                             size_t block, int tid, int nthreads) {
    const int pairs = rows * (kp >> 1);
    constexpr int U = 4;
    for (int i0 = tid; i0 < pairs; i0 += U * nthreads) {
        float a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * nthreads, k2 = i / rows, r = i - k2 * rows, k = 2 * k2;
            const bool ok = i < pairs && r0 + r < n;
            a[u] = ok && k < n ? __ldg(P + (size_t)k * n + r0 + r) : 0.f;
            b[u] = ok && k + 1 < n ? __ldg(P + (size_t)(k + 1) * n + r0 + r) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = i0 + u * nthreads, k2 = i / rows, r = i - k2 * rows;
            if (i < pairs) {
                uint8_t* at = place(r, k2);
                uint32_t h, m, l;
                if (F16) {
                    split2_pair(a[u] * scale, b[u] * scale, h, l);
                    *reinterpret_cast<uint32_t*>(at) = h;
                    *reinterpret_cast<uint32_t*>(at + block) = l;
                } else {
                    split3_pair(a[u], b[u], h, m, l);
                    *reinterpret_cast<uint32_t*>(at) = h;
                    *reinterpret_cast<uint32_t*>(at + block) = m;
                    *reinterpret_cast<uint32_t*>(at + 2 * block) = l;
                }
            }
        }
    }
}

}  // namespace bwla
