// Inline-PTX helpers for the 5th-generation tensor cores (tcgen05) on sm_103a:
// TMEM allocation, shared-memory matrix descriptors, the kind::f16 MMA with A in TMEM, its
// commit to an mbarrier, TMEM loads and stores, and the FP16 slices of an amplitude.
#pragma once

#include <cuda_fp16.h>

#include <cstdint>

namespace svk {

// Shared-memory matrix descriptor: start address, leading / stride byte offsets, the
// fixed version bits (46-47 = 1), no base offset, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor for kind::f16: D = F32, A = B = F16, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_f16(uint32_t M, uint32_t N) {
    return (1u << 4) | (0u << 7) | (0u << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// Byte offset of 16-bit element (row, kk) of a K-major operand in the canonical layout
// without swizzle (core matrix = 8 rows x 8 elements).
__device__ __forceinline__ uint32_t kmajor_off16(uint32_t row, uint32_t kk, uint32_t sbo) {
    return (row >> 3) * sbo + (kk >> 3) * 128u + (row & 7u) * 16u + (kk & 7u) * 2u;
}

// Arrive once on the mbarrier when all previously issued MMAs of this thread complete.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(dst_smem), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 4 consecutive 32-bit TMEM columns of this thread's lane, without waiting: a later
// tmem_wait_st() orders the stores before the TMEM is read by an MMA.
__device__ __forceinline__ void tmem_st4_async(uint32_t taddr, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
                 : "memory");
}

__device__ __forceinline__ void tmem_st8_async(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]),
                   "r"(r[6]), "r"(r[7])
                 : "memory");
}

__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Five loads of 8 consecutive columns (at a0 + q * stride, q = 0..4) and one wait.
__device__ __forceinline__ void tmem_ld8x5(uint32_t a0, uint32_t stride, float (&v)[5][8]) {
    uint32_t r[40];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%40];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%41];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%42];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%43];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%32,%33,%34,%35,%36,%37,%38,%39}, [%44];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]),
          "=r"(r[37]), "=r"(r[38]), "=r"(r[39])
        : "r"(a0), "r"(a0 + stride), "r"(a0 + 2 * stride), "r"(a0 + 3 * stride),
          "r"(a0 + 4 * stride)
        : "memory");
#pragma unroll
    for (int q = 0; q < 5; ++q)
#pragma unroll
        for (int i = 0; i < 8; ++i) v[q][i] = __uint_as_float(r[8 * q + i]);
}

// Two loads of 16 consecutive columns (at a0 and a1) and one wait.
__device__ __forceinline__ void tmem_ld16x2(uint32_t a0, uint32_t a1, float (&v)[16], float (&w)[16]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(a0), "r"(a1)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        v[i] = __uint_as_float(r[i]);
        w[i] = __uint_as_float(r[16 + i]);
    }
}

// D[tmem] (+)= A[tmem] * B[smem]^T with 16-bit inputs (A: one row per lane, two elements
// per 32-bit column), issued by one thread.
__device__ __forceinline__ void mma_f16_tmem_a(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc,
                                               uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// max(m, |a|, |b|) in one three-input maximum (sm_100 and later).
__device__ __forceinline__ float max_abs2(float m, float a, float b) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(fabsf(a)), "f"(fabsf(b)));
    return r;
}

__device__ __forceinline__ uint32_t pack_h2(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// The three slices of a scaled amplitude (|x scale| < 256) at their scale: a1 (an
// integer), a2 2^-9 and a3 2^-18, with |a_i| <= 256; each FP16 pair (re, im) is exact.
// Rounding to the grid 2^e (ties to even, |x| < 2^(e + 22)) adds and subtracts
// c = 1.5 2^(e + 23): the sum keeps a unit in the last place of 2^e, so it is rounded to
// that grid, and the subtraction is exact; the remainders x - a1 and (x - a1) - a2 2^-9
// are exact FP32 differences (one fused multiply-add by -1).  (re, im) go through each
// step together as one packed FP32x2 instruction.
__device__ __forceinline__ void slices(float2 v, float2 scale, uint32_t &w1, uint32_t &w2, uint32_t &w3) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 x = __fmul2_rn(v, scale);
    const float2 r1 = __fadd2_rn(__fadd2_rn(x, make_float2(12582912.f, 12582912.f)),
                                 make_float2(-12582912.f, -12582912.f));              // 1.5 2^23
    const float2 x2 = __ffma2_rn(r1, m1, x);
    const float2 r2 = __fadd2_rn(__fadd2_rn(x2, make_float2(24576.f, 24576.f)),
                                 make_float2(-24576.f, -24576.f));                    // 1.5 2^14
    const float2 x3 = __ffma2_rn(r2, m1, x2);
    const float2 r3 = __fadd2_rn(__fadd2_rn(x3, make_float2(48.f, 48.f)), make_float2(-48.f, -48.f));   // 1.5 2^5
    w1 = pack_h2(r1.x, r1.y);
    w2 = pack_h2(r2.x, r2.y);
    w3 = pack_h2(r3.x, r3.y);
}

}  // namespace svk
