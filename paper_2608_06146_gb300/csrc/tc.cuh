// tc.cuh -- tcgen05 (5th-generation tensor core) helpers for sm_103a: TMEM allocation, UMMA
// shared-memory and instruction descriptors, MMA issue/commit, and TMEM loads/stores.
//
// Operand layouts used throughout (all bf16, 128-byte swizzle, panels of 64 elements = 128 bytes
// per row, 8-row swizzle atoms of 1024 bytes, panels 1024-byte aligned):
//   K-major operand [rows][K]: panel p holds K elements 64p..64p+63 of every row; a K-step of 16
//     elements inside a panel advances the start address by 32 bytes; rows advance by 128 bytes,
//     8-row groups by SBO = 1024 bytes.
//   MN-major operand [K][MN] (e.g. V as the B operand of P.V, stored [token][dim]): panel p holds
//     MN elements 64p..64p+63 of every K row; MN chunks of 64 are LBO = panel bytes apart, groups of
//     8 K rows SBO = 1024 bytes apart; a K-step of 16 rows advances the start address by 2048 bytes.
#pragma once

#include <stdint.h>

// ------------------------------------------------------------------------------------------------
// Descriptors
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes)
{
    uint64_t d = 0;
    d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;   // descriptor version of sm_100-family tcgen05
    d |= (uint64_t)2 << 61;   // 128-byte swizzle
    return d;
}

// kind::f16 instruction descriptor: bf16 A and B, fp32 accumulator, A K-major, B K-major or MN-major.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N, bool b_mn_major)
{
    return (1u << 4)                                  // D: f32
         | (1u << 7)                                  // A: bf16
         | (1u << 10)                                 // B: bf16
         | ((b_mn_major ? 1u : 0u) << 16)             // B major-ness
         | ((uint32_t)(N >> 3) << 17)                 // N / 8
         | ((uint32_t)(M >> 4) << 24);                // M / 16
}

// The same for f16 A and B.
__host__ __device__ constexpr uint32_t umma_idesc_f16(int M, int N, bool b_mn_major)
{
    return umma_idesc_bf16(M, N, b_mn_major) & ~((1u << 7) | (1u << 10));
}

// ------------------------------------------------------------------------------------------------
// TMEM
// ------------------------------------------------------------------------------------------------
// Executed by one full warp (CG = 2: by one warp of each CTA of the pair). Writes the allocated TMEM
// base address to shared memory.
template <int CG = 1>
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    if constexpr (CG == 2)
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                     : "memory");
    else
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                     : "memory");
}
template <int CG = 1>
__device__ __forceinline__ void tmem_relinquish()
{
    if constexpr (CG == 2) asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    else asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
template <int CG = 1>
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    if constexpr (CG == 2)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] . B[smem]^T, issued by one thread.
__device__ __forceinline__ void umma_bf16_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// D[tmem] (+)= A[tmem] . B[smem]^T, issued by one thread. A occupies M lanes x (K/2) columns: column c
// of lane m holds A[m][2c] in its low and A[m][2c+1] in its high 16 bits.
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Warp-collective forms: the whole (converged) warp executes them and one elected lane issues. Keeping
// the issuing warp converged lets descriptors live in uniform registers, which the MMA issue path
// needs to sustain one 128x128x16 MMA every 64 cycles.
__device__ __forceinline__ void umma_bf16_ss_warp(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                  uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p, e;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_bf16_ts_warp(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                                  uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p, e;\n elect.sync _|e, 0xffffffff;\n setp.ne.b32 p, %4, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Eight K-steps (128 elements) of a K-major product in one block, D = A[smem] . B[smem]^T: a step adds
// 32 bytes to both start addresses, the fifth one starts the second 64-element panel (PA and PB bytes
// on). One election and in-block address arithmetic: with a statement per MMA the compiler hoists
// every step's descriptors out of the caller's loop and spills them. CG = 2: one MMA over a CTA pair,
// issued by the leader (M = 256, half of the rows and of D in each CTA, half of B's rows in each).
template <int CG, int PA, int PB>
__device__ __forceinline__ void umma_bf16_ss_k128_warp(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc)
{
    if constexpr (CG == 2)
        asm volatile(
            "{\n .reg .pred e, t, f;\n .reg .b64 a, b;\n elect.sync _|e, 0xffffffff;\n"
            " setp.eq.u32 t, 0, 0;\n setp.ne.u32 f, 0, 0;\n"
            " @e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, f;\n"
            " add.s64 a, %1, 2;\n add.s64 b, %2, 2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, 4;\n add.s64 b, %2, 4;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, 6;\n add.s64 b, %2, 6;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4;\n add.s64 b, %2, %5;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4+2;\n add.s64 b, %2, %5+2;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4+4;\n add.s64 b, %2, %5+4;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4+6;\n add.s64 b, %2, %5+6;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], a, b, %3, t;\n}" ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(PA >> 4), "n"(PB >> 4)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred e, t, f;\n .reg .b64 a, b;\n elect.sync _|e, 0xffffffff;\n"
            " setp.eq.u32 t, 0, 0;\n setp.ne.u32 f, 0, 0;\n"
            " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, f;\n"
            " add.s64 a, %1, 2;\n add.s64 b, %2, 2;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, 4;\n add.s64 b, %2, 4;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, 6;\n add.s64 b, %2, 6;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4;\n add.s64 b, %2, %5;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4+2;\n add.s64 b, %2, %5+2;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4+4;\n add.s64 b, %2, %5+4;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n"
            " add.s64 a, %1, %4+6;\n add.s64 b, %2, %5+6;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, t;\n}" ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(PA >> 4), "n"(PB >> 4)
            : "memory");
}
// Four K-steps (64 elements) of D (+)= A[tmem] . B[smem], B MN-major (a step adds 16 rows, 2048 bytes);
// A's steps start at columns 0, A1, A2 and A3; `accumulate` 0: the first step overwrites D.
template <int CG, int A1 = 8, int A2 = 16, int A3 = 24>
__device__ __forceinline__ void umma_bf16_ts_k64_mn_warp(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                                         uint32_t accumulate)
{
    if constexpr (CG == 2)
        asm volatile(
            "{\n .reg .pred e, t, p;\n .reg .b64 b;\n .reg .b32 a;\n elect.sync _|e, 0xffffffff;\n"
            " setp.eq.u32 t, 0, 0;\n setp.ne.b32 p, %4, 0;\n"
            " @e tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n"
            " add.s32 a, %1, %5;\n add.s64 b, %2, 128;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], [a], b, %3, t;\n"
            " add.s32 a, %1, %6;\n add.s64 b, %2, 256;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], [a], b, %3, t;\n"
            " add.s32 a, %1, %7;\n add.s64 b, %2, 384;\n @e tcgen05.mma.cta_group::2.kind::f16 [%0], [a], b, %3, t;\n}" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "n"(A1), "n"(A2), "n"(A3)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred e, t, p;\n .reg .b64 b;\n .reg .b32 a;\n elect.sync _|e, 0xffffffff;\n"
            " setp.eq.u32 t, 0, 0;\n setp.ne.b32 p, %4, 0;\n"
            " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
            " add.s32 a, %1, %5;\n add.s64 b, %2, 128;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
            " add.s32 a, %1, %6;\n add.s64 b, %2, 256;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
            " add.s32 a, %1, %7;\n add.s64 b, %2, 384;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n}" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate), "n"(A1), "n"(A2), "n"(A3)
            : "memory");
}
// Eight K-steps (128 elements) of D = A[tmem] . B[smem]^T, B K-major (panels of 64 elements, PB bytes apart).
template <int PB>
__device__ __forceinline__ void umma_bf16_ts_k128_warp(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc)
{
    asm volatile(
        "{\n .reg .pred e, t, f;\n .reg .b64 b;\n .reg .b32 a;\n elect.sync _|e, 0xffffffff;\n"
        " setp.eq.u32 t, 0, 0;\n setp.ne.u32 f, 0, 0;\n"
        " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, f;\n"
        " add.s32 a, %1, 8;\n add.s64 b, %2, 2;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
        " add.s32 a, %1, 16;\n add.s64 b, %2, 4;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
        " add.s32 a, %1, 24;\n add.s64 b, %2, 6;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
        " add.s32 a, %1, 32;\n add.s64 b, %2, %4;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
        " add.s32 a, %1, 40;\n add.s64 b, %2, %4+2;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
        " add.s32 a, %1, 48;\n add.s64 b, %2, %4+4;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n"
        " add.s32 a, %1, 56;\n add.s64 b, %2, %4+6;\n @e tcgen05.mma.cta_group::1.kind::f16 [%0], [a], b, %3, t;\n}" ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "n"(PB >> 4)
        : "memory");
}
// As umma_commit_warp for MMAs over a CTA pair: arrives on the barrier at this offset in both CTAs.
__device__ __forceinline__ void umma_commit_pair_warp(uint32_t mbar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}" ::"r"(mbar),
        "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void umma_commit_warp(uint32_t mbar)
{
    asm volatile(
        "{\n .reg .pred e;\n elect.sync _|e, 0xffffffff;\n"
        " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(mbar)
        : "memory");
}

// Arrives once on the mbarrier when every tcgen05 operation issued so far by this thread completes.
__device__ __forceinline__ void umma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: thread i of the warp gets lane (taddr.lane + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
        "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
        "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// 32 lanes x 8 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Packed pairs of fp32 (one instruction for two lanes of arithmetic on sm_100-family GPUs).
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float &lo, float &hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_sub(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Three-input maximum (one instruction on sm_100-family GPUs).
__device__ __forceinline__ float fmax3f(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Bits [s, e) of a 32-bit word, for the part of the column interval [lo, lo + w) that falls in the
// 32 columns starting at base.
__device__ __forceinline__ uint32_t interval_bits(int lo, int w, int base)
{
    const int s = max(lo - base, 0), e = min(lo + w - base, 32);
    if (e <= s) return 0u;
    const uint32_t ones = (e - s) >= 32 ? 0xffffffffu : ((1u << (e - s)) - 1u);
    return ones << s;
}

__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t pred = 0;
    asm volatile(
        "{\n .reg .pred p;\n .reg .b32 r;\n elect.sync r|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(pred));
    return pred;
}
