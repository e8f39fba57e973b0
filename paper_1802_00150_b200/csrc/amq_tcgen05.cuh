// Device-side pieces shared by the tensor-core kernels: bounded mbarrier waits, operand descriptors, tcgen05 instructions with
// the weight operand in tensor memory, reads of tensor memory, unit block scales of the 4-bit operand form.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "amq_pairs.cuh"

namespace amq {

constexpr unsigned WAIT_LIMIT = 1u << 20;   // attempts on an mbarrier before giving up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}

// bounded wait of the single MMA-issuing thread; false when it ran out
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
#pragma unroll 1
    for (unsigned i = 0; i < WAIT_LIMIT; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// the same for the many expander threads: between attempts the thread sleeps, so that waiters do not take
// issue slots from the warps that have work
__device__ __forceinline__ bool mbar_wait_relaxed(uint32_t bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
#pragma unroll 1
    for (unsigned i = 0; i < WAIT_LIMIT; ++i) {
        __nanosleep(40);
        if (mbar_try_wait(bar, parity)) return true;
    }
    return false;
}

// the same for threads with nothing else to do: they sleep between attempts, and give up early once another role of the CTA has
// recorded a failure
__device__ __forceinline__ bool mbar_wait_relaxed(uint32_t bar, uint32_t parity, const volatile int* failed)
{
    if (mbar_try_wait(bar, parity)) return true;
#pragma unroll 1
    for (unsigned i = 0; i < WAIT_LIMIT && !*failed; ++i) {
        __nanosleep(40);
        if (mbar_try_wait(bar, parity)) return true;
    }
    return false;
}

// K-major, 128-byte swizzle: start address (the tile base is 1024-byte aligned), leading byte offset unused (1),
// stride byte offset = 1024 bytes between groups of 8 rows, descriptor version 1, layout type 2
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    return (uint64_t)((addr >> 4) & 0x3fffu) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// true in one lane of the (converged) warp.  The issuing warp runs its loop as a whole and only the tensor-core instructions are
// under this predicate: their operands then stay in uniform registers.  With the loop inside `if (lane == 0)` the compiler moved
// every operand of every MMA into them one by one, and a pipeline step of four MMAs cost the issuing thread 676 clocks whatever
// its N; this way it costs 230-300 (N <= 128: below the pace of the tensor pipe from N = 128 up).
__device__ __forceinline__ bool elect_one()
{
    uint32_t one;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(one));
    return one != 0;
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, int (&v)[8])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
        : "r"(taddr) : "memory");
}

// 32 lanes x 8 NUM columns of tensor memory in the layout of an m16n8 accumulator, complete on return: v[i][c] = the columns
// 8 c + 2 (l mod 4) + {0, 1} of lane l / 4 + 8 i.  (The loads, the wait and the packing are one block: nothing that uses the
// values can be moved above the wait.)
template <int NUM>
__device__ __forceinline__ void tmem_ld_pairs(uint32_t taddr, f32x2 (&v)[4][NUM])
{
    static_assert(NUM >= 1 && NUM <= 4, "");
    const uint32_t lower = taddr + (16u << 16);
    if constexpr (NUM == 1) {
        asm volatile(
            "{\n\t.reg .b32 a<4>, b<4>;\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {a0, a1, a2, a3}, [%4];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {b0, b1, b2, b3}, [%5];\n\t"
            "tcgen05.wait::ld.sync.aligned;\n\t"
            "mov.b64 %0, {a0, a1};\n\tmov.b64 %1, {a2, a3};\n\tmov.b64 %2, {b0, b1};\n\tmov.b64 %3, {b2, b3};\n\t}"
            : "=l"(v[0][0]), "=l"(v[1][0]), "=l"(v[2][0]), "=l"(v[3][0]) : "r"(taddr), "r"(lower) : "memory");
    } else if constexpr (NUM == 2) {
        asm volatile(
            "{\n\t.reg .b32 a<8>, b<8>;\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {a0, a1, a2, a3, a4, a5, a6, a7}, [%8];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {b0, b1, b2, b3, b4, b5, b6, b7}, [%9];\n\t"
            "tcgen05.wait::ld.sync.aligned;\n\t"
            "mov.b64 %0, {a0, a1};\n\tmov.b64 %1, {a2, a3};\n\tmov.b64 %2, {b0, b1};\n\tmov.b64 %3, {b2, b3};\n\t"
            "mov.b64 %4, {a4, a5};\n\tmov.b64 %5, {a6, a7};\n\tmov.b64 %6, {b4, b5};\n\tmov.b64 %7, {b6, b7};\n\t}"
            : "=l"(v[0][0]), "=l"(v[1][0]), "=l"(v[2][0]), "=l"(v[3][0]), "=l"(v[0][1]), "=l"(v[1][1]), "=l"(v[2][1]), "=l"(v[3][1])
            : "r"(taddr), "r"(lower) : "memory");
    } else if constexpr (NUM == 3) {
        asm volatile(
            "{\n\t.reg .b32 a<12>, b<12>;\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {a0, a1, a2, a3, a4, a5, a6, a7}, [%12];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x2.b32 {b0, b1, b2, b3, b4, b5, b6, b7}, [%13];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {a8, a9, a10, a11}, [%14];\n\t"
            "tcgen05.ld.sync.aligned.16x256b.x1.b32 {b8, b9, b10, b11}, [%15];\n\t"
            "tcgen05.wait::ld.sync.aligned;\n\t"
            "mov.b64 %0, {a0, a1};\n\tmov.b64 %1, {a2, a3};\n\tmov.b64 %2, {b0, b1};\n\tmov.b64 %3, {b2, b3};\n\t"
            "mov.b64 %4, {a4, a5};\n\tmov.b64 %5, {a6, a7};\n\tmov.b64 %6, {b4, b5};\n\tmov.b64 %7, {b6, b7};\n\t"
            "mov.b64 %8, {a8, a9};\n\tmov.b64 %9, {a10, a11};\n\tmov.b64 %10, {b8, b9};\n\tmov.b64 %11, {b10, b11};\n\t}"
            : "=l"(v[0][0]), "=l"(v[1][0]), "=l"(v[2][0]), "=l"(v[3][0]), "=l"(v[0][1]), "=l"(v[1][1]), "=l"(v[2][1]), "=l"(v[3][1]),
              "=l"(v[0][2]), "=l"(v[1][2]), "=l"(v[2][2]), "=l"(v[3][2])
            : "r"(taddr), "r"(lower), "r"(taddr + 16), "r"(lower + 16) : "memory");
    } else {
        f32x2 w[4][2];
        f32x2 u[4][2];
        tmem_ld_pairs<2>(taddr, u);
        tmem_ld_pairs<2>(taddr + 16, w);
#pragma unroll
        for (int i = 0; i < 4; ++i) { v[i][0] = u[i][0]; v[i][1] = u[i][1]; v[i][2] = w[i][0]; v[i][3] = w[i][1]; }
    }
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" :: "r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}

// The same with the weight operand in tensor memory (lanes 0..127, 8 columns = 64 nibbles per MMA).
__device__ __forceinline__ void mma_mxf4_stage_ta(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc,
                                                  uint32_t acc_first, uint32_t sf_tmem)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p, q;\n\t"
        ".reg .b64 db;\n\t"
        ".reg .b32 al, bl;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "setp.eq.b32 q, %5, %5;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], [%1], db, %4, [%6], [%6], p;\n\t"
        "add.u32 al, %1, 8;\n\t"
        "add.u32 bl, %2, 2;\n\t"
        "mov.b64 db, {bl, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], [al], db, %4, [%6], [%6], q;\n\t"
        "add.u32 al, %1, 16;\n\t"
        "add.u32 bl, %2, 4;\n\t"
        "mov.b64 db, {bl, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], [al], db, %4, [%6], [%6], q;\n\t"
        "add.u32 al, %1, 24;\n\t"
        "add.u32 bl, %2, 6;\n\t"
        "mov.b64 db, {bl, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.block32 [%0], [al], db, %4, [%6], [%6], q;\n\t"
        "}"
        :: "r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(acc_first), "r"(sf_tmem) : "memory");
}

// Scale factors of the 4-bit form: 16 tensor-memory columns, every byte 0x7F (2^0 in E8M0), written by four warps (one per
// lane quarter); both operands' scale addresses point at this region, whose every byte is the same.
__device__ __forceinline__ void write_unit_scales(uint32_t tmem_base, int sf_col, int warp)
{
    const uint32_t t = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)sf_col;
    const uint32_t one = 0x7F7F7F7Fu;
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};"
        :: "r"(t), "r"(one) : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ float logistic(float v) { return 1.0f / (1.0f + __expf(-v)); }

}  // namespace amq
