// Inline-PTX helpers for the 5th-generation tensor cores of sm_103a:
// tensor-memory (TMEM) allocation, shared-memory matrix descriptors,
// single-thread tcgen05.mma issue with mbarrier completion, and TMEM <->
// register transfers for the epilogue.
#pragma once

#include <stdint.h>

namespace sq {
namespace dev {

// Shared-memory matrix descriptor for a 128-byte-swizzled operand.
//   K-major tiles (rows of 64 bf16 = 128 B, 8-row groups 1024 B apart):
//     lbo unused (16), sbo = 1024; a K step of 16 elements advances the start
//     address by 32 B inside a 64-column block.
//   MN-major tiles (rows along K, 64 MN-elements per 128-B row):
//     lbo = byte distance between consecutive 64-element MN blocks,
//     sbo = 1024 (8 K-rows); a K step of 16 rows advances by 16 * 128 B.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of the 5th-generation tensor core
    d |= (uint64_t)2 << 61;  // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: bf16 A and B, f32 accumulator,
// A K-major, B K-major or MN-major, M x N tile.
__host__ __device__ constexpr uint32_t mma_idesc_bf16(int M, int N, bool b_mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Warp-wide: allocate `cols` TMEM columns, the base address written to smem.
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
                 "r"(cols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// One product over a contraction of steps of 16 elements, issued by one thread
// as one block of instructions.  The issuing thread is the bound of a stream
// of 128 x 128 products (64 cycles each on the tensor core), so each step
// costs it as little as possible: a descriptor's low word holds address / 16
// in 14 bits, every operand here lies below 2^18 bytes, so a step adds a
// constant to that word alone.
//
// D[tmem] = A[smem] * B[smem], both K-major with the same high descriptor
// word, D / 16 steps over one or two 64-column blocks of 16 KiB.
template <int N>
__device__ __forceinline__ void mma_bf16_ss_steps(uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo,
                                                  uint32_t hi, uint32_t idesc) {
    static_assert(N == 4 || N == 8, "one or two 64-column blocks");
    if constexpr (N == 8)
        asm volatile(
            "{\n\t"
            ".reg .pred f, t;\n\t"
            ".reg .b32 la, lb;\n\t"
            ".reg .b64 a, b;\n\t"
            "setp.ne.b32 f, 0, 0;\n\t"
            "setp.eq.b32 t, 0, 0;\n\t"
            "mov.b64 a, {%1, %3};\n\t"
            "mov.b64 b, {%2, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, f;\n\t"
            "add.u32 la, %1, 2;\n\t"
            "add.u32 lb, %2, 2;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 4;\n\t"
            "add.u32 lb, %2, 4;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 6;\n\t"
            "add.u32 lb, %2, 6;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 1024;\n\t"
            "add.u32 lb, %2, 1024;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 1026;\n\t"
            "add.u32 lb, %2, 1026;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 1028;\n\t"
            "add.u32 lb, %2, 1028;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 1030;\n\t"
            "add.u32 lb, %2, 1030;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "}\n\t"
            ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc)
            : "memory");
    else
        asm volatile(
            "{\n\t"
            ".reg .pred f, t;\n\t"
            ".reg .b32 la, lb;\n\t"
            ".reg .b64 a, b;\n\t"
            "setp.ne.b32 f, 0, 0;\n\t"
            "setp.eq.b32 t, 0, 0;\n\t"
            "mov.b64 a, {%1, %3};\n\t"
            "mov.b64 b, {%2, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, f;\n\t"
            "add.u32 la, %1, 2;\n\t"
            "add.u32 lb, %2, 2;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 4;\n\t"
            "add.u32 lb, %2, 4;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "add.u32 la, %1, 6;\n\t"
            "add.u32 lb, %2, 6;\n\t"
            "mov.b64 a, {la, %3};\n\t"
            "mov.b64 b, {lb, %3};\n\t"
            "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %4, t;\n\t"
            "}\n\t"
            ::"r"(d_tmem), "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc)
            : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem] over 8 steps.  A (M rows x K) sits in TMEM
// with row m in lane m and two bf16 per 32-bit column (column c holds elements
// 2c in its low half and 2c + 1 in its high half), so a step advances the A
// address by 8 columns; B is MN-major, a step 16 rows of 128 bytes.
__device__ __forceinline__ void mma_bf16_ts_steps8(uint32_t d_tmem, uint32_t a, uint32_t b_lo,
                                                   uint32_t b_hi, uint32_t idesc,
                                                   uint32_t accumulate) {
    asm volatile(
        "{\n\t"
        ".reg .pred f, t;\n\t"
        ".reg .b32 la, lb;\n\t"
        ".reg .b64 b;\n\t"
        "setp.ne.b32 f, %5, 0;\n\t"
        "setp.eq.b32 t, 0, 0;\n\t"
        "mov.b64 b, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, f;\n\t"
        "add.u32 la, %1, 8;\n\t"
        "add.u32 lb, %2, 128;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "add.u32 la, %1, 16;\n\t"
        "add.u32 lb, %2, 256;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "add.u32 la, %1, 24;\n\t"
        "add.u32 lb, %2, 384;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "add.u32 la, %1, 32;\n\t"
        "add.u32 lb, %2, 512;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "add.u32 la, %1, 40;\n\t"
        "add.u32 lb, %2, 640;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "add.u32 la, %1, 48;\n\t"
        "add.u32 lb, %2, 768;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "add.u32 la, %1, 56;\n\t"
        "add.u32 lb, %2, 896;\n\t"
        "mov.b64 b, {lb, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [la], b, %4, t;\n\t"
        "}\n\t"
        ::"r"(d_tmem), "r"(a), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrive once on `bar` when every tcgen05 operation this thread issued so far
// has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

// Warp-wide: 32 consecutive 32-bit columns of the warp's 32 TMEM lanes; lane
// i of the warp receives lane (base lane + i).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
        "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
          "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
          "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
          "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr));
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
        "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]),
        "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]),
        "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_wait_st() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

}  // namespace dev
}  // namespace sq
