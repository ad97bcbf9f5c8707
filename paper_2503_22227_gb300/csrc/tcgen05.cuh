// Fifth-generation tensor cores (tcgen05) for one CTA: TMEM allocation, fp16
// products with fp32 accumulators, and reads of the accumulators.  Operands
// lie in shared memory in the unswizzled K-major layout: 16-byte rows of 8
// elements, 8 rows to a core matrix.
#pragma once

#include <stdint.h>

#include "bulk.cuh"

namespace catfhe {

// `cols` (a power of two, at least 32) TMEM columns; the base address goes to
// *slot in shared memory.  Executed by one whole warp; it may wait for other
// CTAs on the SM to free theirs, which none of them does only after this one.
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(slot)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

// Executed by the warp that allocated.
__device__ __forceinline__ void tmem_free(uint32_t base, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols)
                 : "memory");
}

__device__ __forceinline__ void tcgen05_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tcgen05_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory operand descriptor: unswizzled K-major, `lead` bytes from one
// core matrix to the next along K and `stride` bytes along M or N.
__device__ __forceinline__ uint64_t mma_desc(const void *p, uint32_t lead, uint32_t stride) {
    return uint64_t((smem_u32(p) >> 4) & 0x3fff) | uint64_t((lead >> 4) & 0x3fff) << 16 |
           uint64_t((stride >> 4) & 0x3fff) << 32 | uint64_t(1) << 46;
}

// Instruction descriptor: fp16 operands, fp32 accumulators, 128 rows, n columns.
__device__ __forceinline__ constexpr uint32_t mma_idesc(uint32_t n) {
    return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}

// D[128 x n] = A B^T (+ D), 16 elements of K; issued by one thread.
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                        bool accumulate) {
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
        "}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(uint32_t(accumulate))
        : "memory");
}

// One arrival on bar when this thread's products so far have completed.
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}

// 16 accumulator columns of this thread's row (each warp reads 32 rows: `addr`
// carries the first in bits 16 and up).  The values are there after
// tmem_wait16 on them.
__device__ __forceinline__ void tmem_load16(uint32_t addr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
          "=r"(v[14]), "=r"(v[15])
        : "r"(addr)
        : "memory");
}

__device__ __forceinline__ void tmem_wait16(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                   "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                   "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :
                 : "memory");
}

}  // namespace catfhe
