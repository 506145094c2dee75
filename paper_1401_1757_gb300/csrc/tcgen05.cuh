// tcgen05.cuh -- PTX wrappers of the 5th-generation tensor cores and of tiled TMA
// copies, and the host's tensor-map encoder.
#pragma once

#include <cuda.h>

#include <cstdint>

#include "rsv_device.cuh"

namespace rsv {

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
        "[%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory operand descriptors, K-major: rows of 128 (64) bytes in the 128-byte
// (64-byte) swizzle, 8-row groups 1024 (512) bytes apart.
__device__ __forceinline__ uint64_t swizzled_desc(const void* smem, uint32_t group_bytes, uint32_t layout) {
    const uint64_t addr = smem_u32(smem);
    uint64_t d = 0;
    d |= (addr >> 4) & 0x3FFFull;                // start address
    d |= (uint64_t)1 << 16;                      // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(group_bytes >> 4) << 32;     // stride byte offset: 8 rows
    d |= (uint64_t)1 << 46;                      // descriptor version (tcgen05)
    d |= (uint64_t)layout << 61;                 // 2: 128-byte swizzle, 4: 64-byte
    return d;
}
__device__ __forceinline__ uint64_t sw128_desc(const void* smem) { return swizzled_desc(smem, 1024, 2); }
__device__ __forceinline__ uint64_t sw64_desc(const void* smem) { return swizzled_desc(smem, 512, 4); }

// kind::f16 instruction descriptor: FP32 accumulate, A and B both BF16 or both FP16, K-major.
__host__ __device__ constexpr uint32_t f16_idesc(bool bf16, int m, int n) {
    return (1u << 4) | (bf16 ? (1u << 7) | (1u << 10) : 0u) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// D (TMEM) [+]= A . B with A from shared memory
__device__ __forceinline__ void mma_f16_ss(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}
// D (TMEM) [+]= A . B with A from tensor memory
__device__ __forceinline__ void mma_f16_ts(uint32_t tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem),
        "r"(a_tmem), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 16 columns of this warp's 32 lanes from TMEM, without waiting: the values
// may be used only after tmem_wait_ld.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
// Wait for this thread's TMEM loads; the registers pass through an empty asm
// after the wait, so that no use of them is scheduled before it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(bar))
                 : "memory");
}

// One thread of a converged warp.  The compiler knows that code under it is run by one thread and
// keeps the operands of the instructions that it issues in uniform registers.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// One warp allocates (frees) `cols` TMEM columns; the address goes to *slot.
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free(uint32_t tmem, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

// ---- pairs of CTAs (a cluster of two): one instruction multiplies 256 rows, 128 of each
// CTA's A, with B of which each CTA holds half the columns' rows; issued by rank 0.
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// the address of rank 0's copy of a shared variable
__device__ __forceinline__ uint32_t of_rank0(const void* p) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
    return r;
}
// After fence_before: orders what was done in tensor memory and no other memory, so that it does not
// wait for the thread's stores (with .release 1,500 cycles more until the waiting thread saw it).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// into this CTA's shared memory, completing on a barrier of either CTA
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
        "[%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
// COLL: whether A stays in the collector buffer for the next products, or is taken from it
enum { COLL_NONE, COLL_FILL, COLL_USE, COLL_LAST };
template <int COLL = COLL_NONE>
__device__ __forceinline__ void mma_f16_ss_pair(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum) {
#define RSV_MMA_PAIR(op)                                                   \
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"         \
                 "tcgen05.mma.cta_group::2.kind::f16" op " [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem), \
                 "l"(a), "l"(b), "r"(idesc), "r"(accum)                    \
                 : "memory")
    if constexpr (COLL == COLL_FILL) RSV_MMA_PAIR(".collector::a::fill");
    else if constexpr (COLL == COLL_USE) RSV_MMA_PAIR(".collector::a::use");
    else if constexpr (COLL == COLL_LAST) RSV_MMA_PAIR(".collector::a::lastuse");
    else RSV_MMA_PAIR("");
#undef RSV_MMA_PAIR
}
// arrives at the barrier's copies in both CTAs
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_free_pair(uint32_t tmem, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}

// ---- host: tensor maps through the driver entry point ---------------------
// 2-D map of 16-bit elements over [rows][cols] (cols contiguous, row pitch in
// elements), box box_cols x box_rows; false where the encoder is missing or refuses.
bool encode_map_16bit(CUtensorMap* m, CUtensorMapDataType type, const void* ptr, uint64_t cols, uint64_t rows,
                      uint64_t pitch, uint32_t box_cols, uint32_t box_rows, CUtensorMapSwizzle swizzle);

}  // namespace rsv
