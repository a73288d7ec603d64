// Building blocks of the tcgen05 kernels: mbarriers, TMA loads, matrix and
// instruction descriptors, tensor-memory access.
//
// Every mbarrier wait is bounded (about 2 s on the global timer): on a
// timeout a kernel raises its error flag, still waits (bounded) for the
// copies it issued, frees its TMEM and returns.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace lbms {

constexpr uint64_t kWaitNs = 2000000000ull;    // bound of every mbarrier wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Whether the phase of parity `par` is complete (waits a short, bounded time
// in hardware).
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t par) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(par)
        : "memory");
    return done;
}

// Waits for the completion of the phase of parity `par`; false after kWaitNs.
// The timer is read only once the first tries have failed: a read costs more
// than a wait on a phase that is already complete.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t par) {
    for (int i = 0; i < 16; ++i)
        if (mbar_try(bar, par)) return true;
    const uint64_t t0 = global_ns();
    while (true) {
        for (int i = 0; i < 16; ++i)
            if (mbar_try(bar, par)) return true;
        if (global_ns() - t0 > kWaitNs) return false;
    }
}

// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
    return p;
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Shared-memory matrix descriptor: start address >> 4 (bits 0-13), leading
// and stride byte offsets >> 4 (bits 16-29, 32-45), the fixed 0b001 of bits
// 46-48, base offset 0, swizzle mode (bits 61-63): 2 = 128 B, 4 = 64 B.
// The swizzle is a function of the shared-memory address, as TMA wrote it,
// so a start any whole number of rows into a tile reads the right rows.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lead, uint32_t stride, uint32_t row_bytes) {
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(lead >> 4) << 16) | ((uint64_t)(stride >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)(row_bytes == 128 ? 2 : 4) << 61);
}

// Descriptors advance by bytes >> 4 added to the start address (shared memory
// ends far below the field's 256 KB, so no carry leaves it).
//
// K-major operand: rows of row_bytes (64 or 128, one swizzle span of BF16),
// 8-row groups 8 row_bytes apart; a 16-element K slice starts 32 bytes on.
__device__ __forceinline__ uint64_t kmajor_desc(uint32_t saddr, uint32_t row_bytes) {
    return smem_desc(saddr, 16, 8 * row_bytes, row_bytes);
}

// MN-major operand: K rows of row_bytes (32 or 64 MN elements), 8-row groups
// 8 row_bytes apart; the next row_bytes / 2 MN elements start `lead` bytes on.
__device__ __forceinline__ uint64_t mnmajor_desc(uint32_t saddr, uint32_t lead, uint32_t row_bytes) {
    return smem_desc(saddr, lead, 8 * row_bytes, row_bytes);
}

// Instruction descriptor of tcgen05.mma kind::f16: D FP32 (bits 4-5 = 1), A
// and B BF16 (bits 7-9 = 1, 10-12 = 1), MN-major operands (bits 15, 16),
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N, bool mn_major) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (mn_major ? (3u << 15) : 0u) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma_f16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, bool accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"((uint32_t)accumulate));
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t cols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t tmem, uint32_t cols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols) : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// 32 columns of the warp's 32 TMEM lanes: lane l gets its row's values.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
        "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}

// 2-D tensor map of a BF16 matrix: inner extent `inner` elements, `rows` rows
// `ld` elements apart, boxes of row_bytes / 2 x box_rows with the 64- or
// 128-byte swizzle; elements outside the extents read as zero.
bool make_map(CUtensorMap* map, const void* base, int inner, int rows, int ld, int row_bytes, int box_rows);

}  // namespace lbms
