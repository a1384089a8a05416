// Inline-PTX wrappers for the sm_100-family tensor-core path (tcgen05 + TMEM + mbarrier), written for sm_103a.
//
// Conventions used by the kernels in this library:
//   * one CTA, cta_group::1, M = 128: accumulator row i is TMEM lane i, column j is TMEM column base + j (FP32);
//   * operands A and B come from shared memory through 64-bit matrix descriptors, K-major, no swizzle: the matrix
//     is tiled into core matrices of 8 rows x 16 bytes (128 contiguous bytes, row r at offset 16 r); the byte
//     distance between core matrices adjacent along K is the leading-dimension byte offset (LBO) and along M/N the
//     stride-dimension byte offset (SBO);
//   * the instruction descriptor selects FP32 accumulation, K-major A and B, and N, M;
//   * completion of the MMAs issued by one thread is signalled on an mbarrier by tcgen05.commit; every wait on
//     it has an iteration limit after which the kernel raises an error flag instead of spinning on.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rascal {

__device__ inline uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// whole warp: allocates ncols (power of 2, >= 32) TMEM columns, writes the base address to *dst
__device__ inline void tmem_alloc(uint32_t* dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
                 : "memory");
}
__device__ inline void tmem_relinquish() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory"); }
__device__ inline void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ inline void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ inline void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ inline void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// non-blocking test of the phase (no suspension)
__device__ inline bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; returns false on timeout. Polls with the non-blocking test and a short sleep between polls, so that
// the bound counts polls (a single poll when max_iter is 1) and a waiting warp takes few issue slots.
__device__ inline bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, uint32_t max_iter = (1u << 22)) {
    for (uint32_t it = 0; it < max_iter; ++it) {
        if (mbar_test_wait(bar, parity)) return true;
        __nanosleep(20);
    }
    return false;
}

// the same for waits inside a pipeline, which are short: polls before it sleeps
__device__ inline bool mbar_wait_spin(uint64_t* bar, uint32_t parity) {
    for (int it = 0; it < 512; ++it)
        if (mbar_test_wait(bar, parity)) return true;
    return mbar_wait_bounded(bar, parity);
}

// One lane waits for its whole warp (32 polling lanes take issue slots from the working warps); every lane gets the outcome.
// The shuffle passes it on but orders no memory: the __syncwarp does, so that what the wait acquired holds for all lanes
// before they read or refill what the barrier guards. All lanes call it; wait is false where there is nothing to wait for.
__device__ inline bool mbar_wait_warp(bool wait, uint64_t* bar, uint32_t parity) {
    bool ok = true;
    if (wait && (threadIdx.x & 31) == 0) ok = mbar_wait_spin(bar, parity);
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();
    return ok;
}

__device__ inline void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ inline void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic-proxy shared-memory writes -> visible to the tensor core (async proxy)
__device__ inline void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ inline uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version for tcgen05
    return d;                // base offset 0, no swizzle
}

// K-major operand in the 64-byte swizzled layout: 8-row atoms of 8 x 64 bytes (SBO between atoms), the 16-byte chunk
// c of row r stored at chunk c ^ ((r >> 1) & 3), as a TMA load with 64-byte swizzling writes it. The start address
// may be advanced by the K offset in bytes inside the atom; atoms start on 512-byte boundaries.
__device__ inline uint64_t smem_desc_sw64(uint32_t saddr, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;                     // leading byte offset: unused for swizzled K-major operands
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;                     // descriptor version for tcgen05
    d |= (uint64_t)4 << 61;                     // swizzling mode: 64 bytes
    return d;
}
__device__ inline uint32_t sw64_off(int row, int chunk) {
    return (uint32_t)((row >> 3) * 512 + (row & 7) * 64 + ((chunk ^ ((row >> 1) & 3)) << 4));
}

// the same with 128-byte rows: 8-row atoms of 1024 bytes, chunk c of row r at chunk c ^ (r & 7)
__device__ inline uint64_t smem_desc_sw128(uint32_t saddr, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;                     // swizzling mode: 128 bytes
    return d;
}
__device__ inline uint32_t sw128_off(int row, int chunk) {
    return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((chunk ^ (row & 7)) << 4));
}

// instruction descriptor: D FP32, A/B format (1 = BF16 for kind::f16, 2 = TF32 for kind::tf32), K-major A and B
__device__ inline uint32_t instr_desc(uint32_t ab_format, uint32_t M, uint32_t N) {
    return (1u << 4) | (ab_format << 7) | (ab_format << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

__device__ inline void mma_bf16_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ inline void mma_tf32_ss(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ inline void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 32 lanes x 32 bit, 16 consecutive columns: thread t of the warp gets row (lane base + t), columns col..col+15.
// The wait is in the same asm statement so that no use of the registers can be scheduled before it.
__device__ inline void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];\n\ttcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

// TMA: 2-D tiled load of one box into shared memory (128-byte aligned destination; the innermost coordinate times
// the element size a multiple of 16 bytes), completion counted in bytes on an mbarrier armed by expect_tx.
__device__ inline void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ inline void tma_load_2d(void* sdst, const void* tmap, int x, int y, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(sdst)),
        "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// Bulk (non-tensor) asynchronous copy shared -> global by the issuing thread: both addresses 16-byte aligned,
// size a multiple of 16 bytes. The writers of the source make their stores visible to the async proxy
// (fence_proxy_async_smem) before the barrier that precedes the issue. Completion is tracked per thread in bulk
// groups: wait_read<N> returns once at most N committed groups still read shared memory.
__device__ inline void bulk_store(void* gdst, const void* ssrc, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(gdst), "r"(smem_u32(ssrc)),
                 "r"(bytes)
                 : "memory");
}
__device__ inline void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void bulk_wait_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ inline void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// 4-byte asynchronous global -> shared copy (no register round trip, many in flight per thread); cp_async_wait_all
// then a barrier make the copies visible to the CTA.
__device__ inline void cp_async4(void* sdst, const void* gsrc) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(sdst)), "l"(gsrc) : "memory");
}
__device__ inline void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// 16-byte (L2-only) and 4-byte copies that fill the destination with zeros beyond src_bytes (0 = all zeros, nothing
// is read)
__device__ inline void cp_async16_zfill(void* sdst, const void* gsrc, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(sdst)), "l"(gsrc), "r"(src_bytes)
                 : "memory");
}
__device__ inline void cp_async4_zfill(void* sdst, const void* gsrc, uint32_t src_bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(sdst)), "l"(gsrc), "r"(src_bytes)
                 : "memory");
}
// one arrival on an mbarrier once this thread's cp.async copies so far have landed
__device__ inline void cp_async_arrive(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

}  // namespace rascal
