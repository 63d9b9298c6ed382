// Blackwell tensor-core primitives (tcgen05, TMEM, mbarrier) in inline PTX, used by the split-slice
// products of tc_gemm.cu.  One CTA issues its MMAs from one thread; the accumulator lives in tensor
// memory (TMEM: 128 lanes x 512 columns of 32 bits per SM), allocated and freed by one warp.
//
// Shared-memory operands are K-major without swizzle: the canonical layout is a grid of "core
// matrices" of 8 rows x 16 bytes (8 x 8 bf16), each 128 contiguous bytes; the descriptor gives the
// byte distance between core matrices adjacent along K (leading byte offset) and along M or N
// (stride byte offset).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace hbsd {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start >> 4 in bits 0-13, leading byte offset >> 4 in 16-29,
// stride byte offset >> 4 in 32-45, the descriptor version 1 in bits 46-47, no swizzle (bits 61-63 = 0)
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16 with bf16 A and B, FP32 accumulator, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// the same with FP16 A and B
__host__ __device__ constexpr uint32_t idesc_f16_f32(int M, int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_alloc(uint32_t* slot_smem, uint32_t ncols) {   // one full warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(slot_smem)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {   // the allocating warp
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols));
}
__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::); }
// generic-proxy stores to shared memory made visible to the tensor core's (async proxy) reads
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// D(tmem) (+)= A(smem) B(smem)^T, issued by one thread
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}
// the mbarrier completes (one arrival) when every MMA this thread issued before has finished
__device__ __forceinline__ void mma_commit(uint64_t* mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                     smem_u32(mbar)));
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(mbar)), "r"(count));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* mbar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait: false when the phase did not complete within about `limit_ns` of %globaltimer
__device__ __forceinline__ bool mbar_wait(uint64_t* mbar, uint32_t parity, uint64_t limit_ns) {
    if (mbar_try_wait(mbar, parity)) return true;   // the timer is read only by a wait that has to spin
    uint64_t t0;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t0));
    for (;;) {
        if (mbar_try_wait(mbar, parity)) return true;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
        if (t - t0 > limit_ns) return false;
    }
}

// the same for a whole warp, which goes on in step whatever comes: tcgen05.ld and the warp barriers after a wait need all
// lanes, and a limit that only some of them reached would split the warp for good.  A lane that gives up sets *failed
// (shared memory), which also ends every later wait of the CTA that has to spin; the caller drops its results.  (A
// vote after each wait instead: the Gram 1.6% slower; the spin inlined: 1.3%.)
static __device__ __noinline__ void warp_wait_spin(uint64_t* mbar, uint32_t parity, uint64_t limit_ns, int* failed) {
    uint64_t t0;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t0));
    for (;;) {
        if (mbar_try_wait(mbar, parity) || *reinterpret_cast<volatile int*>(failed) != 0) return;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
        if (t - t0 > limit_ns) *reinterpret_cast<volatile int*>(failed) = 1;
    }
}
__device__ __forceinline__ void warp_wait(uint64_t* mbar, uint32_t parity, uint64_t limit_ns, int* failed) {
    if (!mbar_try_wait(mbar, parity)) warp_wait_spin(mbar, parity, limit_ns, failed);
}
// by the issuing thread, when it is done or has given up: its MMAs end (a fresh mbarrier of one arrival) before the CTA
// frees tensor memory and leaves its shared memory, whatever the other warps still wait for
__device__ __forceinline__ void mma_drain(uint64_t* mbar, uint64_t limit_ns) {
    mma_commit(mbar);
    (void)mbar_wait(mbar, 0u, limit_ns);
}

// 32 lanes (this warp's quarter of TMEM) x 16 columns of 32-bit values starting at taddr
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// byte offset of element (row, k) in a K-major no-swizzle tile of 16 K-columns: core matrices
// (row / 8, k / 8) at (k / 8) * 128 + (row / 8) * 256, rows of 16 bytes inside
__device__ __forceinline__ uint32_t kmajor16_offset(int row, int k) {
    return (uint32_t)((k >> 3) * 128 + (row >> 3) * 256 + (row & 7) * 16 + (k & 7) * 2);
}

}  // namespace tc
}  // namespace hbsd
