// tc.cuh -- 5th-generation tensor core (tcgen05) building blocks for sm_103a: tensor
// memory allocation, shared-memory matrix descriptors, BF16 MMA with FP32 accumulation
// in tensor memory, completion tracking through an mbarrier, and accumulator loads.
//
// Operand layout used throughout ("K-major, no swizzle"): a matrix of R rows x K
// columns (BF16) is stored as 8-row x 8-column core matrices of 128 contiguous bytes
// (row r of a core matrix at byte 16 r). Core matrices adjacent along K are kLbo = 128
// bytes apart; adjacent 8-row groups are sbo = (K / 8) * 128 bytes apart. So element
// (r, k) sits at byte   (r / 8) * sbo + (k / 8) * 128 + (r % 8) * 16 + (k % 8) * 2.
// One MMA consumes K = 16 columns: its operand descriptor starts 256 bytes further per
// K step.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pic {
namespace tc {

constexpr uint32_t kLbo = 128;

__host__ __device__ __forceinline__ uint32_t canon_offset(int r, int k, int K) {
    return (uint32_t)((r >> 3) * (K >> 3) * 128 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// The same matrix with its rows contiguous ("MN-major, no swizzle"): core matrices of 8
// rows x 8 columns whose columns are 16 bytes of 8 rows each. With kLbo = 128 bytes between
// core matrices along K and (K / 8) * 128 between 8-row groups, element (r, k) sits at
// (r / 8) * sbo + 16 k + (r % 8) * 2, so 8 rows of one column are one 16-byte store. One MMA
// still moves 256 bytes along K.
__host__ __device__ __forceinline__ uint32_t mn_offset(int r, int k, int K) {
    return (uint32_t)((r >> 3) * (K >> 3) * 128 + k * 16 + (r & 7) * 2);
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor (K-major, no swizzle): start address, leading byte
// offset (between core matrices along K), stride byte offset (between 8-row groups),
// descriptor version 1.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// Instruction descriptor of kind::f16: D in FP32, A and B in BF16, both K-major,
// shape M x N.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The same with both operands MN-major.
__host__ __device__ constexpr uint32_t make_idesc_mn(int M, int N) { return make_idesc(M, N) | (1u << 15) | (1u << 16); }

// Whole warp: allocate ncols (power of two >= 32) tensor-memory columns; the address is
// written to *dst (shared memory).
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(dst)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
}

// Whole warp.
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}

// Bounded wait for phase `phase` of the barrier; false if the limit ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase) {
    for (int it = 0; it < (1 << 24); ++it)
        if (mbar_try_wait(bar, phase)) return true;
    return false;
}

// Non-blocking test whether phase `phase` of the barrier has completed.
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}

// The wait with a caller's limit: `limit` non-blocking polls when limit > 0 (a short
// limit lets a test make the wait run out), the default bound of mbar_wait otherwise.
// After a false return the operation is still in flight: the caller drains it with
// mbar_wait before it frees the memory the operation uses.
__device__ __forceinline__ bool mbar_wait_lim(uint64_t* bar, uint32_t phase, uint32_t limit) {
    if (limit == 0) return mbar_wait(bar, phase);
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_test_wait(bar, phase)) return true;
    return false;
}

// D (tensor memory) = A B^T (+ D when accumulate != 0), A and B from descriptors.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// The barrier receives one arrival when all MMAs issued so far by this thread finish.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                     smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }
// Make this thread's generic-proxy shared-memory writes visible to the tensor cores.
__device__ __forceinline__ void fence_smem_to_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// 16 consecutive FP32 accumulator columns of the warp's 32 tensor-memory lanes: thread t
// of warp w gets lane 32 w + t.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; i++) v[i] = __uint_as_float(r[i]);
}

}  // namespace tc
}  // namespace pic
