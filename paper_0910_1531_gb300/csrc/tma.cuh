// Tensor Memory Accelerator (TMA) tile copies and mbarrier waits, in inline PTX.
//
// Column tiles of the half spectra are moved between global and shared memory with
// cp.async.bulk.tensor (one instruction per tile, issued by one thread): loads complete
// on an mbarrier (transaction-count based), stores are tracked with bulk async groups.
// Every wait is bounded: after kMaxSpins polls it gives up, and the kernel reports
// DEV_TIMEOUT instead of spinning forever.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace tma {

constexpr long long kMaxSpins = 1LL << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// Make this thread's generic-proxy shared-memory writes visible to the async proxy (TMA store).
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        "  .reg .pred p;\n"
        "  mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "  selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase with the given parity to complete; false if `polls` polls ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long polls = kMaxSpins) {
    for (long long i = 0; i < polls; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// 3D tiled load global -> shared; completes `bar`'s transaction count.  x must be a multiple
// of 16 bytes / element size (the callers' tile origins are multiples of the tile width).
__device__ __forceinline__ void load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// The same for a 4D tensor.
__device__ __forceinline__ void load_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int c, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(c), "r"(smem_u32(bar))
        : "memory");
}

// 1D bulk copy global -> shared of `bytes` (a multiple of 16; both addresses 16-byte aligned);
// completes `bar`'s transaction count.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Per-thread asynchronous copy of 16 bytes global -> shared (cp.async, cached in L2 only; both
// addresses 16-byte aligned).  The issuing thread commits its copies as a group and waits for
// them with cp_wait_all(); like a load, such a copy always completes (no bound needed).
__device__ __forceinline__ void cp16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 3D tiled store shared -> global (elements outside the tensor are not written).
__device__ __forceinline__ void store_3d(const CUtensorMap* map, int x, int y, int z, const void* src) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];"
                 ::"l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_u32(src))
                 : "memory");
}

__device__ __forceinline__ void store_4d(const CUtensorMap* map, int x, int y, int z, int c, const void* src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];"
                 ::"l"(map), "r"(x), "r"(y), "r"(z), "r"(c), "r"(smem_u32(src))
                 : "memory");
}

__device__ __forceinline__ void commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// the bulk stores committed so far have finished reading shared memory
__device__ __forceinline__ void wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// the bulk stores committed so far are complete
__device__ __forceinline__ void wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

}  // namespace tma

// Host: encode a 3D tiled tensor map over 8-byte elements (a float2, or half a double2).
// dims/strides in elements/bytes as cuTensorMapEncodeTiled wants them.
cudaError_t tma_encode_3d(CUtensorMap* map, void* base, unsigned long long d0, unsigned long long d1,
                          unsigned long long d2, unsigned long long stride1_bytes, unsigned long long stride2_bytes,
                          unsigned b0, unsigned b1, unsigned b2);

// The same for a 4D tensor (strides of the dimensions past the innermost).
cudaError_t tma_encode_4d(CUtensorMap* map, void* base, const unsigned long long dims[4],
                          const unsigned long long stride_bytes[3], const unsigned box[4]);
