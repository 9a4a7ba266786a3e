// Launch helpers shared by the launchers of the pass kernels.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace {
// Allow each kernel the device's opt-in shared memory per block minus its static shared memory.
template <typename K> cudaError_t set_max_smem(K kernel) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

// SMs of the current device.
inline int sm_count() {
    int dev = 0, n = 1;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) n = 1;
    return n;
}

// Blocks of a persistent kernel that fit on the GPU at once (at least one per SM).  The answers for
// the kernels a thread launched last are kept: a plan launches few kernels, each with one
// shared-memory size, many times.
inline int resident_blocks_of(const void* kernel, int threads, size_t smem) {
    struct Entry {
        const void* kernel;
        size_t smem;
        int device, threads, blocks;
    };
    constexpr int kEntries = 16;
    thread_local Entry cache[kEntries] = {};
    thread_local int next = 0;
    int dev = 0, sms = 1, occ = 0;
    cudaGetDevice(&dev);
    for (const Entry& e : cache)
        if (e.kernel == kernel && e.smem == smem && e.threads == threads && e.device == dev) return e.blocks;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
    cache[next] = {kernel, smem, dev, threads, sms * (occ < 1 ? 1 : occ)};
    const int blocks = cache[next].blocks;
    next = (next + 1) % kEntries;
    return blocks;
}
template <typename... KArgs> int resident_blocks(void (*kernel)(KArgs...), int threads, size_t smem) {
    return resident_blocks_of((const void*)kernel, threads, smem);
}
}  // namespace
