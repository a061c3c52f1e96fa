// A kernel's limit of dynamic shared memory.  The limit belongs to the kernel in a device's
// context, and handles of several graphs, created and used by several host threads, share it: it
// is only ever raised, and reading, comparing and setting it is one step (two threads that both
// read the old value could otherwise leave the smaller of their two sizes, and the larger handle's
// launches would be refused).
#pragma once

#include <cuda_runtime_api.h>

#include <mutex>

namespace qldpc {

// Raises the limit of `fn` on the current device to `smem` bytes.
inline cudaError_t allow_smem(const void *fn, size_t smem) {
    static std::mutex lock;
    const std::lock_guard<std::mutex> held(lock);
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, fn);
    if (e != cudaSuccess || (size_t)a.maxDynamicSharedSizeBytes >= smem) return e;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

}  // namespace qldpc
