// Raising a kernel's dynamic shared memory beyond the default.
#pragma once

#include <cstddef>
#include <mutex>

#include <cuda_runtime.h>

namespace vqe {

// Static shared memory of a kernel: a property of the compiled code, looked up once.
inline cudaError_t static_smem_of(const void *kern, int &bytes) {
    struct Entry {
        const void *kern;
        int bytes;
    };
    static std::mutex mu;
    static Entry known[128];
    static int n_known = 0;
    const std::lock_guard<std::mutex> lock(mu);
    for (int i = 0; i < n_known; ++i)
        if (known[i].kern == kern) {
            bytes = known[i].bytes;
            return cudaSuccess;
        }
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, kern);
    if (e != cudaSuccess) return e;
    bytes = (int)a.sharedSizeBytes;
    if (n_known < 128) known[n_known++] = Entry{kern, bytes};
    return cudaSuccess;
}

// Lets `kern` launch with `smem` bytes of dynamic shared memory.  The default 48 KiB
// hold the static part too, so larger launches ask from 40 KiB on.  The limit belongs
// to the kernel in the whole process, and handles on other threads launch it with
// other sizes: it is always set to the most the device has, never to this launch's
// size, which would refuse a larger launch that another thread is about to make.
inline cudaError_t allow_smem(const void *kern, size_t smem) {
    if (smem <= 40 * 1024) return cudaSuccess;
    int device = 0, most = 0, used = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
    if (e == cudaSuccess) e = static_smem_of(kern, used);
    if (e != cudaSuccess) return e;
    if (smem > (size_t)(most - used)) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most - used);
}

}  // namespace vqe
