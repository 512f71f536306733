// smem_optin.cuh -- dynamic shared memory above the default 48 KB.
//
// The limit is an attribute of a kernel on one device, so a process with plans
// on several devices raises it on each.  A kernel's launcher calls this before
// every launch with the kernel's constant size: nothing where 48 KB do, else
// one look at the current device and at a bit per kernel and device.  A failure
// is not remembered; threads that race raise the limit twice to the same value.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace vloc {

template <auto Kernel> cudaError_t smem_optin(size_t bytes) {
    if (bytes <= 48 * 1024) return cudaSuccess;
    static std::atomic<unsigned long long> raised{0};  // bit per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e) return e;
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
    if (raised.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) raised.fetch_or(bit, std::memory_order_release);
    else cudaGetLastError();  // reported here, not by a later check
    return e;
}

}  // namespace vloc
