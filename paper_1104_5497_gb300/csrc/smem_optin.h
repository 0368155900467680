// smem_optin.h -- the opt-in to more than 48 KB of dynamic shared memory, once per kernel and device.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>

// The attribute belongs to the kernel on one device: a process that uses another device afterwards
// needs it there too.  Kernel: a __global__ function; bytes: the same on every call.  Safe from
// several threads (two that come first both set it).
template <auto Kernel>
cudaError_t allow_dynamic_smem(size_t bytes) {
    static std::atomic<unsigned long long> done{0};   // a bit per device; beyond 64 it is set on every call
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}
