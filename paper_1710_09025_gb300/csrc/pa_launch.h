// pa_launch.h -- host helpers of the kernel launches.
#pragma once
#include <atomic>
#include <cuda_runtime.h>

namespace pa {

// dynamic shared memory of a kernel, asked for once per device (done: a bit each)
template <class Kernel>
inline cudaError_t allow_smem(Kernel kern, int bytes, std::atomic<unsigned long long>& done)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || (dev < 64 && done.load(std::memory_order_acquire) >> dev & 1)) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && dev < 64) done.fetch_or(1ull << dev, std::memory_order_release);
    return e;
}

}  // namespace pa
