// A kernel's limit of dynamic shared memory, set once per device.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdint>

namespace cs {

// cudaFuncSetAttribute holds for the current device alone, so a process with
// contexts on several devices has to set it on each: `done` (one per kernel, a
// function-local static) holds a bit for every device it is set on. Two threads
// may both find it unset; both set it. Devices from the 64th on set it at every
// launch.
inline void allow_smem(std::atomic<uint64_t> &done, const void *kernel, int bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess)
        done.fetch_or(bit, std::memory_order_release);
}

}  // namespace cs
