// fr_smem.h -- opting kernels in to their dynamic shared memory.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

// More than 48 KB per CTA (static and dynamic) has to be allowed, and that holds for a kernel on the device that
// is current at the call: one object per kernel, which asks once for each device it is launched on.
// A device beyond the 64 it remembers, or a call that failed, is asked for again.
class SmemOptIn {
    std::atomic<uint64_t> done_{0};

public:
    template <typename K>
    void operator()(K *kernel, size_t bytes)
    {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess) return;   // (the launch reports it)
        const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
        if (done_.load(std::memory_order_acquire) & bit) return;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess)
            done_.fetch_or(bit, std::memory_order_release);
    }
};
