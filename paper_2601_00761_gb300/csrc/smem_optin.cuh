// smem_optin.cuh -- a kernel's opt-in to more than 48 KB of dynamic shared memory.
//
// cudaFuncSetAttribute applies to the current device alone, and a later call
// replaces the limit of an earlier one. Each launch site therefore keeps one of
// these as a function static: it asks once per device, and asks again only for
// more, under a lock, so that of two threads with different needs the larger
// limit stays. A launch with nothing to ask for costs a cudaGetDevice and a load.
#pragma once

#include <atomic>
#include <mutex>

#include <cuda_runtime_api.h>

namespace sre {

class SmemOptIn {
public:
    cudaError_t allow(const void *kernel, size_t bytes) {
        int dev = 0;
        const cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= DEVICES) return set(kernel, bytes);
        if (granted_[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
        std::lock_guard<std::mutex> lk(mu_);
        if (granted_[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
        const cudaError_t s = set(kernel, bytes);
        if (s == cudaSuccess) granted_[dev].store(bytes, std::memory_order_release);
        return s;
    }

private:
    static constexpr int DEVICES = 64;
    static cudaError_t set(const void *kernel, size_t bytes) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    }
    std::mutex mu_;
    std::atomic<size_t> granted_[DEVICES] = {};
};

} // namespace sre
