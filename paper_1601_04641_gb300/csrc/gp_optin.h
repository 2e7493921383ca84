// gp_optin.h -- a kernel's opt-in to more than 48 KB of dynamic shared memory.
//
// cudaFuncSetAttribute acts on the current device alone, and a process may
// hold handles on several: what has been opted in to is kept per device.  The
// limit only ever rises, under a lock, so that a thread's smaller launch
// cannot lower it between another thread's opt-in and launch.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>
#include <mutex>

namespace gpcn {

constexpr int kOptInDevices = 64;

class SmemOptIn {
public:
    // Calls set(bytes) unless `bytes` or more is set on device dev already
    // (each time for a device beyond those kept).
    template <class Set> cudaError_t raise(int dev, int bytes, Set set) {
        if (dev < 0 || dev >= kOptInDevices) return set(bytes);
        if (done_[dev].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
        std::lock_guard<std::mutex> lock(mutex_);
        if (done_[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
        const cudaError_t e = set(bytes);
        if (e == cudaSuccess) done_[dev].store(bytes, std::memory_order_release);
        return e;
    }

private:
    std::atomic<int> done_[kOptInDevices] = {};
    std::mutex mutex_;
};

// One SmemOptIn per kernel (a function-local static of its launcher).
template <class Kernel> inline cudaError_t opt_in_smem(SmemOptIn &kept, Kernel *kernel, size_t smem) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    return kept.raise(dev, (int)smem, [&](int bytes) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    });
}

}  // namespace gpcn
