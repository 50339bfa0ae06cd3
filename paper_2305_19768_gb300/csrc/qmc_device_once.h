// Settings that belong to a device (a kernel's dynamic shared memory limit), made
// once for each device that is current when they are needed.
#pragma once
#include <atomic>
#include <cstdint>

// True once set() has succeeded for device `dev`; a failure is not remembered.
// `done` holds a bit per device; beyond 64 devices set() runs every time. Safe
// from several threads (set() may then run more than once for a device).
template <class F>
inline bool qmc_once_per_device(std::atomic<uint64_t> &done, int dev, F set) {
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ULL << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return true;
    if (!set()) return false;
    done.fetch_or(bit, std::memory_order_release);
    return true;
}

#if defined(__CUDACC__)
// `kernel` may use up to `bytes` of dynamic shared memory on the current device
template <class K>
inline bool qmc_allow_smem(std::atomic<uint64_t> &done, K *kernel, int bytes) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    return qmc_once_per_device(done, dev, [&] {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    });
}
#endif
