// What the host side keeps about devices, for every thread and every device of the process.
#pragma once
#include <cuda_runtime.h>
#include <atomic>
#include <mutex>

namespace goq {

constexpr int kMaxDevices = 64;   // (beyond them nothing is kept)

// SMs of the current device, 148 where it cannot be asked. A device's slot goes from 0 to its one value: threads that come first together write the same.
inline int sm_count() {
    static std::atomic<int> known[kMaxDevices];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 148;
    const bool kept = dev >= 0 && dev < kMaxDevices;
    if (kept && (n = known[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
    if (kept) known[dev].store(n, std::memory_order_relaxed);
    return n;
}

// The dynamic shared memory limit of a kernel is a per-device attribute: remember, per device, the largest size it has been raised to (one cache object per
// kernel instantiation, a function-local static at the call site). Raised by one thread at a time: a smaller call that set the attribute between another
// thread's setting and its note of it would leave a limit below the size that is noted.
struct SmemAttrCache {
    std::atomic<size_t> set[kMaxDevices] = {};
    std::mutex raise;
};
template <class Kernel>
inline cudaError_t ensure_dynamic_smem(Kernel kernel, size_t smem, SmemAttrCache& cache) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool tracked = dev >= 0 && dev < kMaxDevices;
    if (tracked && smem <= cache.set[dev].load(std::memory_order_acquire)) return cudaSuccess;
    std::lock_guard<std::mutex> lock(cache.raise);
    if (tracked && smem <= cache.set[dev].load(std::memory_order_relaxed)) return cudaSuccess;
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess && tracked) cache.set[dev].store(smem, std::memory_order_release);
    return e;
}

}  // namespace goq
