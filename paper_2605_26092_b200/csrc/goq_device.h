// What the host side keeps about devices, for every thread and every device of the process.
#pragma once
#include <cuda_runtime.h>
#include <atomic>

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

}  // namespace goq
