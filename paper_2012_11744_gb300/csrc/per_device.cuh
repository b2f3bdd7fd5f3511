// What a process does once on each device.  Function attributes and occupancy
// belong to a device and a kernel; contexts on several devices and several
// threads share the library, so nothing of the kind is kept in a plain static.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstddef>

namespace paris {

constexpr int kMaxDevices = 64;  // further devices ask each time

// The devices on which a kernel has been let use more than 48 KB of dynamic
// shared memory (a static of the place that launches it).
struct SmemOptIn {
    std::atomic<bool> done[kMaxDevices];
};

// Lets the kernel use up to `bytes` of it on the current device; the same
// bytes in all calls for a kernel.
inline cudaError_t allow_smem(SmemOptIn& o, const void* kernel, size_t bytes) {
    int dev = -1;
    const cudaError_t g = cudaGetDevice(&dev);
    if (g != cudaSuccess) return g;
    const bool kept = dev >= 0 && dev < kMaxDevices;
    if (kept && o.done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && kept) o.done[dev].store(true, std::memory_order_release);
    return e;
}

// One number per device (0: not asked yet).
struct DeviceValue {
    std::atomic<int> v[kMaxDevices];
};

// The current device's value, from ask(dev) at first; 1 if that fails.
template <typename Ask>
int device_value(DeviceValue& d, Ask ask) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) {
        cudaGetLastError();
        return 1;
    }
    const bool kept = dev < kMaxDevices;
    int n = kept ? d.v[dev].load(std::memory_order_relaxed) : 0;
    if (n > 0) return n;
    n = ask(dev);
    if (n < 1) {
        cudaGetLastError();
        return 1;
    }
    if (kept) d.v[dev].store(n, std::memory_order_relaxed);
    return n;
}

}  // namespace paris
