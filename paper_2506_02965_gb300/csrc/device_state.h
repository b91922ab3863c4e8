// Host: what the launchers look up or set once per device of the process (a function attribute
// and the SM count belong to the device that is current when they are set or read).
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace moe {

constexpr int kMaxDevices = 64;  // devices with a place of their own; others are looked up each time

// The current device, or -1.
inline int current_device() {
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess ? dev : -1;
}

// SMs of the current device (148 without one, for host-only rules). Two threads on their first call
// both look it up and store the same value.
inline int sm_count() {
    static std::atomic<int> count[kMaxDevices] = {};
    const int dev = current_device();
    const bool kept = dev >= 0 && dev < kMaxDevices;
    int n = kept ? count[dev].load(std::memory_order_relaxed) : 0;
    if (n > 0) return n;
    if (dev < 0 || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
    if (kept) count[dev].store(n, std::memory_order_relaxed);
    return n;
}

// Runs `set` once per device and kernel: for attributes that cudaFuncSetAttribute gives a kernel on
// the current device only.
template <auto Kernel, typename Set>
inline cudaError_t once_per_device(Set set) {
    static std::atomic<bool> done[kMaxDevices] = {};
    const int dev = current_device();
    const bool kept = dev >= 0 && dev < kMaxDevices;
    if (kept && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e = set();
    if (e == cudaSuccess && kept) done[dev].store(true, std::memory_order_release);
    return e;
}

// Lets Kernel use `bytes` of dynamic shared memory on the current device.
template <auto Kernel>
inline cudaError_t allow_dynamic_smem(size_t bytes) {
    return once_per_device<Kernel>(
        [=] { return cudaFuncSetAttribute((const void*)Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); });
}

}  // namespace moe
