// Host state of the kernel launchers, kept per device and safe with several
// threads: the shared-memory opt-in of a kernel and the SM count.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>

namespace hatq {

constexpr int kMaxDev = 64;
// Dynamic shared memory a kernel may ask for: 227 KB less 1 KB for its static variables.
constexpr int kMaxDynamicSmem = 227 * 1024 - 1024;

inline cudaError_t current_device(int *dev) {
    const cudaError_t e = cudaGetDevice(dev);
    if (e != cudaSuccess) return e;
    return *dev < 0 || *dev >= kMaxDev ? cudaErrorInvalidDevice : cudaSuccess;
}

// The opt-in of one kernel. Every caller sets the same value, the most that any
// launch may need, so neither the order nor the number of threads that set it
// matters; with the size of the launch at hand, two threads could leave the
// smaller size set last and every larger launch of the kernel would fail.
class SmemOptIn {
    std::atomic<bool> done_[kMaxDev] = {};

public:
    cudaError_t set(int dev, const void *kernel) {
        if (done_[dev].load(std::memory_order_acquire)) return cudaSuccess;
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamicSmem);
        if (e == cudaSuccess) done_[dev].store(true, std::memory_order_release);
        return e;
    }
};

// SMs of a device (at least 1).
inline cudaError_t device_sms(int dev, int *sms) {
    static std::atomic<int> count[kMaxDev] = {};
    *sms = count[dev].load(std::memory_order_relaxed);
    if (*sms) return cudaSuccess;
    const cudaError_t e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (*sms < 1) *sms = 1;
    count[dev].store(*sms, std::memory_order_relaxed);
    return cudaSuccess;
}

}  // namespace hatq
