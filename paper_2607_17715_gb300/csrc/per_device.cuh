// What the launchers set up or ask once on each device: kernel attributes (a shared-memory opt-in, a
// register count) belong to a device, and a process may hold contexts on several.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace c2kv {
namespace {

// make() on the current device: called at a device's first use and kept (threads that meet there may
// each call it; it gives the same value).  T: a small value type.
template <class T>
class PerDevice {
public:
    template <class Make>
    T get(const Make& make) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return make();
        if (state_[dev].load(std::memory_order_acquire) == kKept) return value_[dev];
        const T v = make();
        int empty = kEmpty;
        if (state_[dev].compare_exchange_strong(empty, kWriting)) {
            value_[dev] = v;
            state_[dev].store(kKept, std::memory_order_release);
        }
        return v;
    }

private:
    static constexpr int kDevices = 64;        // (beyond: made at each call)
    enum { kEmpty, kWriting, kKept };
    std::atomic<int> state_[kDevices] = {};
    T value_[kDevices] = {};
};

// SMs of the current device.
inline int device_sms() {
    static PerDevice<int> sms;
    return sms.get([] {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1)
            return 1;
        return n;
    });
}

// `kernel` may take `bytes` of dynamic shared memory on the current device (`kept`: one per kernel).
inline cudaError_t opt_in_smem(PerDevice<cudaError_t>& kept, const void* kernel, size_t bytes) {
    return kept.get([&] { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); });
}

}  // namespace
}  // namespace c2kv
