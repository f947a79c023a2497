// State that belongs to a device's copy of the library's code: set once per device, not once per process, since handles
// of one process may live on several devices.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>

namespace ddamg {

// once(f) runs f on the first call with each current device, until f returns 0; returns f's value, 0 when there was
// nothing to do, or the (positive) CUDA error that hid the device.  Any thread may call: two that meet both run f.
// (Devices numbered 64 and up run it on every call.)
struct DeviceOnce {
    std::atomic<unsigned long long> done{0};
    template <class F>
    int operator()(F f) {
        int dev = 0;
        if (const cudaError_t e = cudaGetDevice(&dev)) return (int)e;
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
        if (done.load(std::memory_order_acquire) & bit) return 0;
        const int rc = f();
        if (rc == 0) done.fetch_or(bit, std::memory_order_release);
        return rc;
    }
};

// Lets Kernel take up to `bytes` of dynamic shared memory on the current device (more than 48 KB needs asking for).
template <auto Kernel>
inline cudaError_t allow_smem(int bytes) {
    static DeviceOnce once;
    return (cudaError_t)once(
        [&] { return (int)cudaFuncSetAttribute(reinterpret_cast<const void*>(Kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

}  // namespace ddamg
