// Facts and settings that belong to a device, not to the process: a kernel's shared-memory opt-in
// (cudaFuncSetAttribute sets it for the current device only), the SM count.  Host code, no kernels.
#pragma once
#include <cuda_runtime_api.h>

#include <mutex>

namespace mone {

// A value for each device, made by `init(T&)` the first time it is asked for with that device current
// (a driver call on every launch would cost more than a small kernel).  A failed init is reported and
// tried again by the next call.  Safe from several threads.
template <typename T>
class PerDevice {
    static constexpr int kMax = 64;
    std::mutex mu_;
    bool done_[kMax] = {};
    T v_[kMax] = {};

public:
    template <typename Init>
    cudaError_t get(const T** out, Init&& init) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kMax) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lk(mu_);
        if (!done_[dev]) {
            T v{};
            if ((e = init(v)) != cudaSuccess) return e;
            v_[dev] = v;
            done_[dev] = true;
        }
        *out = &v_[dev];  // never written again
        return cudaSuccess;
    }
};

// Dynamic shared memory of `kernel` opted in to on the current device; `once` belongs to the kernel and `smem`
// is the same on every call.
struct SmemOptIn {};
inline cudaError_t smem_opt_in(const void* kernel, size_t smem, PerDevice<SmemOptIn>& once) {
    const SmemOptIn* v;
    return once.get(&v, [&](SmemOptIn&) { return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); });
}

// Multiprocessors of the current device.
inline cudaError_t sm_count(int* n) {
    static PerDevice<int> sms;
    const int* v;
    const cudaError_t e = sms.get(&v, [](int& s) {
        int dev = 0;
        const cudaError_t r = cudaGetDevice(&dev);
        return r != cudaSuccess ? r : cudaDeviceGetAttribute(&s, cudaDevAttrMultiProcessorCount, dev);
    });
    if (e == cudaSuccess) *n = *v;
    return e;
}

}  // namespace mone
