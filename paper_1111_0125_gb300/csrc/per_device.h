// Values that belong to a device, made on their first use there: kernel
// attributes (a grant on one device says nothing about the next) and
// occupancies.  A handle may live on any device of the process.
#pragma once

#include <mutex>

#include <cuda_runtime.h>

namespace stg {

constexpr int kMaxDevices = 64;

// make() for device `dev`, called until it succeeds (a value that is not T{})
// and then kept.  One set of values per call site: F is its lambda's type.
template <class F>
auto per_device(int dev, const F &make) -> decltype(make())
{
    typedef decltype(make()) T;
    static std::mutex mutex;
    static T value[kMaxDevices] = {};
    if (dev < 0 || dev >= kMaxDevices) return make();
    std::lock_guard<std::mutex> lock(mutex);
    if (value[dev] == T{}) value[dev] = make();
    return value[dev];
}

// the same for the current device
template <class F>
auto per_device(const F &make) -> decltype(make())
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return {};
    return per_device(dev, make);
}

// streaming multiprocessors of the current device
inline int num_sms()
{
    const int n = per_device([] {
        int dev = 0, m = 0;
        cudaGetDevice(&dev);
        return cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? m : 0;
    });
    return n > 0 ? n : 152;
}

// true where `kernel` may use `smem` bytes of dynamic shared memory on the
// current device
template <class K>
bool grant_smem(K *kernel, int smem)
{
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
}

}  // namespace stg
