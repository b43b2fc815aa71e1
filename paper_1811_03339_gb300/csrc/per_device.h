// What a launch needs to know of or to set on the current device, once per device: function
// attributes and SM counts belong to a device, so a process-wide flag would leave a second device
// without them.  Safe from several host threads; the lookups take about 0.1 us.
#pragma once

#include <cuda_runtime.h>

#include <stddef.h>

#include <map>
#include <mutex>
#include <set>
#include <utility>

namespace fem3 {

// the current device's SM count
inline cudaError_t device_sms(int *sms) {
    static std::mutex mu;
    static std::map<int, int> known;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    const auto it = known.find(dev);
    if (it != known.end()) {
        *sms = it->second;
        return cudaSuccess;
    }
    e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) known[dev] = *sms;
    return e;
}

// lets launches of `kernel` on the current device take up to `bytes` of dynamic shared memory
// (always the same number for a kernel)
inline cudaError_t device_smem(const void *kernel, size_t bytes) {
    static std::mutex mu;
    static std::set<std::pair<int, const void *>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    if (done.count({dev, kernel})) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) done.insert({dev, kernel});
    return e;
}

}  // namespace fem3
