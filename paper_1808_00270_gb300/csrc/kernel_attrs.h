// kernel_attrs.h -- attributes of kernels that launches depend on.
//
// The dynamic shared memory a kernel may use belongs to the function, not to a
// launch: set to each launch's own size, one context would lower the limit
// between another's call and its launch (contexts on other host threads), or
// leave it below what an earlier one needs.  So it is set once per device and
// function, to the most that the device gives, and never lowered.
#pragma once

#include <map>
#include <mutex>
#include <set>
#include <utility>

#include <cuda_runtime.h>

namespace gld {

// Before a launch of kern with smem bytes of dynamic shared memory (nonportable:
// in clusters of up to 16 CTAs).  Up to 32 KB no kernel here passes the 48 KB
// that every launch has (static shared memory is at most 16 KB).
inline cudaError_t allow_smem(const void* kern, size_t smem, bool nonportable = false)
{
    static std::mutex mu;
    static std::set<std::pair<int, const void*>> set;
    if (smem <= 32 * 1024 && !nonportable) return cudaSuccess;
    int dev = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (set.count({dev, kern})) return cudaSuccess;
    cudaFuncAttributes fa{};
    e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kern);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess && nonportable) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) set.insert({dev, kern});
    return e;
}

template <class... A>
cudaError_t allow_smem(void (*kern)(A...), size_t smem, bool nonportable = false)
{
    return allow_smem((const void*)kern, smem, nonportable);
}

// Threads of a kernel, in blocks of `block` without dynamic shared memory, that
// the device holds at once (0: the question failed); asked once per device and
// function.
template <class... A>
int resident_threads(void (*kern)(A...), int block)
{
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, int> known;
    int dev = 0, sms = 0, blocks = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_pair(dev, (const void*)kern);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kern, block, 0) != cudaSuccess)
        return 0;
    return known[key] = sms * blocks * block;
}

}  // namespace gld
