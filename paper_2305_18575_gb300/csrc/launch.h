// launch.h -- launch attributes and occupancy of the search kernels (host side).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>
#include <utility>

namespace rei {

// the dynamic shared memory limit of a kernel, raised once per device to the
// opt-in maximum (so that launches need no attribute call), and occupancy
// queries remembered per (device, kernel, threads, shared memory)
inline std::mutex g_attr_mu;
inline std::map<std::pair<int, const void *>, bool> g_attr_set;
inline std::map<std::tuple<int, const void *, uint32_t, size_t>, int> g_occ;

inline cudaError_t prepare(const void *fn) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_attr_mu);
    auto key = std::make_pair(dev, fn);
    if (g_attr_set.count(key)) return cudaSuccess;
    int optin = 0;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e != cudaSuccess) return e;
    g_attr_set[key] = true;
    return cudaSuccess;
}

// the largest dynamic shared memory one launch of `fn` can take on the
// current device: the opt-in maximum per CTA less the kernel's static shared
// memory
inline cudaError_t smem_max_of(const void *fn, size_t *bytes) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, fn);
    if (e != cudaSuccess) return e;
    *bytes = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
    return cudaSuccess;
}

inline cudaError_t occupancy(const void *fn, uint32_t threads, size_t smem, int *bps) {
    cudaError_t e = prepare(fn);
    if (e != cudaSuccess) return e;
    int dev = 0;
    cudaGetDevice(&dev);
    {
        std::lock_guard<std::mutex> lk(g_attr_mu);
        auto it = g_occ.find(std::make_tuple(dev, fn, threads, smem));
        if (it != g_occ.end()) {
            *bps = it->second;
            return cudaSuccess;
        }
    }
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, fn, (int)threads, smem);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_attr_mu);
    g_occ[std::make_tuple(dev, fn, threads, smem)] = *bps;
    return cudaSuccess;
}

}  // namespace rei
