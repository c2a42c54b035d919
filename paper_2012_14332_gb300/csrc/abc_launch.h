// abc_launch.h -- launch helpers shared by the kernels' translation units.
#pragma once
#include <cstddef>
#include <map>
#include <mutex>
#include <tuple>
#include <utility>
#include <cuda_runtime.h>

#include "abc_kernels.h"

namespace abcgb {

// The kernel's dynamic shared-memory limit is one value per kernel and device:
// it is only ever raised, to the largest size launched so far, so a call with
// a shorter horizon never lowers it below what a longer one needs. Up to 32 KB
// the default limit (48 KB with the kernel's static shared memory) always holds.
template <typename K>
cudaError_t raise_smem_limit(K kernel, size_t smem)
{
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, size_t> limit;   // largest limit set per kernel and device
    if (smem <= 32 * 1024) return cudaSuccess;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    size_t& lim = limit[std::make_pair((const void*)kernel, dev)];
    if (lim < smem) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        lim = smem;
    }
    return cudaSuccess;
}

// Resident blocks per SM times the SM count, for a kernel, block size, dynamic
// shared memory size and device; looked up once and cached (the launch path
// then makes no occupancy query).
template <typename K>
cudaError_t grid_for(K kernel, size_t smem, int* grid, int threads = kBlockThreads)
{
    static std::mutex mu;
    static std::map<std::tuple<const void*, int, int, size_t>, int> cache;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = raise_smem_limit(kernel, smem);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_tuple((const void*)kernel, dev, threads, smem);
    auto it = cache.find(key);
    if (it != cache.end()) {
        *grid = it->second;
        return cudaSuccess;
    }
    int sms = 0, per_sm = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    *grid = sms * (per_sm > 0 ? per_sm : 1);
    cache[key] = *grid;
    return cudaSuccess;
}

#define ABC_MODE_DISPATCH(fn, mode, ...)                        \
    ((mode) == kFast ? fn<kFast>(__VA_ARGS__)                   \
     : (mode) == kExact ? fn<kExact>(__VA_ARGS__)               \
     : (mode) == (kFast | kLiteral) ? fn<kFast | kLiteral>(__VA_ARGS__) \
                                  : fn<kExact | kLiteral>(__VA_ARGS__))

}  // namespace abcgb
