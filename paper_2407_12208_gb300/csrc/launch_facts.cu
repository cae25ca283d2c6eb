// launch_facts.cu -- what the launchers ask of the runtime about a kernel,
// remembered per device (internal.h).
#include <map>
#include <mutex>
#include <tuple>

#include "internal.h"

namespace km {

namespace {
std::mutex g_mu;
std::map<std::tuple<int, const void*>, cudaError_t> g_smem;             // (device, kernel): limit raised
std::map<std::tuple<int, const void*, int, size_t>, int> g_per_sm;      // (device, kernel, block, bytes)
}  // namespace

cudaError_t allow_max_smem_of(const void* func) try {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_mu);
    const auto key = std::make_tuple(dev, func);
    if (g_smem.count(key)) return cudaSuccess;
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, func);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxBlockSmem - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess) g_smem[key] = e;
    return e;
} catch (...) {
    return cudaErrorMemoryAllocation;
}

cudaError_t blocks_per_sm_of(const void* func, int block, size_t smem, int* out) try {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_mu);
    const auto key = std::make_tuple(dev, func, block, smem);
    const auto it = g_per_sm.find(key);
    if (it != g_per_sm.end()) {
        *out = it->second;
        return cudaSuccess;
    }
    int n = 1;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, func, block, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) n = 1;
    if (g_per_sm.size() > 4096) g_per_sm.clear();  // (sizes vary with d and k)
    g_per_sm[key] = *out = n;
    return cudaSuccess;
} catch (...) {
    return cudaErrorMemoryAllocation;
}

}  // namespace km
