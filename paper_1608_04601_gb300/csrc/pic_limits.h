// pic_limits.h -- dynamic shared-memory limits of the kernels (host code).
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>
#include <vector>

namespace pic {

// Raises a kernel's dynamic shared-memory limit on the current device to at least `bytes`, once per (kernel,
// device, size): the attribute belongs to one device, so a context on another one sets its own. Kernels are
// told apart by their address (instantiations can share a type). A call that failed is made again next time.
inline cudaError_t raise_smem_limit(const void* kern, size_t bytes) {
    struct Limit {
        const void* kern;
        int dev;
        size_t bytes;
    };
    static std::mutex mu;
    static std::vector<Limit> limits;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    Limit* known = nullptr;
    for (Limit& l : limits)
        if (l.kern == kern && l.dev == dev) known = &l;
    if (known && bytes <= known->bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    if (known) known->bytes = bytes;
    else limits.push_back({kern, dev, bytes});
    return cudaSuccess;
}

}  // namespace pic
