// The limit of a kernel's dynamic shared memory is state of the (device, kernel), not of a launch:
// set by one host thread to the little its product needs, it makes the launch of another thread,
// which raised it just before, fail.  It is only ever raised here, under a lock.
#pragma once

#include <cuda_runtime_api.h>

#include <map>
#include <mutex>
#include <utility>

namespace spg {

// Lets launches of `kern` on the current device have up to `bytes` of dynamic shared memory.
inline cudaError_t allow_dynamic_smem(const void *kern, int bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void *>, int> allowed;
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(mu);
    int &now = allowed[{device, kern}];
    if (bytes <= now) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) now = bytes;
    return e;
}

}  // namespace spg
