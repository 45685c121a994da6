// Limits of a kernel that belong to the function and not to a launch: its dynamic
// shared memory and whether clusters of more than 8 CTAs are allowed.  The runtime
// keeps them per function and device for the whole process, and contexts run in
// threads of their own, with operators of different sizes: a limit is therefore raised
// when a launch needs more and never lowered, so that no thread can take from another
// what it has just asked for.
#include <cuda_runtime_api.h>

#include <map>
#include <mutex>
#include <utility>

#include "limits.h"

namespace sie {

struct KernelLimit {
    size_t smem = 48 * 1024;  // what every kernel has without asking
    bool wide = false;
};
static std::map<std::pair<const void*, int>, KernelLimit> g_limits;
static std::mutex g_limits_mu;

cudaError_t kernel_limit(const void* fn, size_t smem, bool wide_cluster)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_limits_mu);
    KernelLimit& k = g_limits[{fn, dev}];
    if (smem > k.smem) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k.smem = smem;
    }
    if (wide_cluster && !k.wide) {
        e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
        k.wide = true;
    }
    return cudaSuccess;
}

}  // namespace sie
