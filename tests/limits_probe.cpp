// Test probe: the library's kernel limits (paper_2003_11679_gb300/csrc/limits.cpp) over
// a stand-in for the CUDA runtime's per-process table of function attributes, compiled
// together with that file by tests/test_limits_host.py for a CPU check.
#include <map>
#include <mutex>
#include <thread>
#include <tuple>
#include <vector>

#include "../paper_2003_11679_gb300/csrc/limits.h"

static thread_local int t_dev = 0;
static std::mutex mu;
static std::map<std::tuple<const void*, int, int>, int> table;  // (function, device, attribute)

extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* d)
{
    *d = t_dev;
    return cudaSuccess;
}
extern "C" cudaError_t CUDARTAPI cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v)
{
    std::lock_guard<std::mutex> lk(mu);
    if (v > 227 * 1024) return cudaErrorInvalidValue;
    table[std::make_tuple(f, t_dev, (int)a)] = v;
    return cudaSuccess;
}
static int value(const void* f, int dev, cudaFuncAttribute a)
{
    std::lock_guard<std::mutex> lk(mu);
    auto it = table.find(std::make_tuple(f, dev, (int)a));
    return it == table.end() ? -1 : it->second;
}

static const char kernels[4] = {0, 1, 2, 3};

// threads asking for sizes of their own, then "launching": the launches that found less than they need
extern "C" int limits_race(int rounds)
{
    const size_t size[4] = {60000, 200000, 90000, 120000};
    std::vector<int> low(4, 0);
    std::vector<std::thread> th;
    for (int i = 0; i < 4; i++)
        th.emplace_back([&, i] {
            for (int r = 0; r < rounds; r++) {
                if (sie::kernel_limit(kernels, size[i]) != cudaSuccess) low[i]++;
                std::this_thread::yield();
                if (value(kernels, 0, cudaFuncAttributeMaxDynamicSharedMemorySize) < (int)size[i]) low[i]++;
            }
        });
    for (auto& t : th) t.join();
    return low[0] + low[1] + low[2] + low[3];
}

// the limit on each of two devices after both asked (device 1 first for kernel 1)
extern "C" void limits_devices(int* out)
{
    for (int d : {1, 0}) {
        t_dev = d;
        sie::kernel_limit(kernels + 1, 100000, d == 0);
    }
    t_dev = 0;
    out[0] = value(kernels + 1, 0, cudaFuncAttributeMaxDynamicSharedMemorySize);
    out[1] = value(kernels + 1, 1, cudaFuncAttributeMaxDynamicSharedMemorySize);
    out[2] = value(kernels + 1, 0, cudaFuncAttributeNonPortableClusterSizeAllowed);
    out[3] = value(kernels + 1, 1, cudaFuncAttributeNonPortableClusterSizeAllowed);
}

// a refused size is an error and leaves what was granted; 48 KB need no call
extern "C" int limits_refused(int* out)
{
    const cudaError_t a = sie::kernel_limit(kernels + 2, 48 * 1024);
    out[0] = value(kernels + 2, 0, cudaFuncAttributeMaxDynamicSharedMemorySize);
    const cudaError_t b = sie::kernel_limit(kernels + 2, 70000), c = sie::kernel_limit(kernels + 2, 300000);
    out[1] = value(kernels + 2, 0, cudaFuncAttributeMaxDynamicSharedMemorySize);
    return (a == cudaSuccess && b == cudaSuccess && c != cudaSuccess) ? 0 : 1;
}
