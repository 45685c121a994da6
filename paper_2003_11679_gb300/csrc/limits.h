// Process-wide limits of kernels (limits.cpp).
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>

namespace sie {
// on the current device, allow kernel fn at least smem bytes of dynamic shared memory
// and, for wide_cluster, clusters of more than 8 CTAs; before every launch that needs it
cudaError_t kernel_limit(const void* fn, size_t smem, bool wide_cluster = false);
}  // namespace sie
