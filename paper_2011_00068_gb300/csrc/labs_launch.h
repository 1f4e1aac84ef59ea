// labs_launch.h -- host side of launches whose shared memory is above the default 48 KB.
#pragma once

#include <cuda_runtime.h>

namespace labsgpu {

// A kernel's limit of dynamic shared memory belongs to the process (per device): several
// contexts, lengths and host threads share a kernel and ask for different sizes.  So the limit
// is always set to what the device allows, never to one launch's need, which another thread's
// smaller one could replace between that call and the launch.
// static_bytes: the kernel's own shared arrays.
inline cudaError_t allow_shared(const void* fn, int static_bytes)
{
    int dev = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most - static_bytes);
    return e;
}

// The same with the kernel's attributes asked for (about 1 us more).
inline cudaError_t allow_shared(const void* fn, cudaFuncAttributes* attributes = nullptr)
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess) e = allow_shared(fn, (int)fa.sharedSizeBytes);
    if (attributes != nullptr) *attributes = fa;
    return e;
}

}  // namespace labsgpu
