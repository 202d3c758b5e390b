// smem_limit.h -- the dynamic shared memory that a kernel's launches may ask for.
#pragma once

#include <cstddef>

#include <cuda_runtime.h>

namespace slpic {

// The limit is an attribute of the kernel, one for all handles.  A handle that set it to its
// own need would lower it under a larger live one, so every handle sets the same value: all
// that the device has beside the kernel's static shared memory.  (A launch still takes only
// what it asks for.)  cudaErrorInvalidValue where `need` bytes do not fit.
template <typename F>
inline cudaError_t allow_dynamic_smem(F *kernel, size_t need)
{
    int dev = 0, most = 0;
    cudaFuncAttributes at;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncGetAttributes(&at, kernel);
    if (e != cudaSuccess)
        return e;
    if (need + at.sharedSizeBytes > (size_t)most)
        return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                most - (int)at.sharedSizeBytes);
}

}  // namespace slpic
