// Dynamic shared memory that every launch here may have, and the opt-in for more.  The
// limit belongs to the function on the device that is current, so it is looked
// up before each launch (or graph) that needs more, not remembered per process;
// and it goes to the most the device has, never down, so that neither another
// handle nor another thread takes it away again.
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

namespace ekl {

constexpr size_t SMEM_DEFAULT = 40 * 1024;  // (48 KB with the kernel's static shared memory)
inline cudaError_t smem_opt_in(const void *kernel, size_t bytes)
{
    if (bytes <= SMEM_DEFAULT) return cudaSuccess;
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
    if (e != cudaSuccess || bytes <= (size_t)fa.maxDynamicSharedSizeBytes) return e;
    int dev = 0, most = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    most -= (int)fa.sharedSizeBytes;
    if (most < 0 || bytes > (size_t)most) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

}  // namespace ekl
