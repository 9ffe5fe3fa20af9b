// Host side: the dynamic shared memory that a kernel may be launched with.
#pragma once

#include <cuda_runtime.h>

// Raises the kernel's limit of dynamic shared memory to all that a block can have
// beside its static part.  The limit belongs to the kernel on the device, not to a
// launch: always the same value, so that threads which launch objects of different
// sizes cannot lower it between one another's call and launch.  Set where the
// objects are made.
inline cudaError_t qs_raise_smem_limit(const void *fn, size_t *limit = nullptr) {
    cudaFuncAttributes at;
    int dev = 0, most = 0;
    cudaError_t e = cudaFuncGetAttributes(&at, fn);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    most -= (int)at.sharedSizeBytes;
    if (limit) *limit = (size_t)most;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}
