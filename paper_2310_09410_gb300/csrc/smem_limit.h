// Dynamic shared memory of kernels that take more than the default 48 KB.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace opf {

// Lets launches of `fn` take `bytes` of dynamic shared memory; nonzero when
// that is more than a block can have.  The limit belongs to the kernel in its
// context, so to every handle, batch and thread that launches it, and plans
// keep launching long after they were built: it is only ever raised, and
// always to all that a block can have beside the kernel's static memory, so no
// caller can take away what another one counts on.
inline int allow_dynamic_smem(const void *fn, size_t bytes) {
    cudaFuncAttributes at;
    int dev = 0, optin = 0;
    if (cudaFuncGetAttributes(&at, fn) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return -1;
    const long long most = (long long)optin - (long long)at.sharedSizeBytes;
    if ((long long)bytes > most) return -1;
    if (at.maxDynamicSharedSizeBytes >= most) return 0;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) == cudaSuccess ? 0 : -1;
}

}  // namespace opf
