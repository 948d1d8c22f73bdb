// launch.cuh - host helper of the kernels' set-up.
#pragma once

#include <cuda_runtime.h>

namespace mdgb {

// Let a kernel's launches take all the dynamic shared memory that the current device allows beside its
// static shared memory.
template <typename K>
inline void allow_max_smem(K kernel) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return;
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

}  // namespace mdgb
