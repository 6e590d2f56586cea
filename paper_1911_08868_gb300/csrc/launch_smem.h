// Dynamic shared memory of the kernels that take more than the default 48 KB.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

#include "pcbp_internal.h"

namespace pcbp {

// Lets `kern` be launched with all the dynamic shared memory a block of the current device can have.
// The limit belongs to the kernel, not to the launch, and a launch above it fails.  The size of a
// launch depends on its batch, so a launcher that set the limit to its own size could lower it
// between another host thread's setting and launch (PC_ECUDA there, seen with one thread decoding
// single frames of N = 2048 and another batches of them); every launcher sets this one value.
template <auto kern>
cudaError_t allow_dynamic_smem()
{
    static std::atomic<int> fixed{-1};       // the kernel's static shared memory, known when compiled
    int own = fixed.load(std::memory_order_relaxed);
    if (own < 0) {
        cudaFuncAttributes a;
        const cudaError_t e = cudaFuncGetAttributes(&a, kern);
        if (e != cudaSuccess) return e;
        own = int(a.sharedSizeBytes);
        fixed.store(own, std::memory_order_relaxed);
    }
    DeviceInfo di;
    if (device_info(&di) != PC_OK) return cudaErrorInvalidDevice;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, di.smem_optin - own);
}

}  // namespace pcbp
