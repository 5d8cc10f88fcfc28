// wl_launch.cuh -- one walker launch, or the occupancy query that admits it.
#pragma once

#include "wl_kernels.cuh"

namespace wl {

inline cudaError_t launch_or_query(void (*fn)(const WalkArgs), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                   const WalkArgs& a, int* bps)
{
    // The dynamic shared-memory limit is a property of the kernel function,
    // shared by every handle: raise it to the device maximum (outside stream
    // capture) and never lower it, so a captured launch of one handle stays
    // valid whatever shape another handle uses.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (!bps) {
        cudaError_t e = cudaStreamIsCapturing(s, &cap);
        if (e != cudaSuccess) return e;
    }
    if (cap == cudaStreamCaptureStatusNone) {
        int dev = 0, optin = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     optin > (int)smem ? optin : (int)smem);
        // one split of an SM's memory for every walker kernel: a kernel that asks for
        // another one waits until the SM is empty, and handles no longer overlap
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
        if (e != cudaSuccess) return e;
    }
    if (bps) return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, fn, (int)block.x, smem);
    clear_stale_error();
    fn<<<grid, block, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace wl
