// How the library launches its kernels.
#pragma once

#include <atomic>

#include <cuda_runtime.h>

namespace ubep {

// Launch that lets the kernel be placed while its predecessor in the stream drains (the
// kernels above call griddep_wait() before they read anything).  `together`: a cooperative
// launch -- the kernel's CTAs wait for flags that other CTAs of the same grid publish, so they
// must all be resident at once; the runtime then refuses a grid that cannot be (a synchronous
// error instead of CTAs spinning until their bounded waits run out) and starts the grid only
// when every CTA has a place.  Such a kernel is not launched ahead of its predecessor's end.
template <typename... KArgs, typename... Args>
static cudaError_t launch_overlapped(void (*kern)(KArgs...), int grid, int block, size_t smem, cudaStream_t st,
                                     bool together, int cluster, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    if (together) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
    } else {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = (unsigned)cluster;
        attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// The dynamic shared-memory limit of a kernel is a sticky attribute: per kernel instance and
// device only a larger request has to reach the runtime (the call costs host time that an
// enqueue-bound caller sees on every dispatch).  `granted` belongs to one kernel instance.
constexpr int kAttrDevices = 64;
static cudaError_t allow_dynamic_smem(const void* kern, int bytes, std::atomic<int>* granted) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool cached = dev >= 0 && dev < kAttrDevices;
    if (cached && granted[dev].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && cached) granted[dev].store(bytes, std::memory_order_relaxed);
    return e;
}

}  // namespace ubep
