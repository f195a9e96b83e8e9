// Per-device facts the launch code caches: the SM count, and "this kernel's attribute has been set on
// this device" flags.  All of it is safe to use from several host threads on several devices: the
// cached values are idempotent and held in atomics indexed by device.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <utility>

namespace gf {

constexpr int MAX_DEVICES = 64;

// Index of the current device, or -1 if it cannot be had or is beyond MAX_DEVICES.
inline int current_device()
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return -1;
    return dev;
}

// Number of SMs of the current device (0 on failure).
inline int sm_count()
{
    static std::atomic<int> cached[MAX_DEVICES];          // zero-initialised: 0 = not asked yet
    const int dev = current_device();
    if (dev < 0) return 0;
    int n = cached[dev].load(std::memory_order_relaxed);
    if (n == 0) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
        cached[dev].store(n, std::memory_order_relaxed);
    }
    return n;
}

// One flag per device, for work that has to happen once per device and may harmlessly happen twice
// (cudaFuncSetAttribute of a kernel).
struct PerDeviceFlag {
    std::atomic<bool> done[MAX_DEVICES];
    bool is_set(int dev) const { return done[dev].load(std::memory_order_acquire); }
    void set(int dev) { done[dev].store(true, std::memory_order_release); }
};

// Launches with programmatic stream serialisation: the grid may be scheduled while the kernel ahead of it in the stream drains
// (from the moment all of that kernel's CTAs have executed griddepcontrol.launch_dependents or left), sets itself up meanwhile, and
// holds at its griddepcontrol.wait, which a kernel launched this way executes before its first access to global memory, until
// that kernel has completed and flushed.
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
// The same in clusters of `cluster` CTAs.
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, unsigned cluster, cudaStream_t st, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace gf
