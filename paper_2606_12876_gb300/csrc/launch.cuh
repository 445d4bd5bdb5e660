// Kernel launches of the GEMV translation units: programmatic dependent launch, clusters, and
// the per-kernel attributes set once. Internal; not part of the ABI.
#pragma once

#include <map>
#include <mutex>
#include <tuple>

#include "aq_internal.cuh"

namespace aq {

// Launch with the programmatic-stream-serialization attribute (PDL), so the kernel's CTAs may
// become resident while the preceding kernel in the stream drains; every kernel launched this
// way calls griddepcontrol.wait before it reads anything another kernel may have written. csize:
// CTAs per cluster along x (1: no clusters).
template <typename... KArgs, typename... Args>
aq_status launch_pdl_cluster(int csize, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)csize;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = csize > 1 ? 2 : 1;
    return cuda_ok(cudaLaunchKernelEx(&cfg, kern, (KArgs)args...), "cudaLaunchKernelEx");
}

template <typename... KArgs, typename... Args>
aq_status launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                     Args... args) {
    return launch_pdl_cluster(1, kern, grid, block, smem, st, args...);
}

// Raises the kernel's dynamic shared-memory limit and returns its occupancy. Both are cached
// per (kernel, device, slot), slot being the prefix m where the shared-memory size depends on
// it, so the CUDA attribute calls happen once, before any stream capture that later calls
// reuse.
template <typename K>
aq_status prepare(K kern, size_t smem, int threads, int slot, int* ctas_per_sm) {
    static std::mutex mu;
    static std::map<std::tuple<const void*, int, int>, int> cache;
    int dev = 0;
    if (cudaError_t e = cudaGetDevice(&dev); e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    const auto key = std::make_tuple((const void*)kern, dev, slot);
    std::lock_guard<std::mutex> lock(mu);
    if (auto it = cache.find(key); it != cache.end()) {
        *ctas_per_sm = it->second;
        return AQ_OK;
    }
    DeviceInfo di;
    if (aq_status e = device_info(&di); e != AQ_OK) return e;
    cudaFuncAttributes fa;
    if (cudaError_t e = cudaFuncGetAttributes(&fa, kern); e != cudaSuccess)
        return cuda_fail(e, "cudaFuncGetAttributes");
    const int dyn_max = di.smem_optin - (int)fa.sharedSizeBytes;
    if ((int)smem > dyn_max) return AQ_ERR_UNSUPPORTED;
    // Allow the largest size any slot of this kernel may need (the attribute is per kernel).
    if (cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             dyn_max);
        e != cudaSuccess)
        return cuda_fail(e, "cudaFuncSetAttribute");
    // Every kernel of the library asks for the same (largest) shared-memory carve-out, so
    // consecutive launches never force an SM to re-split its L1 / shared-memory storage.
    if (cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                             (int)cudaSharedmemCarveoutMaxShared);
        e != cudaSuccess)
        return cuda_fail(e, "cudaFuncSetAttribute");
    if (cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas_per_sm, kern, threads,
                                                                      smem);
        e != cudaSuccess)
        return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (*ctas_per_sm < 1) return AQ_ERR_UNSUPPORTED;
    cache[key] = *ctas_per_sm;
    return AQ_OK;
}

}  // namespace aq
