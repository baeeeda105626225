// Launches with programmatic dependent launch (internal to the library).
//
// Every call of the library is a short chain of kernels on the caller's stream.  Each is launched
// with the programmatic-stream-serialization attribute: its CTAs may be scheduled while the kernel
// before it drains, and they wait (griddepcontrol.wait) before they read or write any global memory.
// The order stays transitive because every kernel launched this way waits before it lets the next
// one in (griddepcontrol.launch_dependents) and before it ends: a kernel has completed only after
// the one before it has.
#pragma once

#include <cuda_runtime.h>

namespace dssd {

template <class Params>
cudaError_t launch_pdl(void (*kernel)(Params), unsigned grid, unsigned block, cudaStream_t stream, const Params &params,
                       size_t smem = 0, unsigned cluster = 1)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;  // at most 48 KB
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, params);
}

// An entry point of the driver, which the library is not linked against; nullptr if there is none of that name.
template <class Fn>
Fn driver_call(const char *name)
{
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    const cudaError_t e = cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &found);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? reinterpret_cast<Fn>(fn) : nullptr;
}

}  // namespace dssd
