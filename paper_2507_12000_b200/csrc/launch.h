// Launches with programmatic dependent launch (internal to the library).
//
// Every call of the library is a short chain of kernels on the caller's stream.  Each is launched
// with the programmatic-stream-serialization attribute: its CTAs may be scheduled while the kernel
// before it drains, and they wait (griddepcontrol.wait) before they read or write any global memory.
// The order stays transitive because every kernel launched this way waits before it lets the next
// one in (griddepcontrol.launch_dependents) and before it ends: a kernel has completed only after
// the one before it has.
#pragma once

#include <atomic>

#include <cuda.h>
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

// One small answer (0 .. 31) per context, asked for on the first call made in it.  A device that was reset, or a second
// context on it, is asked again.
class PerContext {
public:
    template <class Ask>
    int get(Ask ask)
    {
        typedef CUresult (*ContextId)(CUcontext, unsigned long long *);
        static const ContextId context_id = driver_call<ContextId>("cuCtxGetId");
        unsigned long long id = 0;  // (an id is never given twice)
        const bool has_id = context_id && context_id(nullptr, &id) == CUDA_SUCCESS;
        if (has_id)
            for (const auto &k : known) {
                const unsigned long long w = k.load(std::memory_order_acquire);
                if (w / 32 == id + 1) return (int)(w % 32);
            }
        const int answer = ask();
        if (has_id) known[turn.fetch_add(1, std::memory_order_relaxed) % 16].store((id + 1) * 32 + (unsigned long long)answer, std::memory_order_release);
        return answer;
    }

private:
    std::atomic<unsigned long long> known[16]{};  // (id + 1) * 32 + the answer; 0: empty
    std::atomic<unsigned> turn{0};
};

// Clusters beyond the portable size of eight have to be allowed for each kernel in each context, and a device (or the part of one
// that the process was given) may not have a processing cluster of that many SMs.
template <class Params>
bool allow_cluster(void (*kernel)(Params), unsigned ctas, unsigned threads)
{
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = ctas;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    return cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0;
}

}  // namespace dssd
