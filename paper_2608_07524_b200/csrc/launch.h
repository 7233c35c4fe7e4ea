// Kernel launches of libdcp (host side).
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

namespace dcp {

// Launches `kern` so that its CTAs may start while the kernel before it in the stream still runs (programmatic stream
// serialisation): what comes before its grid_wait() (barriers, tensor memory, descriptor prefetch) and the launch itself
// then overlap that kernel.  A call is a chain of two to seven kernels, most of them a few microseconds long.
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t stream, A&&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

// Lets KERN use `bytes` of dynamic shared memory, once per device (the attribute stays with the function).
template <auto KERN>
cudaError_t allow_smem(int bytes) {
    static std::atomic<uint64_t> done{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(KERN, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}

}  // namespace dcp
