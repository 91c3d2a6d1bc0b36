// Chained launches: a kernel that may start while the previous one on its stream
// still runs (programmatic stream serialization).
#pragma once

#include <cuda_runtime.h>

namespace fdlbm {
namespace {

// Wait for the previous launch of the chain: its results are visible after this,
// and nothing that it reads or writes is touched before.  A no-op in a kernel
// launched without the attribute.
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Let the next launch's blocks be scheduled once every block has come here (or
// ended).  It comes after a block's work: earlier, the waiting blocks of the next
// launch take SM slots unevenly.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t chained_launch(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, const A &...args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace
}  // namespace fdlbm
