// Chains of dependent launches (programmatic dependent launch): in a captured chain the next kernel is
// launched as the last blocks of the one before it exit, and waits for its writes where it first touches
// memory, so that launching passes under the flush.  A kernel does not ask for its successor any earlier:
// blocks of one warp that come while their predecessors still hold most slots pile up on the free ones
// (1024 x 1024 on the moments 5.8 us per step unchained, 5.7 chained, 7.2 when asked for at the top).
// 0.1 to 0.3 us of each launch (us per step, unchained and chained: internal walls at 960 x 320 3.97 and
// 3.84, moments of 128^2 1.89 and 1.78, omega != 1 at 64^2 1.41 and 1.22, at 1000^2 11.5 and 11.35).
#pragma once

#include <cuda_runtime.h>

namespace lbrs {

// At the top of a kernel that may stand in a chain, before its first access to memory: waits until the
// launch before it has ended and its writes are visible.  Without a chain it does nothing.
__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launch; chained: as the next of a chain whose every kernel begins with chain_begin.
template <class... P, class... A>
cudaError_t launch_in_chain(bool chained, void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t s, const A&... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace lbrs
