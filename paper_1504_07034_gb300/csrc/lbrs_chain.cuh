// Chains of dependent launches (programmatic dependent launch): in a captured chain the next kernel is
// launched as the last blocks of the one before it exit, and waits for its writes where it first touches
// memory, so that launching passes under the flush.  A kernel does not ask for its successor any earlier:
// blocks of one warp that come while their predecessors still hold most slots pile up on the free ones
// (1024 x 1024 on the moments 5.8 us per step unchained, 5.7 chained, 7.2 when asked for at the top).
// 0.1 to 0.3 us of each launch (us per step, unchained and chained: internal walls at 960 x 320 3.97 and
// 3.84, moments of 128^2 1.89 and 1.78, omega != 1 at 64^2 1.41 and 1.22, at 1000^2 11.5 and 11.35).
//
// A chained kernel is resident while the one before it still writes, so what that one writes is not
// read-only for its lifetime: neither __ldg nor a plain load that the compiler may take for one (a const
// __restrict__ pointer) may read it, because such loads go through the non-coherent path and may move
// above the wait.  chain_load reads it.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace lbrs {

// At the top of a kernel that may stand in a chain, before its first access to memory: waits until the
// launch before it has ended and its writes are visible.  Without a chain it does nothing.
__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Loads of what the launch before wrote: coherent, and behind chain_begin (volatile statements keep their
// order).
__device__ __forceinline__ float chain_load(const float* p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned long long chain_load(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.global.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ __half chain_load(const __half* p)
{
    unsigned short v;
    asm volatile("ld.global.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return __ushort_as_half(v);
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
