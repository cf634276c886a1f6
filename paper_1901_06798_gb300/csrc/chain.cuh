// chain.cuh -- launches that overlap their start with the end of the one before.
//
// A level step is a chain of short kernels on one stream.  Launched with
// programmatic stream serialisation, a kernel's CTAs are placed as soon as every CTA
// of the kernel before it has started or left; each waits, before it touches
// memory, until that kernel has finished and its writes are visible.  What is
// saved is part of each launch: 17.1 -> 16.2 us for a step of a 200^2 grid (three
// kernels), 74 us for the unsplit step of 1024^2 cells that took 77.
#pragma once
#include <cuda_runtime.h>
#include <utility>

namespace tsu {

// First statement of every kernel that is launched by launch_chained.  Such a kernel
// runs while the kernel before it still writes, so no pointer of it, or of a function
// it calls, is __restrict__: that would promise data that never changes while the
// kernel runs, and let the compiler load it ahead of the wait or past the coherent
// caches.
__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
int launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&c, kernel, P(std::forward<A>(args))...);
}

}  // namespace tsu
