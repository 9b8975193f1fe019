// Launches whose latency overlaps the end of the kernel before them in the stream
// (programmatic dependent launch). Every kernel launched by launch_after() calls
// dependency_wait() before it touches global memory: it returns when the kernels before it
// have completed and their writes are visible, so the order of effects is that of plain
// launches. No kernel lets its dependents start before it ends: their blocks would take
// shared and tensor memory that its own later waves use (net forward of 8 x 640x480: 237 us
// with, 218 without, 234 with plain launches; training step of 3 x 315x237: 189, 184, 223).
#pragma once

#include <cuda_runtime.h>

namespace sgad {

// Waits; loads through the given pointers stay behind the wait. (A pointer to const with
// __restrict__ may be read by loads that the compiler is free to move across the wait: to it
// the memory never changes during the kernel. After this it knows nothing of the pointer.)
template <class... P>
__device__ __forceinline__ void dependency_wait(P &...p)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (([](P &q) { asm volatile("" : "+l"(q)); })(p), ...);
}

template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

}  // namespace sgad
