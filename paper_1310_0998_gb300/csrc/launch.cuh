// Programmatic launch order of a chain of kernels on one stream.
#pragma once
#include <cuda_runtime.h>

namespace dpd {

// A kernel of such a chain waits for the one before it (which has waited for
// its own predecessor), and lets the next one start: the next one's launch,
// and what it does before its own wait, pass behind the rest of this kernel.
// What runs before the wait reads nothing that the kernel before writes, and
// writes nothing that it reads; what runs after it uses ordinary loads (not the
// read-only path, whose lines may be older than the wait).  Without a
// predecessor in programmatic order the wait returns at once.
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch in programmatic order: for kernels that call wait_for_previous alone.
template <typename... P, typename... A>
inline void launch_step(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute a{};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &a;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, kernel, args...);
}

}  // namespace dpd
