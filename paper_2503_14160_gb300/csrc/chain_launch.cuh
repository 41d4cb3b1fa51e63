// Launches of a chain of dependent kernels (programmatic dependent launch). A plan's iteration is
// some ten short kernels, each needing all of the one before, so the gap between them counts: with
// the attribute below a kernel's blocks may be placed while the kernel before still runs, and
// after_previous(), called before such a kernel touches anything of the others, waits until that one has completed
// and its writes are visible. Every kernel of a chain waits, so completion is transitive: whatever
// follows a kernel on the stream sees everything before it. The wait has no limit of its own: it
// ends when the kernel before ends, as an ordinary launch would begin.
// A chained kernel begins before that wait ends, so what the others write is not read-only for its
// whole life: it and the functions it calls read global memory by plain loads, never through
// `const T *__restrict__` or __ldg, which would allow non-coherent loads and let the compiler move
// them over the wait (a host test looks through the sources for it).
// Measured with the node that cleared the evaluation's counter gone too: an iteration of the 20-tree
// query 59 -> 48.5 us.
#pragma once

#include <cuda_runtime.h>

namespace cp {

#ifdef __CUDACC__
// Waits for the kernel before, then lets the next one's blocks be placed.
static __device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// kern<<<grid, block, smem, st>>>(args...) with the attribute. The kernel calls
// after_previous() before it reads or writes global memory.
template <typename... P, typename... A>
inline void launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);   // an error is the last error, as of <<<>>>
}
#endif

}  // namespace cp
