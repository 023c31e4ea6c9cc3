// cs_launch.cuh -- chains of short kernels within one entry point.
#pragma once

#include <cuda_runtime.h>

namespace cs {

// Programmatic dependent launch.  A kernel launched by launch_after may become
// resident as soon as every block of the kernel before it has passed
// launch_dependents (or ended), and must pass wait_for_primary, which waits
// for the whole end of the kernel before, ahead of its first access to global
// memory that any earlier work of the stream touches.  Every kernel of a
// chain waits, so the end of one is the end of all before it.
//
// After the wait it reads what the chain's earlier kernels wrote by plain loads or
// __ldcg: not by __ldg, and not through __restrict__ kernel parameters.  It
// lives from before those writes on, and the read-only path is defined only for
// data that nothing writes while the kernel lives; through a __restrict__
// parameter the compiler may take that path, or move a load above the wait,
// whose memory clobber does not bind it.  Tables that the host had written before
// the chain's first launch are free of the rule.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_primary() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_after(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace cs
