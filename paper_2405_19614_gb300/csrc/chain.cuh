// Launches of one call that follow one another (programmatic dependent launch):
// the blocks of a chained kernel are started while the kernel before it still
// runs and wait there, so that its launch costs nothing between the two.
//
//  - chain_go() lets the next chained kernel's blocks start once every block of
//    this one has called it (or ended);
//  - chain_wait() waits until the kernel before has ended and its writes are
//    visible.  Every thread of a chained kernel calls it before its first
//    access to global memory, so that a kernel's end implies the end of all
//    before it;
//  - without launch_chained both do nothing.
//
// Only launches of one call on one stream are chained, never the first: what
// the caller put on the stream, events and graph captures around a call see
// ordinary launches.  Chained are short kernels, where the launch is a good part
// of the time (a 100k-Gaussian tracking step 150.9 -> 141.0 us, a 300k render
// 129.2 -> 125.7).  The onesweep passes are not: the blocks waiting for the next
// pass take the places of running ones (four passes over 1M keys and what
// follows: 20 us slower).
#pragma once

#include <cuda_runtime.h>

namespace gs {

__device__ __forceinline__ void chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);  // errors are read by launch_status
}

}  // namespace gs
