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
// of the time (unchained and chained, passes back to back: a 100k-Gaussian tracking
// step 127 and 111 us, a 300k render 114 and 102, a 300k mapping step 345 and 326).
// The onesweep passes are not: the blocks waiting for the next
// pass take the places of running ones (four passes over 1M keys and what
// follows: 20 us slower).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace gs {

__device__ __forceinline__ void chain_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A launch with its attributes: chained (or not), in clusters of `cluster` blocks.
// A call stops at the first launch that is refused: the kernels behind it read
// what it would have written (places in a list among it).
template <typename... P, typename... A>
[[nodiscard]] inline gs_status_t launch_with(bool chained, int cluster, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                        cudaStream_t s, A... args)
{
    cudaLaunchAttribute attr[2] = {};
    cudaLaunchConfig_t cfg = {};
    if (chained) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs++].val.clusterDim.z = 1;
    }
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    return launch_status();
}

template <typename... P, typename... A>
[[nodiscard]] inline gs_status_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args)
{
    return launch_with(true, 1, kernel, grid, block, smem, s, args...);
}

// Clears n words for the kernel chained after it (a memset would end before that
// kernel's launch begins).
static __global__ void chain_clear_kernel(uint32_t *p, uint32_t n)
{
    chain_go();
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) p[i] = 0u;
}

[[nodiscard]] inline gs_status_t launch_clear(uint32_t *p, uint32_t n, cudaStream_t s)
{
    const unsigned blocks = (n + 1023) / 1024;
    chain_clear_kernel<<<blocks < 512 ? blocks : 512, n < 256 ? 32 : 256, 0, s>>>(p, n);
    return launch_status();
}

}  // namespace gs
