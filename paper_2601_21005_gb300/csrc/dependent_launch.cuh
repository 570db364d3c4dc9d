// Programmatic stream serialisation: a kernel launched by launch_dependent may start while the last
// blocks of the kernel before it run, and what it does before dependents_wait() overlaps that kernel's
// end and the launch.  dependents_wait() returns when the kernel before has completed and its stores
// are visible.  A kernel that waits before it lets the next one start (dependents_launch) vouches for
// everything older too: so before the wait a kernel may read what the kernel directly before it does
// not write.  What that one does write is loaded by asm volatile loads (the ld*_written forms,
// cp.async), which stay behind the wait: the compiler may move a plain or __ldg load above it.
#pragma once
#include <cuda_runtime.h>

namespace sgw {

__device__ __forceinline__ void dependents_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// cluster: blocks of a thread-block cluster along x (1: none)
template <class... P, class... A>
static void launch_dependent(void (*kern)(P...), dim3 grid, int threads, size_t smem, unsigned cluster, cudaStream_t st,
                             A... args) {
    cudaLaunchAttribute at[2] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

}  // namespace sgw
