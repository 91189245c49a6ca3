// griddep.cuh -- programmatic dependent launch: a kernel launched with the attribute may
// start once every CTA of the kernel before it has called griddep_launch() (or has exited)
// and runs concurrently with it until griddep_wait(), which returns when that kernel has
// completed and its writes are visible.  Both are no-ops in a kernel launched without the
// attribute.  A kernel whose predecessor was itself launched this way must wait in at least
// one CTA, so that "complete" covers the whole chain; every kernel here does.
#pragma once
#include <cuda_runtime.h>

namespace ptylm {

__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch `fn` (cluster > 1: with that cluster size), overlapping the kernel before it on the
// stream up to its griddep_wait().
inline cudaError_t launch_dependent(const void* fn, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t stream,
                                    int cluster = 1) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = cluster;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = cluster > 1 ? 2 : 1;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace ptylm
