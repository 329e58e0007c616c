// Launch helper shared by the kernels that are started with programmatic dependent launch.
#pragma once
#include <cuda_runtime.h>
#include <cstdlib>
#include <utility>

namespace gleam {

// Programmatic dependent launch.  A kernel started through launch_overlapped with allow = true may
// be scheduled while the kernel before it on the stream is still draining; it calls
// grid_dependency_wait() as its first statement, which holds it until that kernel has completed and
// its writes are visible, so only the launch latency and the block start-up overlap.
// grid_launch_dependents() right after the wait lets the next such kernel be scheduled as soon as
// every block of this one has started; without it the next one is scheduled as the blocks of this one end.  Measured
// on B200: the early start is a gain between launches whose blocks all run at once and end together (cine: 8 % per
// step), and in the short launches that build the tables of the sampled positions; elsewhere early blocks fill the SMs
// unevenly or sit next to a long tail (up to 27 % in the row-tile passes, 20 % in multi-round launches of the row
// kernels), and those kernels wait without letting the next one in.
// Such a kernel is running while the one before it still writes, so nothing that it reads is constant for its lifetime: the
// kernels read with plain loads, no __ldg and no const __restrict__ parameters, from which the compiler makes read-only
// (non-coherent) ones.  Measured equal or faster (cine, 8 prepared steps and VJPs, 318.5 -> 316.7 us).
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// GLEAM_NO_OVERLAP=1 launches these kernels fully serialised (tuning aid, read once).
inline bool overlap_enabled() {
    static int v = -1;
    if (v < 0) { const char* e = getenv("GLEAM_NO_OVERLAP"); v = (e && e[0] == '1') ? 0 : 1; }
    return v == 1;
}

// cluster > 1: blocks in clusters of that many
inline void launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&at)[2], bool allow, dim3 grid, dim3 block,
                               size_t smem, cudaStream_t s, unsigned cluster) {
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
    unsigned n = 0;
    if (allow && overlap_enabled()) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster; at[n].val.clusterDim.y = 1; at[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = at; cfg.numAttrs = n;
}
template <class... KArgs, class... Args>
inline cudaError_t launch_overlapped(bool allow, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                     cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    launch_config(cfg, at, allow, grid, block, smem, s, 1);
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
template <class... KArgs, class... Args>
inline cudaError_t launch_overlapped_cluster(unsigned cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                             cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[2];
    launch_config(cfg, at, true, grid, block, smem, s, cluster);
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace gleam
