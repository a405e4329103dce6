// Launches that overlap the end of the kernel before them.
//
// One call is a chain of short kernels (pyramid, FAST, NMS, top-N,
// orientation), each starting from descriptors that the host wrote before the
// chain.  Launched with `pdl` (programmatic stream serialization), a kernel may
// start while its predecessor still runs: it reads descriptors, sets up its
// barriers and then waits (pdl_wait) for the predecessor's grid to complete
// and its writes to be visible.  A kernel launched this way waits in every
// thread before it ends, on every path (one that gives up on an expired wait
// among them), so a kernel's completion implies its predecessors'; one that is
// launched plainly starts behind them and need not wait.
// pdl_trigger lets the next kernel of the chain start; it is called first
// thing, so that kernel's blocks take their places as soon as the SMs have
// room.  Without `pdl` both are no-ops.
// What a kernel of the chain writes is read by the later ones with plain loads:
// they may be resident while it is written, and the non-coherent path (__ldg)
// is for data that does not change while the reading kernel runs.  That path is
// left to what the host wrote before the chain (descriptors, item tables).
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace ofk {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// cluster: blocks per cluster (1: none).
template <typename... P, typename... A>
inline void launch_chain(void (*kernel)(P...), dim3 grid, int block, int smem, cudaStream_t st, bool pdl, int cluster,
                         A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (pdl) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster;
        at[n].val.clusterDim.y = 1;
        at[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    cudaLaunchKernelEx(&cfg, kernel, P(std::forward<A>(args))...);
}

}  // namespace ofk
