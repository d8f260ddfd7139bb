// Programmatic dependent launch.
//
// Launched with the programmatic-serialization attribute, a kernel may be scheduled while its predecessor on the
// stream is still running: once every CTA of the predecessor has called grid_dep_launch() or left. grid_dep_wait()
// returns when the predecessor has completed and its memory operations are visible. In a kernel launched without the
// attribute both calls return at once. Two patterns are used:
//
// Chains (a training step of the surrogate): each kernel consumes what the one before it wrote. Its CTAs park in
// grid_dep_wait(), which hides the launch latency.
//  * every kernel of a chain calls grid_dep_wait() before any global-memory access (read or write) and before
//    allocating tensor memory, except reads of data that no launch from its predecessor's predecessor on writes;
//    that one is complete when the predecessor's CTAs start their successor, because
//  * a kernel of a chain calls grid_dep_launch() only after its own grid_dep_wait(); so at most one kernel waits ahead
//    of the running one, too.
//
// Independent launches (the rows of tune_eval_archs): kernels that read only what was written before the first of them
// and whose outputs, counters included, are disjoint. The first is launched without the attribute. Each but the last
// calls grid_dep_launch() at its start, so that the next one's CTAs take the places that its own leave, and one CTA
// of each calls grid_dep_wait() before it ends, so that a launch is complete only after all before it.
//  * the last one does not call grid_dep_launch(): what follows it on the stream, a chain whose kernels read early
//    among it, starts when all of them are complete.
//  * a launch's CTAs start after all CTAs of the one before it have, so that waiting CTAs keep no place from them.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace pdl {

__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

// Both, in the order the rules above require.
__device__ __forceinline__ void grid_dep_enter()
{
    grid_dep_wait();
    grid_dep_launch();
}

// kern<<<grid, block, smem, s>>>(args...) with the programmatic-serialization attribute.
template <typename... KArgs, typename... Args>
cudaError_t launch_dep(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

}  // namespace pdl
