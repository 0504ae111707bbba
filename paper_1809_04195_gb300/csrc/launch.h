// Kernel launches that may start before the previous kernel of the stream has ended (programmatic
// stream serialisation).  The kernel runs its prologue (tables, barriers, plan-owned constants) and
// then pdl_wait(), after which the previous kernels' results are visible; pdl_trigger() lets the next
// such kernel do the same (without it that kernel starts when every CTA of this one has ended, which
// still hides the launch itself).  A kernel triggers only after its own wait, so whatever ran before the
// previous kernel has completed when a prologue runs.  What the previous kernel may have written is
// not read-only while this one runs: an argument that is read after the wait and written by another
// kernel carries no `__restrict__` (its loads could be hoisted above the wait, and a `const` one's
// sent through the read-only path), and no asm load of it is without `volatile`.
#pragma once

#include <cuda_runtime.h>

namespace t2sh {

// cluster_z > 1: CTAs of a cluster are neighbours along the grid's z axis
template <typename... P, typename... A>
inline cudaError_t launch_pdl_cluster(void (*kern)(P...), dim3 grid, int cluster_z, int threads, size_t smem,
                                      cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 1;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = (unsigned)cluster_z;
  cfg.attrs = at;
  cfg.numAttrs = cluster_z > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  return launch_pdl_cluster(kern, grid, 1, threads, smem, st, args...);
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace t2sh
