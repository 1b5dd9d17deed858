// Kernel launches that overlap with the end of the kernel before them in the stream (programmatic dependent launch).
//
// Most kernels of a training step take 3 .. 20 us, and a dependent launch that waits for the whole device to drain adds
// 1 .. 2 us of launch latency, barrier set-up, TMEM allocation and descriptor fetches to each.  Launched this way a
// kernel's CTAs become resident as soon as every CTA of the kernel before has called pdl_trigger() or left, and do
// their set-up while that one's last CTAs finish.
//
// The rule that makes this safe: every kernel launched with pdl_launch calls pdl_wait() in all of its threads before
// its first access to global memory (but for a look at the status word, which may come too early to see that the step
// is void already: then its work is for nothing); the wait returns when the kernel before has completed and its writes
// are visible.  As that kernel waited for its own predecessor in the same way, completion is transitive: nothing later
// in the stream, and no event recorded in it, sees anything early.
//
// The loads behind the wait are ordinary ones.  __ldg, and a pointer parameter that is both const and __restrict__,
// promise that the data is read-only while the KERNEL runs, which the kernel before may still contradict: such loads may
// be taken from the non-coherent cache, and the compiler may move them in front of the wait, whose "memory" clobber says
// nothing about read-only data.  So inputs are plain const pointers; __restrict__ stays on outputs, which is what lets a
// loop's loads pass its stores.
//
// The tensor-core kernels trigger when their producer warp has issued its last load; the others leave it to their end.
// Earlier triggers make the incoming CTAs hold SMs that other streams' kernels could use.  Steps in us, without this /
// triggers at the start of every kernel / of the tensor-core kernels only / nowhere / as it is: 512 x 128 MLP 146 / 127 /
// 125 / 133 / 122; 4096 x 512 MLP, one stream 907 / 832 / 838 / 843 / 837; LM d 256 on several streams 788 / 793 / 794 /
// 778 / 766, without graphs 876 / 776 / 825 / 788 / 790; CTR with main network 779 / 774 / 773 / 755 / 758.
#pragma once
#include <cuda_runtime.h>
#include <string.h>

namespace erase {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t pdl_launch_cluster(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, unsigned cluster, bool dependent,
                               A&&... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = dependent ? 1 : 0;
  at[1].id = cudaLaunchAttributeClusterDimension;      // (cluster 0: the kernel's own)
  at[1].val.clusterDim.x = cluster; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
cudaError_t pdl_launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  return pdl_launch_cluster(kernel, grid, block, smem, s, 0u, true, static_cast<A&&>(args)...);
}

}  // namespace erase
