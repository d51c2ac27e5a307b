// Kernel launches that overlap the end of the kernel before them
// (programmatic dependent launch).
//
// A reconstruction is a chain of kernels on one stream. Launched plainly, each
// waits for the last CTA of the one before and then pays the launch itself,
// about 2.3 us a kernel here, which small captures feel: a 32x32x256 f-k
// volume took 31 us on a stream and 21 us as a replayed graph.
//
// A kernel launched with `after` may start once every CTA of the kernel before
// it has called pdl_trigger() or exited. It calls pdl_wait() before its first
// access to memory that any earlier kernel touches (reads and writes alike;
// plan tables are constant and may be read before); the wait returns once the
// kernel before has completed and its writes are visible. As every kernel
// of a chain waits before it completes, completion is in order along the
// chain. The first kernel of a call is launched plainly: what precedes it on
// the stream is not the library's.
//
// A chained kernel reads what another kernel of the chain writes with plain
// loads, never with __ldg or through a const __restrict__ pointer: the
// non-coherent path is defined only for memory that nothing writes while the
// kernel is resident, and a chained kernel is resident before its
// predecessors have finished. Plan tables are constant and may take that path.
//
// Kernels of one tile per CTA trigger at their start (the next kernel can
// then only take SM slots that no CTA of this one is left to fill); persistent
// ones when they take their last tile.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace nlos {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_kernel(bool after, void (*k)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                                 A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = after ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
  return cudaGetLastError();
}

}  // namespace nlos
