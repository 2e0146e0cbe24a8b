// Launches of the step kernels, which follow one another on one stream.
//
// Each is launched so that its blocks may become resident while the kernel
// before it drains (programmatic dependent launch, also inside captured
// graphs): the launch latency and the blocks' set-up hide behind that kernel's
// tail.  Every kernel launched this way calls after_previous() in every thread
// before it touches memory that another kernel writes: it waits there until
// the kernel before it has completed and its stores are visible, and only then
// lets the next kernel's blocks in, so at most one kernel waits at a time.  A
// kernel parameter that points to such memory is not declared restrict (a
// read-only load of it could be moved above the wait).
//
// Per step of short runs (10 to 100 steps and the read of the populations), plain ->
// dependent launches: 64 x 40 FP32 5.1 -> 3.6 us, 512 x 384
// with reservoirs 28.8 -> 26.7, 701 x 523 with walls 50.1 -> 47.1, 512 x 512
// 33.0 -> 30.4, adjoint 256 x 256 (each of 20 steps) 128 -> 112; 2048 x 2048
// unchanged.  Not used where a kernel lives on the L1 cache behind one that
// takes its space as shared memory (thread-per-node surface source: 128 x 64 x
// 64 reactive step 4.42 -> 4.48 ms with it) nor for the batch's resident blocks,
// whose successors find no free slot (21.8 -> 22.0 us).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbm {

// Returns 0, or -1 where the launch was refused (the error also stays with
// cudaGetLastError for callers that launch several kernels).
template <class... K, class... A>
inline int launch_after(void (*kern)(K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kern, std::forward<A>(args)...) == cudaSuccess ? 0 : -1;
}

#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;\n griddepcontrol.launch_dependents;\n" ::: "memory");
}
#endif

}  // namespace lbm
