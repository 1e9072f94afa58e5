// Launches of kernels that follow one another on a stream, each reading what the one before wrote.
//
// A launch that waits for the previous kernel to end before it is set up costs about 2 us per step;
// with programmatic stream serialisation the next kernel's blocks are placed while the last ones of
// this kernel finish and wait inside, in wait_for_previous(), for its memory.  Measured: an empty
// kernel 2.05 -> 1.5 us; a step with 121 x 75 x 50 nodes (FP32, tensor field) 22.7 -> 19.5 us, 32^3
// (FP64) 8.3 -> 7.2 us, 24^3 (FP32) 4.2 -> 3.8 us.  Index arithmetic belongs ahead of the wait (24^3
// 3.2 -> 2.9 us with the two divisions of the coordinates there).
//
// The next launch is let in before the wait, so on a small lattice several launches can stand on the
// chip at once: step N + 1 may be placed while N still waits and N - 1 still loads the buffer that N + 1
// will read, whose old lines are then in the L1 that N + 1 uses.  What makes this right is the wait
// itself (griddepcontrol.wait): when it returns, the launches before have completed, and what they
// wrote is visible to this one's loads.  That holds for plain loads behind it.  Read-only loads may be
// moved ahead of it, so nothing that an earlier step writes is read with them.
// With the next launch let in after the wait (two launches at most), whole passes were 24^3 FP32 128 ->
// 117 us and 128 x 128 D2Q9 54 -> 48 us, but 48 x 40 x 32 FP32 at rest 343 -> 376 us, 17 x 16 x 20 198
// -> 206 us and the 64^3 gradient 1.176 -> 1.186 ms; boxes of 100^3 and more alike.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace elbm {

// In every kernel launched by launch_next, once in every thread: lets the next launch be placed, then
// waits until the kernel before this one has ended and its writes are visible.  Nothing that an
// earlier kernel writes may be touched before it.
__device__ __forceinline__ void wait_for_previous() {
  cudaTriggerProgrammaticLaunchCompletion();
  cudaGridDependencySynchronize();
}

template <typename... Params, typename... Args>
inline cudaError_t launch_next(void (*kernel)(Params...), dim3 grid, dim3 block, size_t shared, cudaStream_t s,
                               Args&&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = shared;
  c.stream = s;
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, std::forward<Args>(args)...);
}

}  // namespace elbm
