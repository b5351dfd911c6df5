// dg_stream_launch.h -- kernel launches that overlap with the end of their
// predecessor in the stream.
#pragma once
#include <cuda_runtime.h>

namespace dg {

// Launch with programmatic stream serialisation: the chip sets the kernel up
// while its predecessor drains, which hides most of a launch on small meshes
// (8^3, FP64, order 2, 13 kernels per step: 105 us with plain launches, 74 so).
// The kernel's first statement is stream_wait().
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
  // the caller gets the error: not left for the next cudaGetLastError, here or in
  // another library, to report as its own
  if (e != cudaSuccess) (void)cudaGetLastError();
  return e;
}

}  // namespace dg
