// chained_launch.h -- launches of the kernels that follow one another inside one call (the
// factor's sweep, GPTQ's block loop), by programmatic dependent launch: the kernel before each lets
// it be scheduled as soon as it starts, and it waits for that kernel's writes before its first read
// of them, so those launches do not each wait out a launch's latency.  The first kernel of a call
// is launched in stream order.
#pragma once
#include <cuda_runtime.h>

namespace hscale {

template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, unsigned block, int smem, cudaStream_t stream,
                           Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace hscale
