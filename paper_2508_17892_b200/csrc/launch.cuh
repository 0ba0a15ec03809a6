// Host-side launch helper shared by the kernels' launchers.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace ilre {

// Launch that may overlap the end of the kernel before it in the stream (programmatic dependent
// launch): every kernel launched so calls grid_dep_wait() before it touches memory that the kernel before
// it may write or still read.  The first kernel of a call lets the next one in only after that wait, so
// that within a call everything of earlier calls is done.  The first kernel takes part too: its launch
// latency and set-up pass while the call before it ends.  A call behind another, plain launch of the
// first kernel -> this one: 1024-token attention 31.4 -> 28.6 us, key fill of 1024 tokens
// 22.6 -> 20.7, recall of 4096 tokens 46.3 -> 45.1, of 32768 tokens 95.2 -> 91.8 us.
template <typename... Params, typename... Args>
cudaError_t launch_after_previous(void (*kernel)(Params...), int grid, int block, size_t smem,
                                  cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace ilre
