// Launches of the step sequence (internal).
#pragma once
#include <cuda_runtime.h>

namespace ebit_detail {

// Launches kernel k, which begins with chained_start(), on stream st so that
// its blocks may become resident while the launch before it drains: the gap
// between two dependent kernels (1-2 us) then holds the second one's start.  An
// error is the runtime's last error, as after <<<>>>.
template <typename... P, typename... A>
inline void launch_chained(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... a) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, static_cast<P>(a)...);
}

}  // namespace ebit_detail
