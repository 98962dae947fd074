// Host-side launch helper shared by the step's kernel files: programmatic
// dependent launches.
#pragma once

#include "ps_internal.cuh"

namespace ps {

// Launch with programmatic stream serialization: the kernel may be scheduled
// while its predecessor finishes (its CTAs wait in with_args until the
// predecessor's writes are visible), hiding the gap between dependent kernels.
template <typename... KArgs, typename... Args>
inline void launch_k(void (*kernel)(KArgs...), int grid, int block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace ps
