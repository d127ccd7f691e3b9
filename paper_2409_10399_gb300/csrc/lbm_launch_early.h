// Launch of a step kernel with programmatic dependent launch.
#pragma once
#include <cuda_runtime.h>

namespace lbm {

// Launch whose blocks may be scheduled before the end of the kernel before it
// (wait_previous in the kernel).  As after <<<>>>, a refused launch is what the
// caller's next cudaGetLastError returns.
template <class K, class... A>
static void launch_early(K kern, dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace lbm
