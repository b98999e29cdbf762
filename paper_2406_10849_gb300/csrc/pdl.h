// Launch with programmatic stream serialisation: the kernel may start before its
// predecessor in the stream has finished, and waits for it itself (pdl_wait in
// ptx.cuh).  The half-step's launches are microseconds long on small problems; the
// next one's start-up then runs beside the last one's tail.
#pragma once
#include <cuda_runtime.h>

namespace treeot {

inline cudaError_t launch_pdl(const void* fn, int grid, int block, size_t smem, cudaStream_t s, void** args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace treeot
