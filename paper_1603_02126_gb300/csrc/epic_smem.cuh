// Dynamic shared memory of a kernel (sm_103a).
#pragma once

#include <cuda_runtime.h>

namespace epic {

// Lets a kernel take all the shared memory a block may have.  The attribute
// belongs to the kernel, not to a plan or a launch: set to one plan's size it
// would stop an older plan with a larger footprint, or another thread's.
template <typename Kernel>
cudaError_t allow_smem(Kernel kernel) {
  int dev = 0, most = 0;
  cudaFuncAttributes fa{};
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most - static_cast<int>(fa.sharedSizeBytes));
  return e;
}

}  // namespace epic
