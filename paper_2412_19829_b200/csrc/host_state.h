// What the library keeps on the host between calls and shares among threads.
#pragma once

#include <cuda_runtime_api.h>

namespace gf {

// cudaFuncAttributeMaxDynamicSharedMemorySize of a kernel, raised to `bytes` unless it is as high already.
cudaError_t ensure_dynamic_smem(const void* kernel, int dev, int bytes);

}  // namespace gf
