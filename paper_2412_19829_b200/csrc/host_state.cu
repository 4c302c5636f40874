#include "host_state.h"

#include <mutex>
#include <vector>

namespace gf {

cudaError_t ensure_dynamic_smem(const void* kernel, int dev, int bytes) {
  struct Done {
    const void* kernel;
    int dev, bytes;
  };
  static std::mutex mu;
  static std::vector<Done> done;
  // Held until the attribute is set: a kernel is asked for in several sizes, and the last one set is the one in force.
  std::lock_guard<std::mutex> lock(mu);
  for (const Done& x : done)
    if (x.kernel == kernel && x.dev == dev && x.bytes >= bytes) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.push_back(Done{kernel, dev, bytes});
  return e;
}

}  // namespace gf
