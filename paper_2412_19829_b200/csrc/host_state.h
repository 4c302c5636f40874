// What the library keeps on the host between calls and shares among threads.
#pragma once

#include <cuda_runtime_api.h>

#include <mutex>

namespace gf {

// cudaFuncAttributeMaxDynamicSharedMemorySize of a kernel, raised to `bytes` unless it is as high already.
cudaError_t ensure_dynamic_smem(const void* kernel, int dev, int bytes);

// The CTAs of a cut-chain launch wait for one another, so two such kernels must not share the SMs: each could hold some of
// them while its own unplaced CTAs wait for the rest.  Per device the calls that have one are therefore chained by an event:
// such a call starts only when the previous one, from whatever stream or host thread, has finished.  (Not inside a stream
// capture, where an outside event cannot be waited for: there the order of the caller's graphs applies.)  Entered ahead
// of the call's first launch and left behind its last one, because an event between two kernels would part their chain; also
// by a call that fails between its launches (the destructor), since its cut-chain kernel may be among those it has made.
class CutChainOrder {
 public:
  ~CutChainOrder() { (void)leave(); }
  cudaError_t enter(int dev, cudaStream_t stream);
  cudaError_t leave();  // records the event

 private:
  std::unique_lock<std::mutex> lock_;
  int dev_ = 0;
  cudaStream_t stream_ = nullptr;
};

}  // namespace gf
