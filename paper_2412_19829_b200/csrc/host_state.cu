#include "host_state.h"

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

namespace {
std::mutex g_cut_mutex;
cudaEvent_t g_cut_last[64] = {};  // per device: behind the last call that has a cut-chain launch
}  // namespace

cudaError_t CutChainOrder::enter(int dev, cudaStream_t stream) {
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(stream, &capturing);
  if (e != cudaSuccess || capturing != cudaStreamCaptureStatusNone) return e;
  lock_ = std::unique_lock<std::mutex>(g_cut_mutex);
  dev_ = dev;
  stream_ = stream;
  cudaEvent_t& ev = g_cut_last[dev];
  e = ev == nullptr ? cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) : cudaStreamWaitEvent(stream, ev, 0);
  if (e != cudaSuccess) lock_.unlock();
  return e;
}

cudaError_t CutChainOrder::leave() {
  if (!lock_.owns_lock()) return cudaSuccess;
  const cudaError_t e = cudaEventRecord(g_cut_last[dev_], stream_);
  lock_.unlock();
  return e;
}

}  // namespace gf
