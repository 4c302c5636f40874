"""What the library shares among host threads (csrc/host_state.cu), compiled against a CUDA runtime that only pretends."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_19829_b200", "csrc")

# (what a program does not pretend itself)
STUBS = r"""
#include <cuda_runtime_api.h>
extern "C" {
__attribute__((weak)) cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaErrorUnknown; }
__attribute__((weak)) cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus*) { return cudaErrorUnknown; }
__attribute__((weak)) cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned int) { return cudaErrorUnknown; }
__attribute__((weak)) cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaErrorUnknown; }
__attribute__((weak)) cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaErrorUnknown; }
}
"""

SMEM = r"""
#include <atomic>
#include <chrono>
#include <thread>
#include "host_state.h"
std::atomic<int> entered{0}, in_force{0}, calls{0};
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
  ++calls;
  entered = bytes;
  if (bytes == 60000) std::this_thread::sleep_for(std::chrono::milliseconds(300));  // overtaken, if another call may
  in_force = bytes;
  return cudaSuccess;
}
int main() {
  const void* kernel = &entered;
  std::thread small([&] { gf::ensure_dynamic_smem(kernel, 0, 60000); });
  while (entered != 60000) std::this_thread::yield();
  gf::ensure_dynamic_smem(kernel, 0, 116000);
  small.join();
  if (in_force != 116000) return 1;
  gf::ensure_dynamic_smem(kernel, 0, 60000);  // (less than what is in force)
  return in_force == 116000 && calls == 2 ? 0 : 2;
}
"""

ORDER = r"""
#include <cstring>
#include <string>
#include "host_state.h"
std::string log_;
cudaError_t create = cudaSuccess;
extern "C" cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = s == (cudaStream_t)9 ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
extern "C" cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned int) {
  if (create == cudaSuccess) *e = (cudaEvent_t)1;
  return create;
}
extern "C" cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t, unsigned int) {
  log_ += "w" + std::to_string((long)s);
  return cudaSuccess;
}
extern "C" cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  log_ += (e ? "r" : "null") + std::to_string((long)s);
  return cudaSuccess;
}
int main() {
  auto call = [](long stream, bool fails) {
    gf::CutChainOrder order;
    if (order.enter(0, (cudaStream_t)stream) != cudaSuccess || fails) return;
    order.leave();
  };
  create = cudaErrorMemoryAllocation;
  call(1, false);  // no event: not entered, nothing recorded, and the next call is not kept out
  create = cudaSuccess;
  call(1, false);
  call(2, true);   // between its launches: the next call waits for what it has launched
  call(9, true);   // captured: no part in the order
  call(3, false);
  return log_ == "r1" "w2r2" "w3r3" ? 0 : 1;
}
"""


def run(program, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    main = tmp_path / "main.cpp"
    main.write_text(program)
    stubs = tmp_path / "stubs.cpp"
    stubs.write_text(STUBS)
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-I", include, str(main), str(stubs), "-x", "c++",
                           os.path.join(CSRC, "host_state.cu"), "-o", exe])
    return subprocess.run([exe], timeout=60).returncode


def test_the_largest_shared_memory_that_a_thread_has_asked_for_stays_in_force(tmp_path):
    assert run(SMEM, tmp_path) == 0


def test_a_call_that_fails_between_its_launches_leaves_the_order_of_cut_chain_calls(tmp_path):
    assert run(ORDER, tmp_path) == 0
