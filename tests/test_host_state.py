"""What the library shares among host threads (csrc/host_state.cu), compiled against a CUDA runtime that only pretends."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_19829_b200", "csrc")

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


def run(program, tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    main = tmp_path / "main.cpp"
    main.write_text(program)
    exe = str(tmp_path / "check")
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-I", include, str(main), "-x", "c++",
                           os.path.join(CSRC, "host_state.cu"), "-o", exe])
    return subprocess.run([exe], timeout=60).returncode


def test_the_largest_shared_memory_that_a_thread_has_asked_for_stays_in_force(tmp_path):
    assert run(SMEM, tmp_path) == 0
