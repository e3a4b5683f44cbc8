"""The kernels' shared-memory attribute under threads, without a GPU: the host header against a stand-in for the CUDA call."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = "/usr/local/cuda/include"

PROGRAM = r"""
#include "smem_attr.h"
#include <chrono>
#include <thread>
static std::atomic<int> attribute{0}, calls{0};
static std::atomic<bool> inside{false};
// The first caller (it wants more) has set its value and is held up on its way back, the second one comes meanwhile.
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
  ++calls;
  attribute = bytes;
  if (bytes == 150000) { inside = true; std::this_thread::sleep_for(std::chrono::milliseconds(200)); }
  return cudaSuccess;
}
static void kernel() {}
int main() {
  static moehub::SmemAttrOnce once;
  std::thread big([] { moehub::ensure_dynamic_smem(kernel, 150000, 0, once); });
  while (!inside) std::this_thread::yield();
  std::thread small([] { moehub::ensure_dynamic_smem(kernel, 100000, 0, once); });
  big.join();
  small.join();
  if (attribute != 150000) return 1;                     // what the first thread launches with
  moehub::ensure_dynamic_smem(kernel, 150000, 0, once);
  if (attribute != 150000 || calls != 1) return 2;
  moehub::ensure_dynamic_smem(kernel, 160000, 0, once);  // grows
  moehub::ensure_dynamic_smem(kernel, 100000, 1, once);  // another device has its own
  return attribute == 100000 && calls == 3 ? 0 : 3;
}
"""


@pytest.mark.skipif(not os.path.isdir(CUDA_INCLUDE), reason="CUDA headers not here")
def test_a_smaller_request_never_takes_back_a_larger_one(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", os.path.join(ROOT, "paper_2605_05888_b200", "csrc"), "-I", CUDA_INCLUDE,
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
