// Host side of kernels that ask for more dynamic shared memory than the default.
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>
#include <mutex>
#include <stddef.h>

namespace moehub {

// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) applies to the CURRENT device only, so what a kernel's attribute
// was last set to is kept per device (a process may hold plans on several GPUs).
struct SmemAttrOnce {
  std::atomic<size_t> set[64] = {};
};

// The attribute only ever grows: plans of other shapes, on other threads, may need less of the same kernel, and a thread
// that found too little must not set its own smaller value behind one that has just set more.
template <typename Kern>
inline cudaError_t ensure_dynamic_smem(Kern kern, size_t bytes, int device, SmemAttrOnce& once) {
  static std::mutex mutex;
  const bool kept = device >= 0 && device < 64;
  if (kept && once.set[device].load(std::memory_order_acquire) >= bytes) return cudaSuccess;
  std::lock_guard<std::mutex> lock(mutex);
  if (kept && once.set[device].load(std::memory_order_relaxed) >= bytes) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kern), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess && kept) once.set[device].store(bytes, std::memory_order_release);
  return e;
}

}  // namespace moehub
