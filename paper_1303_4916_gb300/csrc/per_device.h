// per_device.h -- what the CUDA runtime keeps for each device: a kernel's limit
// of dynamic shared memory, its occupancy.  Both are asked for once per device
// (on every launch they took as long as the launch), not once per process: a
// process may hold contexts on several devices, and a limit set on one does not
// hold on the next, where a launch above 48 KB then fails.
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>

// ask() >= 0, kept per current device; a negative answer is a failure, is not
// kept, and leaves the runtime's error for the caller's cudaGetLastError.
// Threads that ask at the same time may both ask: the answer is the same.
class PerDevice {
 public:
  static constexpr int kDevices = 64;  // beyond them every call asks
  template <class F>
  int get(F&& ask) {
    int d = -1;
    if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= kDevices) return ask();
    const int kept = v_[d].load(std::memory_order_acquire);
    if (kept > 0) return kept - 1;
    const int v = ask();
    if (v >= 0) v_[d].store(v + 1, std::memory_order_release);
    return v;
  }

 private:
  std::atomic<int> v_[kDevices] = {};  // answer + 1; 0: not asked
};

// Dynamic shared memory of up to `bytes` for the kernel on the current device: 0, or -1.
template <class K>
int hf_smem_limit(PerDevice& kept, K kernel, size_t bytes) {
  return kept.get([&] {
    return cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)bytes) == cudaSuccess
               ? 0
               : -1;
  });
}

// Blocks of `threads` threads and `smem` bytes of dynamic shared memory that an SM of the current device holds, or -1.
template <class K>
int hf_resident_blocks(PerDevice& kept, K kernel, int threads, size_t smem) {
  return kept.get([&] {
    int n = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, reinterpret_cast<const void*>(kernel), threads, smem) ==
                   cudaSuccess
               ? n
               : -1;
  });
}
