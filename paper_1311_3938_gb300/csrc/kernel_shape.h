// What the host has learned about one kernel, by device: the dynamic shared memory it is allowed and
// the grid for one amount of it.  One object per kernel, a static of its launcher; several host threads may
// launch through it, on several devices.
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace aqc {

class KernelShape {
 public:
  // Lets `kern` take smem bytes of dynamic shared memory on the current device.
  template <typename K>
  cudaError_t allow(K kern, size_t smem) {
    std::lock_guard<std::mutex> hold(m_);
    return raise(kern, (int)smem, nullptr);
  }
  // The same, and *grid = what ask(device, &g) gives (kept for the last smem).
  template <typename K, typename Ask>
  cudaError_t grid(K kern, int smem, Ask ask, int* grid) {
    std::lock_guard<std::mutex> hold(m_);
    int device = 0;
    cudaError_t e = raise(kern, smem, &device);
    if (e != cudaSuccess) return e;
    Known* const k = device < kDevices ? &known_[device] : nullptr;
    if (k && k->smem == smem) {
      *grid = k->grid;
      return cudaSuccess;
    }
    e = ask(device, grid);
    if (e == cudaSuccess && k) {
      k->smem = smem;
      k->grid = *grid;
    }
    return e;
  }

 private:
  static constexpr int kDevices = 32;  // beyond: asked every time
  struct Known {
    int allowed = 0, smem = -1, grid = 0;
  };

  template <typename K>
  cudaError_t raise(K kern, int smem, int* device_out) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device_out) *device_out = device;
    if (device < kDevices && smem <= known_[device].allowed) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) {
      (void)cudaGetLastError();  // reported here, not by the next launch
      return e;
    }
    if (device < kDevices) known_[device].allowed = smem;
    return cudaSuccess;
  }

  std::mutex m_;
  Known known_[kDevices];
};

}  // namespace aqc
