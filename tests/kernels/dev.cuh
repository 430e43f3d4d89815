// Host arrays on the device, for the entry points of the kernel tests.
#pragma once
#include <cuda_runtime.h>

#define ENTRY extern "C" __attribute__((visibility("default"))) int

namespace {

template <typename T>
struct Dev {
  T* p = nullptr;
  size_t n;
  explicit Dev(size_t n_, const T* src = nullptr) : n(n_) {
    if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess) p = nullptr;
    if (p && src) cudaMemcpy(p, src, n * sizeof(T), cudaMemcpyHostToDevice);
    else if (p) cudaMemset(p, 0, n * sizeof(T));
  }
  ~Dev() { cudaFree(p); }
  bool get(T* dst) { return cudaMemcpy(dst, p, n * sizeof(T), cudaMemcpyDeviceToHost) == cudaSuccess; }
};

}  // namespace
