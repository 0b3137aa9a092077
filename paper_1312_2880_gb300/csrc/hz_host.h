// Host-side state that belongs to a device and not to the process: what the launchers look up or set once.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace hz {

constexpr int MAX_DEVICES = 64;  // devices beyond are looked up and set at every call

// A step that every device needs once before its first launch of a kernel (shared-memory opt-in, cluster
// size). Safe with concurrent callers: the step may run more than once, and it has run on the
// current device when the call returns.
class OncePerDevice {
 public:
  template <class Step>
  cudaError_t operator()(Step&& step) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < MAX_DEVICES ? 1ull << dev : 0ull;
    if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = step();
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<unsigned long long> done_{0};
};

// An integer property of the current device (`find`, called when it is not yet known; < 1: unknown).
class IntPerDevice {
 public:
  template <class Find>
  int operator()(Find&& find) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    int v = dev < MAX_DEVICES ? v_[dev].load(std::memory_order_acquire) : 0;
    if (v < 1) {
      v = find(dev);
      if (v > 0 && dev < MAX_DEVICES) v_[dev].store(v, std::memory_order_release);
    }
    return v;
  }

 private:
  std::atomic<int> v_[MAX_DEVICES] = {};
};

// SMs of the current device (1 if it cannot be asked).
inline int device_sms() {
  static IntPerDevice sms;
  const int v = sms([](int dev) {
    int n = 0;
    return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? n : 0;
  });
  return v > 0 ? v : 1;
}

}  // namespace hz
