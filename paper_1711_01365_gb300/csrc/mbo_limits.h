// What launchers remember of a kernel: the dynamic shared memory it may use and
// how many of its blocks a device holds.  Both belong to a device, and host threads
// with handles of their own launch the same kernels.
#pragma once
#include <stddef.h>

#include <atomic>
#include <mutex>

namespace mbo {

constexpr int kLimitDevices = 64;

// The shared-memory limit of one kernel.  It only ever grows: a smaller request
// that arrives late must not undo a larger one between its call and its launch.
class SmemLimit {
 public:
  // set(bytes) raises the limit on the current device dev and returns 0 where it did.
  template <class Set> auto raise(int dev, size_t bytes, Set set) -> decltype(set(bytes)) {
    using E = decltype(set(bytes));
    if (bytes <= 48 * 1024) return E(0);  // every kernel's own limit
    std::atomic<size_t>* have = dev >= 0 && dev < kLimitDevices ? &have_[dev] : nullptr;
    if (have && bytes <= have->load(std::memory_order_acquire)) return E(0);
    std::lock_guard<std::mutex> lk(mu_);
    if (have && bytes <= have->load(std::memory_order_relaxed)) return E(0);
    const E e = set(bytes);
    if (have && e == E(0)) have->store(bytes, std::memory_order_release);
    return e;
  }

 private:
  std::mutex mu_;
  std::atomic<size_t> have_[kLimitDevices] = {};
};

// A positive number that depends on the device, asked for once on each.
class DeviceCount {
 public:
  template <class Ask> int get(int dev, Ask ask) {
    if (dev < 0 || dev >= kLimitDevices) return ask();
    int n = n_[dev].load(std::memory_order_relaxed);
    if (!n) n_[dev].store(n = ask(), std::memory_order_relaxed);
    return n;
  }

 private:
  std::atomic<int> n_[kLimitDevices] = {};
};

#ifdef __CUDACC__
inline int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}

template <typename K> inline cudaError_t raise_smem(K kernel, size_t bytes, SmemLimit& limit) {
  if (bytes <= 48 * 1024) return cudaSuccess;
  return limit.raise(current_device(), bytes, [&](size_t b) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
  });
}

inline int device_sms(int dev) {
  static DeviceCount sms;
  return sms.get(dev, [&] {
    int n = 1;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
  });
}
#endif

}  // namespace mbo
