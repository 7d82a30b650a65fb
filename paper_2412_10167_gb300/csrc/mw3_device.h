// What a launcher settles once per device. A kernel's dynamic shared-memory limit, its occupancy
// and the SM count belong to a device, and a process may hold contexts and networks on several
// of them: a process-wide flag would leave every device but the first without the limit.
#pragma once

#include <atomic>
#include <cstdint>

namespace mw3 {

// Runs an action once per device (again while it fails). Threads that meet may both run it: the
// actions kept here may be repeated.
class OncePerDevice {
 public:
  template <class F>
  auto run(int dev, F action) -> decltype(action()) {
    using Status = decltype(action());
    const uint64_t bit = dev >= 0 && dev < 64 ? uint64_t(1) << dev : 0;   // others: every time
    if (done_.load(std::memory_order_acquire) & bit) return Status(0);
    const Status e = action();
    if (e == Status(0)) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

// A positive integer per device, computed at its first use there.
class IntPerDevice {
 public:
  template <class F>
  int get(int dev, F compute) {
    if (dev < 0 || dev >= 64) return compute();
    int v = v_[dev].load(std::memory_order_relaxed);
    if (!v) v_[dev].store(v = compute(), std::memory_order_relaxed);
    return v;
  }

 private:
  std::atomic<int> v_[64] = {};
};

}  // namespace mw3

#ifdef __CUDACC__
#include <cuda_runtime.h>

namespace mw3 {

inline int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}

inline int sm_count() {
  static IntPerDevice n;
  const int dev = current_device();
  return n.get(dev, [&] {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v > 0 ? v : 1;
  });
}

// The kernel's dynamic shared memory may be up to `bytes` on the current device. `once` is a
// static of the launcher of this one kernel.
template <class K>
cudaError_t allow_smem(OncePerDevice& once, K kernel, size_t bytes) {
  return once.run(current_device(), [&] {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  });
}

}  // namespace mw3
#endif
