// Facts and settings that are the device's, kept once per device (no CUDA headers, so that it can
// be compiled and checked on a host without a GPU).
#ifndef FF_DEVICE_H_
#define FF_DEVICE_H_

#include <atomic>
#include <mutex>

#define FF_MAX_DEVICES 64

// A value for each device, made at its first use there.  A kernel's limit of dynamic shared memory
// is set on one device and says nothing about the next, and contexts of several devices and host
// threads may share a process: a plain static flag would leave the second device unset.
template <typename T>
class PerDevice {
 public:
  // The value of device dev: made by make(T&) unless it is there.  Null if dev is out of range or
  // make returns false (the next call tries again).
  template <typename F>
  const T* get(int dev, F make) {
    if (dev < 0 || dev >= FF_MAX_DEVICES) return nullptr;
    if (!have_[dev].load(std::memory_order_acquire)) {
      std::lock_guard<std::mutex> lock(mu_);
      if (!have_[dev].load(std::memory_order_relaxed)) {
        if (!make(value_[dev])) return nullptr;
        have_[dev].store(true, std::memory_order_release);
      }
    }
    return &value_[dev];
  }

 private:
  std::mutex mu_;
  std::atomic<bool> have_[FF_MAX_DEVICES] = {};
  T value_[FF_MAX_DEVICES] = {};
};

#endif  // FF_DEVICE_H_
