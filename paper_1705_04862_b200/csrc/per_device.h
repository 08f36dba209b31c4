// Something that belongs to a device and is looked up or set once on each.  Plain C++, so that it can be tried without one.
#pragma once
#include <mutex>

namespace paac {

template <class T> class PerDevice {
 public:
  // What `make` (bool make(T&)) filled in on the first successful call for this device; nullptr if it fails, which is not
  // remembered, or for a device number out of range.
  template <class Make> const T* get(int device, Make make) {
    if (device < 0 || device >= MAX_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lock(mutex_);
    if (!made_[device]) made_[device] = make(value_[device]);
    return made_[device] ? &value_[device] : nullptr;
  }

 private:
  static constexpr int MAX_DEVICES = 64;
  std::mutex mutex_;
  T value_[MAX_DEVICES] = {};
  bool made_[MAX_DEVICES] = {};
};

}  // namespace paac
