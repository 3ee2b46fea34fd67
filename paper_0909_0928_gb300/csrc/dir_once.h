// dir_once.h -- something found out once per device and then only read (host code).
#pragma once

#include <atomic>
#include <mutex>

namespace dirk {

// get() fills the value of a device at the first call for it and returns it, by
// any number of threads: one of them fills, those that waited for it look again
// before they would, so that a value is never written once it has been handed out.
template <typename T, int MaxDevices>
class OncePerDevice {
  public:
    template <typename Fill>
    const T* get(int dev, Fill&& fill) {
        if (dev < 0 || dev >= MaxDevices) return nullptr;
        if (!known_[dev].load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lock(mutex_);
            if (!known_[dev].load(std::memory_order_relaxed)) {
                fill(value_[dev]);
                known_[dev].store(true, std::memory_order_release);
            }
        }
        return &value_[dev];
    }

  private:
    std::atomic<bool> known_[MaxDevices] = {};
    T value_[MaxDevices] = {};
    std::mutex mutex_;
};

}  // namespace dirk
