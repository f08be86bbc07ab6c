// Values that hold for one CUDA context of one device, such as a kernel's
// raised shared-memory limit.  Host code only.
#pragma once

#include <map>
#include <mutex>
#include <unordered_map>

namespace fa {

// One value per (device, key), made on first use and made again when the
// device's context has changed: a device reset makes a context with a new id.
// The values of the context before are dropped then, so the table holds one
// context per device.  Safe with several threads.
template <class V>
class ContextTable {
  public:
    // The value of `key` in context `ctx` of device `dev`; make(&value) makes
    // it and returns whether to keep it (a value that could not be made is
    // made again by the next call).
    template <class F>
    V get(int dev, unsigned long long ctx, const void *key, F make) {
        std::lock_guard<std::mutex> lock(mu_);
        Device &d = devices_[dev];
        if (d.ctx != ctx) {
            d.values.clear();
            d.ctx = ctx;
        }
        auto it = d.values.find(key);
        if (it != d.values.end()) return it->second;
        V v{};
        if (make(&v)) d.values.emplace(key, v);
        return v;
    }

  private:
    struct Device {
        unsigned long long ctx = 0;
        std::unordered_map<const void *, V> values;
    };
    std::mutex mu_;
    std::map<int, Device> devices_;
};

}  // namespace fa
