// A value for each device: function attributes and occupancy belong to one
// device, and a process may have plans on several.  Host code only.
#pragma once
#include <map>
#include <mutex>

namespace xb {

template <typename T>
class PerDevice {
  public:
    // The device's value in *out.  At the device's first call make(T &) fills it
    // in and returns 0; an error code is returned and not remembered.
    template <typename Make>
    int get(int device, Make make, T *out) {
        std::lock_guard<std::mutex> lock(mu_);
        auto it = values_.find(device);
        if (it == values_.end()) {
            T t{};
            const int r = make(t);
            if (r != 0) return r;
            it = values_.emplace(device, t).first;
        }
        *out = it->second;
        return 0;
    }

  private:
    std::mutex mu_;
    std::map<int, T> values_;
};

}  // namespace xb
