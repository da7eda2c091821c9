// A value found out once per device (kernel attributes set, occupancies): attributes
// belong to a device, so a process that goes on to another one sets them there too.
#pragma once
#include <map>
#include <mutex>

namespace simk {

template <typename T> class PerDevice {
  public:
    // The device's value; make() the first time it is asked for (any thread).
    template <typename Make> T get(int device, Make make)
    {
        std::lock_guard<std::mutex> lock(mu_);
        const auto it = values_.find(device);
        if (it != values_.end()) return it->second;
        return values_.emplace(device, make()).first->second;
    }

  private:
    std::mutex mu_;
    std::map<int, T> values_;
};

} // namespace simk
