// A number per device and slot, found once on each device.
#pragma once

#include <array>
#include <map>
#include <mutex>

namespace sdfg {

template <int SLOTS> class PerDevice {
  public:
    // The number of `slot` on `device`, which must be the current device: what
    // find() returns is a property of that device, and what it sets there (a
    // kernel's attributes) holds there alone.  0 is not kept: the next call asks again.
    template <class Find> int get(int device, int slot, Find find) {
        std::lock_guard<std::mutex> lk(mu_);
        int &n = known_[device][slot];
        if (n == 0) n = find();
        return n;
    }

  private:
    std::mutex mu_;
    std::map<int, std::array<int, SLOTS>> known_;
};

}  // namespace sdfg
