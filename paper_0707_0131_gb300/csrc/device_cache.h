// Answers of a yes / no question about a device, asked once per device.  Host code without CUDA, so
// that it can be checked on the CPU.
#pragma once
#include <map>
#include <mutex>

namespace eig {

class DeviceCache {
    std::mutex mu;
    std::map<int, bool> known;

   public:
    // ask() returns 1 or 0, or a negative number where it could not find out (asked again then)
    template <typename F>
    bool get(int device, F ask) {
        std::lock_guard<std::mutex> lk(mu);
        const auto it = known.find(device);
        if (it != known.end()) return it->second;
        const int a = ask();
        if (a >= 0) known[device] = a > 0;
        return a > 0;
    }
};

}  // namespace eig
